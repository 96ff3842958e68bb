"""Kernel paths at the sizes where they can go wrong, against the CPU oracle:
spins, minima and work counters bit-exact, energies of integer instances equal
and of float ones within 1e-9 relative (both sides sum in FP64 or exactly)."""
import numpy as np
import pytest

import oracle
import workloads as W

torch = pytest.importorskip("torch")
pytestmark = pytest.mark.gpu

isg = pytest.importorskip("paper_0912_3912_gb300")

from test_gpu_parity import _compare, _exp_spread  # noqa: E402


@pytest.fixture(scope="module", autouse=True)
def _built():
    if not torch.cuda.is_available():
        pytest.skip("no GPU")
    from paper_0912_3912_gb300 import build as B
    B.build()
    oracle.build()


def _star_graph(n, dtype, seed):
    """A random graph plus a hub of degree 70 (rows longer than a warp's 32 lanes
    and than 8- and 16-lane groups) and hyper-edges of 2 to 9 members."""
    g = W.random_graph(n, 4.0, seed, dtype=dtype, n_hyper=60, hyper_order=(2, 3, 4, 9))
    rows = np.repeat(np.arange(n), np.diff(g.row_ptr))
    keep = (rows < g.col) & (rows != 5) & (g.col != 5)
    hub = np.arange(10, 80)
    u, v = np.concatenate([rows[keep], np.full(70, 5)]), np.concatenate([g.col[keep], hub])
    w = np.concatenate([g.J[keep], np.resize(g.J, 70)])
    g.row_ptr, g.col, g.J = W.csr_from_edges(n, u, v, w, dtype)
    return g


# General graphs in the sweep family: 8, 16 and 32 lanes per spin, one and two
# replica groups, rows and incidence lists longer than a group of lanes,
# classes smaller and larger than the warps; refreshes in fixed point and FP64.
@pytest.mark.parametrize("R", [3, 8, 13, 32, 45])
@pytest.mark.parametrize("dtype", ["i8", "f32"])
def test_sweep_general_graph_rows_longer_than_a_lane_group(dtype, R):
    _compare([_star_graph(300, dtype, 41)], [R], R, dtype == "i8", max_sweeps=400, restarts=2, refresh_every=3,
             kernel=isg.KERNEL_SWEEP)


@pytest.mark.parametrize("R", [7, 33])
def test_sweep_general_graph_fp64_refresh(R):
    inst = _exp_spread(_star_graph(200, "f32", 43), -45, 25)
    _compare([inst], [R], R, False, max_sweeps=400, restarts=2, refresh_every=2, kernel=isg.KERNEL_SWEEP)
