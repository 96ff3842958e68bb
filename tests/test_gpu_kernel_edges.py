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


# ising_energy: one-CTA instances (up to 2048 spins) and larger ones in parts of
# 1024 sites; 4, 16 and 32 replicas per word group and their remainders; sizes
# that are no multiple of 4 and spins that start on an odd byte; lattices of
# both dimensions; rows of 48 entries and more; hyper-edges.  Integer energies
# are equal; float ones are exact sums rounded once, the oracle's FP64 sums of
# up to 2^14 terms within 1e-12 relative of them.
def _energy_instances(kind):
    if kind == "square":
        return [W.lattice((d, d), True, "gauss", "gauss", seed=d) for d in (3, 45, 46)]
    if kind == "cube":
        return [W.lattice((d, d, d), True, "pm1", "pm1_0", seed=d) for d in (3, 12, 13)]
    if kind == "rows":
        return [W.dense_to_csr(W.sk(n, seed=n)) for n in (48, 49, 210)]
    if kind == "mixed":
        return [W.random_graph(n, 5.0, n, dtype="i8", n_hyper=n // 3, hyper_order=(2, 3, 5)) for n in (7, 2048, 2049)]
    return [W.random_graph(n, 5.0, n, dtype="f32", n_hyper=n // 3, hyper_order=(2, 3, 5)) for n in (8, 1500, 3001)]


@pytest.mark.parametrize("R", [1, 4, 5, 16, 17, 33])
@pytest.mark.parametrize("kind", ["square", "cube", "rows", "mixed", "float"])
def test_energy_sizes_and_replica_groups(kind, R):
    insts = _energy_instances(kind)
    h = isg.Handle(insts)
    rng = np.random.default_rng(R)
    spins = (rng.integers(0, 2, size=R * h.total_spins) * 2 - 1).astype(np.int8)
    for shift in (0, 1, 4):
        buf = torch.empty(spins.size + 8, dtype=torch.int8, device="cuda")[shift:shift + spins.size]
        buf.copy_(torch.from_numpy(spins))
        for _ in range(2):  # a second call finds the sums cleared
            E = h.energy(buf, R).cpu().numpy()
        off = 0
        for b, inst in enumerate(insts):
            ref = oracle.energies(inst, spins[off: off + R * inst.n].reshape(R, inst.n))
            off += R * inst.n
            if inst.dtype == "i8":
                assert np.array_equal(E[b], ref)
            else:
                np.testing.assert_allclose(E[b], ref, rtol=1e-12, atol=1e-9)
    h.close()


# Terms too wide for integer sums keep the FP64 passes.
def test_energy_wide_exponent_range():
    inst = _exp_spread(W.random_graph(2500, 5.0, 7, dtype="f32", n_hyper=100, hyper_order=(3,)), -45, 25)
    R = 6
    h = isg.Handle([inst])
    spins = (np.random.default_rng(1).integers(0, 2, size=(R, inst.n)) * 2 - 1).astype(np.int8)
    E = h.energy(torch.from_numpy(spins).cuda(), R)[0].cpu().numpy()
    np.testing.assert_allclose(E, oracle.energies(inst, spins), rtol=1e-12)
    h.close()
