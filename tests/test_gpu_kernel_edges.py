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


# Pass-based search with gain keys, move for move against the oracle's heap:
# one word per lane and whole trees (1 to 4096 spins, both sides of the flat
# layout's 512 and of each number of reads per lane), records of 31 entries (one
# more goes to the general kernel), hyper-edges of 2 and 3 members over existing
# pairs (targets that occur twice), values of one, two and three words, and FP32
# couplings of equal magnitudes (every move tied).
from test_gpu_fm import _compare as _compare_fm  # noqa: E402


def _fm_graph(kind, n):
    if kind == "pm1":
        return W.random_graph(n, 4.0, n, dtype="i8", n_hyper=n // 6, hyper_order=(2, 3), int_range=1)
    if kind == "int":
        return W.random_graph(n, 6.0, n, dtype="i8", n_hyper=n // 3, hyper_order=(2, 3), int_range=100)
    g = W.random_graph(n, 4.0, n, dtype="f32", n_hyper=n // 3, hyper_order=(2, 3))
    if kind == "ties":
        for k in ("J", "h", "hyper_J"):
            v = getattr(g, k)
            if v is not None:
                setattr(g, k, (np.sign(v) * (1 + np.arange(len(v)) % 2 if k == "h" else 1)).astype(np.float32))
    if kind == "halves":  # equal magnitudes and one tiny field: ties decided by low bits
        g.J = (np.sign(g.J) * np.float32(0.75)).astype(np.float32)
        g.h = np.full(n, 0.0, np.float32)
        g.h[0] = np.float32(2.0 ** -26)
    return _exp_spread(g, -14, 3) if kind == "wide" else g


@pytest.mark.parametrize("n", [1, 2, 33, 127, 129, 256, 257, 512, 513, 1024, 1025, 2049])
@pytest.mark.parametrize("kind", ["pm1", "int", "gauss", "ties", "halves", "wide"])
def test_fm_gain_keys(kind, n):
    _compare_fm([_fm_graph(kind, n)], 5, 1, kind in ("pm1", "int"))


def test_fm_gain_keys_largest_instance_and_mixed_batch():
    insts = [_fm_graph("gauss", 4096), _fm_graph("wide", 700), _fm_graph("halves", 300), _fm_graph("gauss", 90)]
    _compare_fm(insts, 3, 2, False)


@pytest.mark.parametrize("degree", [31, 32])
def test_fm_gain_keys_widest_record(degree):
    n = 64
    u, v = np.triu_indices(n, 1)
    keep = ((v - u) % n <= (degree // 2)) | ((u - v) % n <= (degree // 2)) | ((v - u == n // 2) & (degree % 2 == 1))
    u, v = u[keep], v[keep]
    w = np.random.default_rng(3).standard_normal(len(u)).astype(np.float32)
    rp, col, J = W.csr_from_edges(n, u, v, w, "f32")
    assert np.diff(rp).max() == degree
    _compare_fm([W.Instance(n=n, row_ptr=rp, col=col, J=J, dtype="f32")], 6, 2, False)
