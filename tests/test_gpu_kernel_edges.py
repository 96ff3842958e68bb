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

from test_gpu_parity import _compare, _exp_spread, _oracle, _run  # noqa: E402


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


# Groups of 16 replicas on FP32 lattices (odd and even sides, a last group with
# one replica and with 15), chunks of 4, 8 and 16 sweeps and none (by the number
# of classes), and more replicas than one run's 32 groups hold.
@pytest.mark.parametrize("dims,R", [((9, 9, 9), 17), ((12, 12), 31), ((10, 10, 10), 40), ((7, 7), 513)])
def test_sweep_fp32_lattice_groups(dims, R):
    inst = W.lattice(dims, True, "gauss", "gauss", seed=sum(dims))
    _compare([inst], [R], R, False, max_sweeps=300, restarts=3, refresh_every=5, kernel=isg.KERNEL_SWEEP)


@pytest.mark.parametrize("dtype,R", [("i8", 1030), ("f32", 1025)])
def test_sweep_more_replicas_than_one_run(dtype, R):
    inst = W.random_graph(60, 4.0, 71, dtype=dtype, n_hyper=8)
    _compare([inst], [R], R, dtype == "i8", max_sweeps=60, restarts=2, kernel=isg.KERNEL_SWEEP)


@pytest.mark.parametrize("ncls", [30, 60, 120, 130])
def test_sweep_chunk_lengths(ncls):
    n = 2 * ncls
    inst = W.random_graph(n, 3.0, ncls, dtype="f32")
    order = np.random.default_rng(ncls).permutation(n)
    inst.colour = np.empty(n, np.int32)
    inst.colour[order] = np.arange(n) % ncls  # classes of two spins; conflicting pairs get a class of their own
    rows = np.repeat(np.arange(n), np.diff(inst.row_ptr))
    clash = np.unique(rows[inst.colour[rows] == inst.colour[inst.col]])
    inst.colour[clash] = ncls + np.arange(len(clash))
    _compare([inst], [ncls], 9, False, max_sweeps=200, restarts=3, refresh_every=4, kernel=isg.KERNEL_SWEEP)


# Tiles cut into segments of descents: more descents than segments and fewer,
# descents that never converge (the last one's state is the result) or only some,
# ragged replica groups, both schedules, every mode of the tile kernels.
def _segment_instance(kind):
    if kind == "lattice":
        return W.lattice((9, 9, 9), True, "pm1", "pm1_0", seed=51)
    if kind == "msc":
        return W.random_graph(150, 4.0, 52, dtype="i8", int_range=1, fields=False)
    return W.random_graph(170, 5.0, 53, dtype="f32" if kind == "f32" else "i8", n_hyper=30, hyper_order=(3, 4))


@pytest.mark.parametrize("max_sweeps,restarts,R", [(1, 7, 33), (4, 3, 5), (5, 40, 40), (300, 333, 3), (300, 2, 70)])
@pytest.mark.parametrize("kind", ["lattice", "msc", "i8", "f32"])
def test_tile_segments(kind, max_sweeps, restarts, R):
    _compare([_segment_instance(kind)], [R], R, kind != "f32", max_sweeps=max_sweeps, restarts=restarts,
             refresh_every=3, kernel=isg.KERNEL_MSC if kind in ("lattice", "msc") else isg.KERNEL_TILE)


def test_tile_segments_uneven_batch_and_sequential_schedule():
    insts = [W.random_graph(n, 4.0, 60 + n, dtype="f32", n_hyper=n // 9) for n in (1, 40, 300)]
    _compare(insts, [1, 2, 3], 34, False, max_sweeps=200, restarts=9, schedule=isg.SCHED_SEQUENTIAL,
             kernel=isg.KERNEL_TILE)


# Tile energies, a lane per spin: fewer spins than lanes and one more than a CTA's
# threads, hyper-edges of 2 to 9 members, the highest replica alone in its group of
# 8, and exponents too far apart for one unit or for a lane's sum.
@pytest.mark.parametrize("n,R", [(1, 1), (33, 9), (257, 17), (1025, 32)])
@pytest.mark.parametrize("kind", ["i8", "f32", "wide", "wider"])
def test_tile_energy_sums(kind, n, R):
    inst = W.random_graph(n, 5.0 if n > 1 else 0.0, n, dtype="i8" if kind == "i8" else "f32",
                          n_hyper=n // 4, hyper_order=(2, 3, 4, 9))
    if kind.startswith("wide"):
        inst = _exp_spread(inst, *((-12, 12) if kind == "wide" else (-45, 25)))
    for restarts, max_sweeps in ((1, 100), (3, 2)):
        _compare([inst], [n], R, kind == "i8", max_sweeps=max_sweeps, restarts=restarts, kernel=isg.KERNEL_TILE)


# Tile visits, eight spins at a time: classes of fewer and more spins than that,
# rows of more than the entries fetched together, hyper-edges of 2 to 9 members,
# refreshes in fixed point, in FP64 and (wider) both in one class.
@pytest.mark.parametrize("n,R,schedule", [(7, 5, isg.SCHED_COLOUR), (100, 32, isg.SCHED_COLOUR),
                                          (300, 41, isg.SCHED_COLOUR), (3000, 9, isg.SCHED_COLOUR),
                                          (7, 32, isg.SCHED_SEQUENTIAL), (100, 8, isg.SCHED_SEQUENTIAL)])
@pytest.mark.parametrize("kind", ["i8", "f32", "wide", "wider"])
def test_tile_visits(kind, n, R, schedule):
    dtype = "i8" if kind == "i8" else "f32"
    inst = (_star_graph(n, dtype, n) if n >= 100 else
            W.random_graph(n, 3.0, n, dtype=dtype, n_hyper=3, hyper_order=(2, 3, 4)))
    if kind.startswith("wide"):
        inst = _exp_spread(inst, *((-12, 12) if kind == "wide" else (-45, 25)))
    _compare([inst], [n], R, kind == "i8", max_sweeps=200, restarts=2, refresh_every=3, schedule=schedule,
             kernel=isg.KERNEL_TILE)


# Tile results in whole words of spins and (an odd address, an odd size) byte by byte.
@pytest.mark.parametrize("kind,n", [("i8", 96), ("f32", 96), ("f32", 97), ("i8", 32)])
def test_tile_result_addresses(kind, n):
    inst = W.random_graph(n, 4.0, n, dtype=kind)
    o, _ = _oracle([inst], [n], 35, max_sweeps=100, restarts=2)
    h = isg.Handle([inst])
    kw = dict(max_sweeps=100, restarts=2, kernel=isg.KERNEL_TILE)
    ref = h.local_search([n], 35, **kw)
    for at in (0, 1, 16):
        buf = torch.zeros(35 * n + 16, dtype=torch.int8, device="cuda")[at:at + 35 * n]
        h.local_search([n], 35, out=(buf, ref.energy.clone(), None, ref.minima.clone()), **kw)
        assert np.array_equal(buf.cpu().numpy().reshape(35, n), np.asarray(o[0][0]).reshape(35, n))
    h.close()


# Lattice clusters: every cluster size, both dimensions, rows shorter than, as long
# as and longer than a chunk, slabs of one plane, signs in planes and (slabs of
# 16,384 sites) packed; segments of descents with none, some and all converged;
# results written to an odd address.
@pytest.mark.parametrize("dims,ctas", [((16, 16, 16), 2), ((16, 16, 16), 4), ((32, 32, 32), 2), ((32, 32, 32), 8),
                                       ((64, 64), 4), ((64, 64), 2), ((128, 128), 8), ((128, 128), 2)])
@pytest.mark.parametrize("max_sweeps,restarts,R", [(1, 5, 33), (5, 3, 7), (200, 4, 40)])
def test_lattice_cluster_segments(dims, ctas, max_sweeps, restarts, R):
    inst = W.lattice(dims, True, "pm1", "pm1_0" if dims[0] != 64 else None, seed=dims[0])
    if max_sweeps == 1 and R == 33:
        h = isg.Handle([inst])
        kw = dict(max_sweeps=max_sweeps, restarts=restarts, kernel=isg.KERNEL_MSC, cluster_ctas=ctas)
        ref = h.local_search([R], R, **kw)
        buf = torch.zeros(R * inst.n + 1, dtype=torch.int8, device="cuda")[1:]
        h.local_search([R], R, out=(buf, ref.energy.clone(), None, ref.minima.clone()), **kw)
        assert torch.equal(buf, ref.spins)
        h.close()
    g, gst, _ = _run([inst], [R], R, max_sweeps=max_sweeps, restarts=restarts, kernel=isg.KERNEL_MSC, cluster_ctas=ctas)
    o, ost = _oracle([inst], [R], R, max_sweeps=max_sweeps, restarts=restarts)
    for k in range(3):
        assert np.array_equal(g[0][k], o[0][k])
    assert {k: gst[k] for k in ost} == ost


# The planner's line between one CTA per tile and launches over the whole GPU:
# the same results on both sides of it.
@pytest.mark.parametrize("n", [2000, 12000])
def test_auto_family_of_one_general_graph(n):
    inst = W.random_graph(n, 5.0, 61, dtype="f32", n_hyper=n // 8, hyper_order=(3, 4))
    kw = dict(max_sweeps=300, restarts=2)
    h = isg.Handle([inst])
    assert h.plan_kernel(6, **kw) == (isg.KERNEL_TILE if n == 2000 else isg.KERNEL_SWEEP)
    h.close()
    _compare([inst], [n], 6, False, **kw)


# ising_energy: one-CTA instances (handles of up to 1024 spins) and larger ones in
# parts of 256 sites (below: others of both); 4, 16 and 32 replicas per word group and their remainders; sizes
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


# A warp's lone pending FP32 spin (classes of one spin: fully coupled rows) and two
# and three of them, with refreshes in fixed point, in FP64 and none but the first.
@pytest.mark.parametrize("refresh_every", [0, 1, 3])
@pytest.mark.parametrize("per_class", [1, 2, 3])
@pytest.mark.parametrize("kind", ["f32", "wide", "wider"])
def test_tile_lone_spins(kind, per_class, refresh_every):
    n = 40 * per_class
    u, v = np.triu_indices(n, 1)
    keep = u // per_class != v // per_class  # (spins of one class are not coupled)
    u, v = u[keep], v[keep]
    rng = np.random.default_rng(per_class)
    rp, col, J = W.csr_from_edges(n, u, v, rng.standard_normal(len(u)).astype(np.float32), "f32")
    cls = rng.permutation(n // per_class)
    hyper = np.array([[0, per_class, 2 * per_class], [per_class, 3 * per_class, 4 * per_class]], np.int32).ravel()
    inst = W.Instance(n=n, row_ptr=rp, col=col, J=J, h=rng.standard_normal(n).astype(np.float32),
                      hyper_ptr=np.array([0, 3, 6], np.int64), hyper_members=hyper,
                      hyper_J=np.array([0.5, -0.25], np.float32),
                      colour=cls[np.arange(n) // per_class].astype(np.int32), dtype="f32")
    if kind != "f32":
        inst = _exp_spread(inst, *((-12, 12) if kind == "wide" else (-45, 25)))
    _compare([inst], [n], 37, False, max_sweeps=200, restarts=2, refresh_every=refresh_every, kernel=isg.KERNEL_TILE)


# The index order: sizes around a warp's batch of 32, one segment and several, more
# tiles than CTAs fit, and both orders in turn on one handle.
@pytest.mark.parametrize("restarts,R", [(1, 33), (5, 4)])
@pytest.mark.parametrize("n", [1, 31, 32, 33, 65, 300])
@pytest.mark.parametrize("kind", ["i8", "f32", "wider", "msc"])
def test_tile_index_order(kind, n, restarts, R):
    if kind == "msc":
        inst = W.random_graph(n, min(4.0, n - 1.0), n, dtype="i8", int_range=1, fields=False)
    else:
        inst = W.random_graph(n, min(5.0, n - 1.0), n, dtype="i8" if kind == "i8" else "f32",
                              n_hyper=n // 6, hyper_order=(2, 3, 4))
        inst = _exp_spread(inst, -45, 25) if kind == "wider" else inst
    _compare([inst], [n], R, kind in ("i8", "msc"), max_sweeps=200, restarts=restarts, refresh_every=3,
             schedule=isg.SCHED_SEQUENTIAL, kernel=isg.KERNEL_MSC if kind == "msc" else isg.KERNEL_TILE)


@pytest.mark.parametrize("dtype", ["i8", "f32"])
def test_tile_index_order_of_more_tiles_than_ctas(dtype):
    insts = [W.random_graph(3 + b % 9, 2.0, b, dtype=dtype) for b in range(1300)]
    _compare(insts, list(range(1, 1301)), 3, dtype == "i8", max_sweeps=50, restarts=2,
             schedule=isg.SCHED_SEQUENTIAL, kernel=isg.KERNEL_TILE)


def test_tile_both_orders_on_one_handle():
    inst = W.random_graph(200, 5.0, 8, dtype="f32", n_hyper=20)
    h = isg.Handle([inst])
    for schedule in (isg.SCHED_COLOUR, isg.SCHED_SEQUENTIAL) * 2:
        r = h.local_search([3], 40, max_sweeps=200, restarts=2, schedule=schedule, kernel=isg.KERNEL_TILE)
        s, _, m, _ = oracle.descent(inst, 3, 0, 40, max_sweeps=200, restarts=2, schedule=schedule)
        assert np.array_equal(r.spins.cpu().numpy().reshape(40, -1), s)
        assert np.array_equal(r.minima[0].cpu().numpy(), m)
    h.close()


# FP32 lattices on both sides of the rule between groups of 16 and of 32 replicas
# (three groups of 16; few sites; many), odd and even sides, last groups of one.
@pytest.mark.parametrize("dims,R", [((41, 41, 41), 17), ((41, 41, 41), 33), ((260, 260), 18), ((34, 34, 34), 49),
                                    ((20, 20, 20), 100), ((12, 12, 12), 400), ((16, 16, 16), 513)])
def test_sweep_fp32_lattice_group_sizes(dims, R):
    inst = W.lattice(dims, True, "gauss", "gauss", seed=R)
    _compare([inst], [R], R, False, max_sweeps=12, restarts=2, refresh_every=5, kernel=isg.KERNEL_SWEEP)


# ... and the shapes those do not reach: lattices in one CTA, many instances of up
# to 2048 spins (one CTA each), parts of more than one site a thread with a ragged
# last one (lattices of both dimensions, rows walked by a thread and by a warp).
def _check_energies(insts, R, rtol):
    h = isg.Handle(insts)
    spins = (np.random.default_rng(R).integers(0, 2, size=R * h.total_spins) * 2 - 1).astype(np.int8)
    dev = torch.from_numpy(spins).cuda()
    for _ in range(2):
        E = h.energy(dev, R).cpu().numpy()
    off = 0
    for b, inst in enumerate(insts):
        ref = oracle.energies(inst, spins[off: off + R * inst.n].reshape(R, inst.n))
        off += R * inst.n
        if inst.dtype == "i8":
            assert np.array_equal(E[b], ref)
        else:
            np.testing.assert_allclose(E[b], ref, rtol=rtol, atol=1e-9)
    h.close()


@pytest.mark.parametrize("R", [1, 6, 33])
@pytest.mark.parametrize("J", ["pm1", "gauss"])
@pytest.mark.parametrize("dims", [(3, 3), (31, 31), (32, 32), (10, 10, 10)])
def test_energy_lattice_in_one_cta(dims, J, R):
    _check_energies([W.lattice(dims, True, J, "pm1_0" if J == "pm1" else "gauss", seed=sum(dims))], R, 1e-12)


@pytest.mark.parametrize("kind", ["lattice", "i8", "f32"])
def test_energy_many_instances_of_one_cta(kind):
    rng = np.random.default_rng(7)
    if kind == "lattice":
        insts = [W.lattice((L, L), True, "gauss", "gauss", seed=L) for L in list(range(33, 46)) * 12]
    else:
        insts = [W.random_graph(int(n), 3.0, int(n), dtype=kind, n_hyper=50, hyper_order=(2, 3, 5))
                 for n in np.concatenate([[1025, 2047, 2048], rng.integers(1025, 2049, size=21)])] * 7
    _check_energies(insts, 2, 1e-12)


@pytest.mark.parametrize("dims,J,R", [((45, 45, 45), "gauss", 40), ((64, 64, 64), "pm1", 33), ((90, 90, 90), "gauss", 5),
                                      ((701, 701), "pm1", 17)])
def test_energy_lattice_large_parts(dims, J, R):
    # (a relative bound on sums of up to 3e6 terms of order one that partly cancel)
    _check_energies([W.lattice(dims, True, J, "pm1_0" if J == "pm1" else None, seed=R)], R, 1e-10)


@pytest.mark.parametrize("dtype,R", [("i8", 40), ("f32", 70)])
def test_energy_graph_large_parts(dtype, R):
    n = 90001
    rng = np.random.default_rng(n)
    key = np.unique(rng.integers(0, n, size=3 * n) * np.int64(n) + rng.integers(0, n, size=3 * n))
    u, v = key // n, key % n
    lo, hi = np.minimum(u, v), np.maximum(u, v)
    key = np.unique((lo * np.int64(n) + hi)[lo != hi])
    u, v = key // n, key % n
    w = rng.standard_normal(len(u)).astype(np.float32) if dtype == "f32" else \
        (rng.integers(1, 128, size=len(u)) * (rng.integers(0, 2, size=len(u)) * 2 - 1)).astype(np.int8)
    for hub in (False, True):  # (a hub: rows by warps)
        if hub:
            keep = (u != 17) & (v != 17)
            ends = np.arange(18, n, 3)
            u, v = np.concatenate([u[keep], np.full(len(ends), 17)]), np.concatenate([v[keep], ends])
            w = np.concatenate([w[keep], np.resize(w, len(ends))])
        rp, col, J = W.csr_from_edges(n, u, v, w, dtype)
        h = np.resize(w, n).astype(w.dtype)
        _check_energies([W.Instance(n=n, row_ptr=rp, col=col, J=J, h=h, dtype=dtype)], R, 1e-10)


# Results of the sweep family in whole words of spins and (an odd address, an odd
# size) byte by byte: groups of 8, 16 and 32, a last one partly filled, results of
# converged descents and of some that never converge.
@pytest.mark.parametrize("max_sweeps", [3, 200])
@pytest.mark.parametrize("R", [5, 16, 33, 70])
@pytest.mark.parametrize("kind,n", [("i8", 96), ("f32", 96), ("f32", 97), ("pm1", 512), ("gauss", 343)])
def test_sweep_result_addresses(kind, n, R, max_sweeps):
    if kind in ("pm1", "gauss"):
        inst = W.lattice((round(n ** (1 / 3)),) * 3, True, kind, None, seed=n)
    else:
        inst = W.random_graph(n, 4.0, n, dtype=kind)
    kw = dict(max_sweeps=max_sweeps, restarts=2, kernel=isg.KERNEL_SWEEP)
    _, o = _compare([inst], [n], R, inst.dtype == "i8", **kw)
    h = isg.Handle([inst])
    ref = h.local_search([n], R, **kw)
    for at in (0, 1, 8, 16):
        buf = torch.zeros(R * n + 16, dtype=torch.int8, device="cuda")[at:at + R * n]
        h.local_search([n], R, out=(buf, ref.energy.clone(), None, ref.minima.clone()), **kw)
        assert np.array_equal(buf.cpu().numpy().reshape(R, n), o[0][0])
    h.close()


# Both sides of the size up to which a tile's energies and few pending spins are the
# whole warp's.
@pytest.mark.parametrize("R", [9, 33])
@pytest.mark.parametrize("n", [80, 81])
@pytest.mark.parametrize("kind", ["i8", "f32", "wide", "wider"])
def test_tile_few_spins(kind, n, R):
    inst = W.random_graph(n, 5.0, n, dtype="i8" if kind == "i8" else "f32", n_hyper=n // 4, hyper_order=(2, 3, 4, 9))
    if kind.startswith("wide"):
        inst = _exp_spread(inst, *((-12, 12) if kind == "wide" else (-45, 25)))
    for restarts, max_sweeps in ((1, 100), (3, 2)):
        _compare([inst] * 2, [n, 7], R, kind == "i8", max_sweeps=max_sweeps, restarts=restarts, refresh_every=3,
                 kernel=isg.KERNEL_TILE)
