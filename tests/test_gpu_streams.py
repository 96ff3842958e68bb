"""Calls on the caller's own streams: what a handle builds on a first call is in
place before that call's kernels read it, whatever else the GPU is doing.

The caller's stream is non-blocking (every torch.cuda.Stream is), so nothing
orders it after the default stream, which is kept busy with ordinary work here.
Results are compared with the CPU oracle."""
import numpy as np
import pytest

import oracle
import workloads as W

torch = pytest.importorskip("torch")
pytestmark = pytest.mark.gpu

isg = pytest.importorskip("paper_0912_3912_gb300")

from test_gpu_parity import _exp_spread  # noqa: E402


@pytest.fixture(scope="module", autouse=True)
def _built():
    if not torch.cuda.is_available():
        pytest.skip("no GPU")
    from paper_0912_3912_gb300 import build as B
    B.build()
    oracle.build()


@pytest.fixture(scope="module")
def busy():
    """Queue some 50 ms of copies on the default stream."""
    a = torch.zeros(1 << 28, dtype=torch.float32, device="cuda")
    b = torch.empty_like(a)

    def go():
        torch.cuda.synchronize()
        with torch.cuda.stream(torch.cuda.default_stream()):
            for _ in range(150):
                b.copy_(a)
    return go


def _energy_instance(kind):
    if kind == "lattice":
        return W.lattice((14, 14, 14), True, "pm1", "pm1_0", seed=14)
    g = W.random_graph(5000, 5.0, 5, dtype="f32", n_hyper=300, hyper_order=(2, 3))
    return _exp_spread(g, -45, 25) if kind == "wide" else g  # (wide: the FP64 passes)


def _check_energy(inst, spins, E):
    ref = oracle.energies(inst, spins)
    if inst.dtype == "i8":
        assert np.array_equal(E.cpu().numpy()[0], ref)
    else:  # exact sums rounded once (wide: FP64 sums); the oracle's are FP64
        np.testing.assert_allclose(E.cpu().numpy()[0], ref, rtol=1e-12, atol=1e-9)


@pytest.mark.parametrize("kind", ["lattice", "graph", "wide"])
def test_first_energy_call_on_a_side_stream(kind, busy):
    inst = _energy_instance(kind)
    h = isg.Handle([inst])
    side = torch.cuda.Stream()
    for R in (33, 5):  # (a new replica count builds anew)
        spins = (np.random.default_rng(R).integers(0, 2, size=(R, inst.n)) * 2 - 1).astype(np.int8)
        dev = torch.from_numpy(spins).cuda()
        busy()
        with torch.cuda.stream(side):
            E = [h.energy(dev, R) for _ in range(2)]
        side.synchronize()
        for e in E:
            _check_energy(inst, spins, e)
    torch.cuda.synchronize()
    h.close()


# A first call that is only captured builds what the handle keeps all the same.
@pytest.mark.parametrize("kind", ["lattice", "graph", "wide"])
def test_first_energy_call_under_capture(kind):
    inst = _energy_instance(kind)
    R = 9
    spins = (np.random.default_rng(R).integers(0, 2, size=(R, inst.n)) * 2 - 1).astype(np.int8)
    dev = torch.from_numpy(spins).cuda()
    h = isg.Handle([inst])
    g = torch.cuda.CUDAGraph()
    with torch.cuda.graph(g, capture_error_mode="relaxed"):
        captured = h.energy(dev, R)
    _check_energy(inst, spins, h.energy(dev, R))
    for _ in range(2):
        g.replay()
    _check_energy(inst, spins, captured)
    torch.cuda.synchronize()
    del g
    h.close()


# First searches of a fresh handle, family by family: the instance's own copies,
# work lists and zeroed buffers; the dense family against a second call.
@pytest.mark.parametrize("kind", ["tile", "msc", "cluster", "sweep", "passes", "dense", "dense_library"])
def test_first_search_on_a_side_stream(kind, busy):
    if kind == "tile":
        inst, R, kw = W.random_graph(500, 5.0, 3, dtype="f32", n_hyper=40), 40, dict(kernel=isg.KERNEL_TILE)
    elif kind == "sweep":
        inst, R, kw = W.random_graph(500, 5.0, 4, dtype="i8", n_hyper=40), 20, dict(kernel=isg.KERNEL_SWEEP)
    elif kind == "passes":
        inst, R, kw = W.random_graph(400, 5.0, 6, dtype="f32", n_hyper=40), 6, {}
    elif kind.startswith("dense"):
        inst, R = W.sk(300, seed=8), 70
        kw = dict(kernel=isg.KERNEL_DENSE_TC, schedule=isg.SCHED_SEQUENTIAL,
                  dense_variant=isg.DENSE_LIBRARY if kind == "dense_library" else isg.DENSE_OWN)
    else:
        inst = W.lattice((16, 16, 16), True, "pm1", "pm1_0", seed=9)
        R, kw = 33, dict(kernel=isg.KERNEL_MSC, cluster_ctas=1 if kind == "msc" else 4)
    side = torch.cuda.Stream()
    busy()
    h = isg.Handle([inst])
    with torch.cuda.stream(side):
        if kind == "passes":
            spins, E, extra, _ = h.fm_search([5], R, stats=False)
        else:
            r = h.local_search([5], R, max_sweeps=200, stats=False, **kw)
            spins, E, extra = r.spins, r.energy, r.minima
    side.synchronize()
    spins, E = spins.cpu().numpy().reshape(R, inst.n), E[0].cpu().numpy()
    extra = extra[0].cpu().numpy()
    torch.cuda.synchronize()
    if kind == "passes":
        for k in range(R):
            s, e, p = oracle.fm_search(inst, oracle.random_start(inst.n, 5, 0, k, 0))
            assert np.array_equal(spins[k], s) and extra[k] == p
            assert abs(E[k] - e) <= 1e-9 * (1 + abs(e))
    elif kind.startswith("dense"):
        again = h.local_search([5], R, max_sweeps=200, **kw)
        assert np.array_equal(spins, again.spins.cpu().numpy().reshape(R, inst.n))
        assert np.array_equal(E, again.energy[0].cpu().numpy())
    else:
        s, e, m, _ = oracle.descent(inst, 5, 0, R, max_sweeps=200)
        assert np.array_equal(spins, s) and np.array_equal(extra, m)
        np.testing.assert_allclose(E, e, rtol=1e-9, atol=1e-9)
    h.close()


# The same for the pass-based search, whose first call builds the move records:
# that call is captured and never run.
@pytest.mark.parametrize("dtype", ["i8", "f32"])
def test_first_passes_call_under_capture(dtype):
    inst = W.random_graph(300, 5.0, 12, dtype=dtype, n_hyper=40, hyper_order=(2, 3))
    R = 4
    h = isg.Handle([inst])
    g = torch.cuda.CUDAGraph()
    with torch.cuda.graph(g, capture_error_mode="relaxed"):
        h.fm_search([5], R, stats=False)
    torch.cuda.synchronize()
    del g
    spins, E, passes, _ = h.fm_search([5], R)
    spins = spins.cpu().numpy().reshape(R, inst.n)
    for k in range(R):
        s, e, p = oracle.fm_search(inst, oracle.random_start(inst.n, 5, 0, k, 0))
        assert np.array_equal(spins[k], s) and int(passes[0, k]) == p
        assert abs(float(E[0, k]) - e) <= 1e-9 * (1 + abs(e))
    h.close()


# A search without work counters returns to the host once it is queued where one
# kernel serves the instance: also for the few large instances that AUTO gives to the
# sweep family, whose sweeps then loop on the device.  Chunks of 16 sweeps and of
# fewer (by the colour classes), budgets, searches that end in the first chunk and
# that never converge, several instances, both value types; twice on one handle.
def _auto_case(kind):
    if kind == "classes":  # 68 colour classes: chunks of 4 sweeps
        n = 25000
        rng = np.random.default_rng(3)
        u = rng.integers(0, n, size=n)
        v = (u + rng.integers(1, n, size=n)) % n
        colour = rng.integers(0, 68, size=n).astype(np.int32)
        key = np.unique((np.minimum(u, v) * np.int64(n) + np.maximum(u, v))[colour[u] != colour[v]])
        w = rng.integers(1, 4, size=len(key)).astype(np.int8)
        rp, col, J = W.csr_from_edges(n, key // n, key % n, w, "i8")
        return [W.Instance(n=n, row_ptr=rp, col=col, J=J, colour=colour, dtype="i8")], 3, dict(max_sweeps=30)
    if kind == "square":
        return [W.lattice((150, 150), True, "gauss", "gauss", seed=2)], 21, dict(max_sweeps=300, restarts=3)
    if kind == "two":
        return [W.lattice((140 + k, 140 + k), True, "gauss", None, seed=k) for k in range(2)], 5, \
            dict(max_sweeps=300, restarts=2)
    inst = W.random_graph(12000, 5.0, 61, dtype="i8" if kind == "int" else "f32", n_hyper=1500, hyper_order=(3, 4))
    return [inst], 6, {"budget": dict(max_sweeps=300, restarts=50, sweep_budget=45), "one": dict(max_sweeps=1),
                       "capped": dict(max_sweeps=3, restarts=2)}.get(kind, dict(max_sweeps=300, restarts=2))


@pytest.mark.parametrize("kind", ["graph", "int", "square", "two", "budget", "one", "capped", "classes"])
def test_auto_search_without_stats_does_not_hold_the_host(kind, busy):
    insts, R, kw = _auto_case(kind)
    seeds = list(range(5, 5 + len(insts)))
    h = isg.Handle(insts)
    assert h.plan_kernel(R, **kw) == isg.KERNEL_SWEEP
    h.local_search(seeds, R, stats=False, **kw)  # (builds its graph and scratch)
    before = torch.cuda.Event()
    busy()
    before.record()
    r = h.local_search(seeds, R, stats=False, **kw)
    held = before.query()
    waited = h.local_search(seeds, R, **kw)
    again = h.local_search(seeds, R, stats=False, **kw)
    torch.cuda.synchronize()
    for b, inst in enumerate(insts):
        s, e, m, _ = oracle.descent(inst, seeds[b], b, R, **kw)
        for got in (r, waited, again):
            assert np.array_equal(h.spins_of(got.spins, b, R).cpu().numpy(), s)
            assert np.array_equal(got.minima[b].cpu().numpy(), m)
            np.testing.assert_allclose(got.energy[b].cpu().numpy(), e, rtol=1e-9, atol=1e-9)
    assert not held, "the call held the host until the stream had caught up"
    h.close()


def test_auto_search_without_stats_is_refused_under_capture():
    insts, R, kw = _auto_case("graph")
    h = isg.Handle(insts)
    ref = h.local_search([5], R, stats=False, **kw)
    side = torch.cuda.Stream()
    g = torch.cuda.CUDAGraph()
    torch.cuda.synchronize()
    with torch.cuda.stream(side):
        g.capture_begin(capture_error_mode="relaxed")
        with pytest.raises(isg.IsingError):
            h.local_search([5], R, stats=False, out=(ref.spins, ref.energy, None, ref.minima), **kw)
        g.capture_end()
    del g
    r = h.local_search([5], R, stats=False, **kw)
    assert torch.equal(r.spins, ref.spins)
    h.close()


# A handle closed, and one whose scratch grows, while such a search still runs.
def test_auto_search_without_stats_outlives_nothing_it_needs(busy):
    insts, R, kw = _auto_case("graph")
    s, _, m, _ = oracle.descent(insts[0], 5, 0, R, **kw)
    s40, _, _, _ = oracle.descent(insts[0], 6, 0, 40, **kw)
    for close in (True, False):
        h = isg.Handle(insts)
        h.local_search([5], R, stats=False, **kw)
        busy()
        r = h.local_search([5], R, stats=False, **kw)
        if close:
            h.close()
        else:
            wider = h.local_search([6], 40, stats=False, **kw)
        torch.cuda.synchronize()
        assert np.array_equal(r.spins.cpu().numpy().reshape(R, -1), s)
        assert np.array_equal(r.minima[0].cpu().numpy(), m)
        if not close:
            assert np.array_equal(wider.spins.cpu().numpy().reshape(40, -1), s40)
            h.close()


# Two handles of one kernel and different sizes, from two host threads: neither
# changes what the other may launch.
def test_cluster_launches_of_two_sizes_from_two_threads():
    import threading
    cases = [(W.lattice((32, 32, 32), True, "pm1", seed=1), 8), (W.lattice((16, 16, 16), True, "pm1", seed=2), 4)]
    failures, results = [], {}

    def work(k):
        inst, ctas = cases[k]
        kw = dict(max_sweeps=2, kernel=isg.KERNEL_MSC, cluster_ctas=ctas, stats=False)
        try:
            h = isg.Handle([inst])
            out = None
            wide = (torch.empty(64 * inst.n, dtype=torch.int8, device="cuda"),
                    torch.empty((1, 64), dtype=torch.float64, device="cuda"), None,
                    torch.empty((1, 64), dtype=torch.int32, device="cuda"))
            with torch.cuda.stream(torch.cuda.Stream()):
                for i in range(4000):
                    if k and i % 2:  # (the small one is planned anew for every call)
                        h.local_search([7], 64, out=wide, **kw)
                        continue
                    r = h.local_search([7], 32, out=out, **kw)
                    out = (r.spins, r.energy, None, r.minima)
            torch.cuda.synchronize()
            results[k] = r.spins.cpu().numpy()
            h.close()
        except Exception as e:  # noqa: BLE001 (reported by the main thread)
            failures.append(e)

    threads = [threading.Thread(target=work, args=(k,)) for k in range(2)]
    for t in threads:
        t.start()
    for t in threads:
        t.join()
    assert not failures, failures
    for k, (inst, _) in enumerate(cases):
        s, _, _, _ = oracle.descent(inst, 7, 0, 32, max_sweeps=2)
        assert np.array_equal(results[k].reshape(32, inst.n), s)
