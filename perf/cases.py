"""What a user of this library has it do: local searches (descent with restarts),
pass-based searches and energies of given configurations, each through the
package's public calls (Handle.local_search, Handle.fm_search, Handle.energy).

listed() holds the cases, draw(rng) gives more of the same ranges, prepare(case,
seed) builds the instance and its handle, run(state) is one call, work(case) says
what a call cannot do without and exact(case, seed) gives the energies a call
returns, from 64-bit arithmetic without the library, where that is quick.
"""
from types import SimpleNamespace

import numpy as np
import torch

import paper_0912_3912_gb300 as isg

DESCENTS = 1 << 30  # "until the sweep budget is used up"


def listed():
    return [
        # One small planar instance, few replicas: the latency of a call (a
        # user's inner loop over many small problems).
        dict(name="descent_square16_pm1", op="descent", graph="lattice", d=2, L=16, J="pm1", field=False,
             R=64, restarts=10, max_sweeps=1000, budget=0),
        # A 3D +/-J glass with integer fields, many replicas: sampling low
        # energies of one mid-size instance.
        dict(name="descent_cube32_pm1_field", op="descent", graph="lattice", d=3, L=32, J="pm1", field=True,
             R=1024, restarts=10, max_sweeps=100, budget=0),
        # Many uneven hardware-graph instances at once, Gaussian couplings and
        # 3-spin terms: a batch of problems for one annealer topology.
        dict(name="descent_chimera_batch", op="descent", graph="chimera", count=1024, lo=4, hi=16,
             R=32, restarts=1, max_sweeps=1000, budget=0),
        # A fully connected Gaussian glass in the paper's sequential order.
        dict(name="descent_sk4096", op="descent", graph="sk", n=4096, R=4096, restarts=1, max_sweeps=1000, budget=0),
        # The million-spin Gaussian lattice under a sweep budget: throughput.
        dict(name="descent_cube100_gauss", op="descent", graph="lattice", d=3, L=100, J="gauss", field=False,
             R=16, restarts=DESCENTS, max_sweeps=1000, budget=1000),
        # The same size with +/-1 couplings.
        dict(name="descent_cube100_pm1", op="descent", graph="lattice", d=3, L=100, J="pm1", field=False,
             R=16, restarts=DESCENTS, max_sweeps=1000, budget=1000),
        # An odd side (no checkerboard, so more than two colour classes), fields
        # and a replica count that fills no power of two.
        dict(name="descent_cube45_odd", op="descent", graph="lattice", d=3, L=45, J="gauss", field=True,
             R=21, restarts=4, max_sweeps=1000, budget=0),
        # A random sparse graph with 3- and 4-spin terms beyond one CTA's
        # memory: the general path.
        dict(name="descent_graph_hyper", op="descent", graph="random", n=60013, degree=6, hyper=15000, J="gauss",
             R=40, restarts=2, max_sweeps=1000, budget=0),
        # Pass-based search, small integer instance: 64 x 10 starts.
        dict(name="passes_square16_pm1", op="passes", graph="lattice", d=2, L=16, J="pm1", field=False,
             R=64, restarts=10),
        # Pass-based search at the size of the paper's 50 x 50 timing: few long
        # searches, so the latency of one move.
        dict(name="passes_square50_gauss", op="passes", graph="lattice", d=2, L=50, J="gauss", field=False,
             R=61, restarts=1),
        # Pass-based search over a batch of uneven hardware-graph instances.
        dict(name="passes_chimera_batch", op="passes", graph="chimera", count=128, lo=4, hi=16, R=32, restarts=1),
        # Energies of given configurations of the million-spin lattice.
        dict(name="energy_cube100_gauss", op="energy", graph="lattice", d=3, L=100, J="gauss", field=False, R=16),
    ]


def _log(rng, lo, hi):
    """A whole number in [lo, hi], even over its logarithm."""
    return max(lo, min(hi, int(round(lo * (hi / lo) ** rng.random()))))


def draw(rng):
    kind = rng.randrange(9)
    J = rng.choice(["pm1", "gauss"])
    field = rng.random() < 0.5
    if kind == 0:  # small planar instances
        return dict(op="descent", graph="lattice", d=2, L=_log(rng, 5, 128), J=J, field=field, R=_log(rng, 1, 256),
                    restarts=_log(rng, 1, 10), max_sweeps=1000, budget=0)
    if kind == 1:  # mid-size cubes, many replicas
        return dict(op="descent", graph="lattice", d=3, L=_log(rng, 8, 32), J="pm1", field=field,
                    R=_log(rng, 32, 1024), restarts=_log(rng, 1, 10), max_sweeps=100, budget=0)
    if kind == 2:  # large cubes under a sweep budget
        L = _log(rng, 34, 100)
        cap = (16 if L % 2 == 0 else 8) * 10**6
        return dict(op="descent", graph="lattice", d=3, L=L, J=J, field=field, R=min(_log(rng, 3, 64), cap // L**3),
                    restarts=DESCENTS, max_sweeps=1000, budget=_log(rng, 100, 1000))
    if kind == 3:
        lo = rng.randint(4, 12)
        return dict(op="descent", graph="chimera", count=_log(rng, 1, 1024), lo=lo, hi=rng.randint(lo, 16),
                    R=_log(rng, 1, 32), restarts=1, max_sweeps=1000, budget=0)
    if kind == 4:
        return dict(op="descent", graph="sk", n=_log(rng, 128, 4096), R=_log(rng, 32, 4096), restarts=1,
                    max_sweeps=1000, budget=0)
    if kind == 5:
        n = _log(rng, 200, 60000)
        return dict(op="descent", graph="random", n=n, degree=rng.randint(3, 6), hyper=int(n * rng.random() / 4),
                    J=rng.choice(["int", "gauss"]), R=_log(rng, 1, 64), restarts=_log(rng, 1, 4), max_sweeps=1000,
                    budget=0)
    if kind == 6:
        return dict(op="passes", graph="lattice", d=2, L=_log(rng, 6, 50), J=J, field=field, R=_log(rng, 1, 64),
                    restarts=_log(rng, 1, 10))
    if kind == 7:
        lo = rng.randint(4, 12)
        return dict(op="passes", graph="chimera", count=_log(rng, 1, 128), lo=lo, hi=rng.randint(lo, 16),
                    R=_log(rng, 1, 32), restarts=1)
    g = rng.randrange(3)
    if g == 0:
        return dict(op="energy", graph="lattice", d=3, L=_log(rng, 10, 100), J=J, field=field, R=_log(rng, 1, 16))
    if g == 1:
        return dict(op="energy", graph="chimera", count=_log(rng, 1, 256), lo=4, hi=16, R=_log(rng, 1, 32))
    n = _log(rng, 200, 60000)
    return dict(op="energy", graph="random", n=n, degree=rng.randint(3, 6), hyper=int(n * rng.random() / 4),
                J=rng.choice(["int", "gauss"]), R=_log(rng, 1, 64))


# ------------------------------------------------------------------ instances
def _instance(n, row_ptr, col, J, h=None, hyper=None, colour=None, J_dense=None):
    """The argument of isg.Handle: symmetric CSR couplings (or a dense matrix)."""
    hp, hm, hJ = hyper if hyper is not None else (None, None, None)
    f32 = J_dense is not None or J.dtype == np.float32
    return SimpleNamespace(n=n, row_ptr=row_ptr, col=col, J=J, J_dense=J_dense, h=h, hyper_ptr=hp,
                           hyper_members=hm, hyper_J=hJ, colour=colour, dtype="f32" if f32 else "i8")


def _csr(n, u, v, w):
    """Symmetric CSR, rows sorted by column, of distinct edges u-v."""
    row, col, val = np.concatenate([u, v]), np.concatenate([v, u]), np.concatenate([w, w])
    order = np.argsort(row * np.int64(n) + col, kind="stable")
    row_ptr = np.zeros(n + 1, np.int64)
    np.cumsum(np.bincount(row, minlength=n), out=row_ptr[1:])
    return row_ptr, col[order].astype(np.int32), val[order]


def _draw_J(rng, kind, size):
    if kind == "gauss":
        return rng.standard_normal(size, dtype=np.float32)
    if kind == "pm1":
        return (rng.integers(0, 2, size=size, dtype=np.int8) * 2 - 1).astype(np.int8)
    return (rng.integers(1, 4, size=size, dtype=np.int8) * (rng.integers(0, 2, size=size, dtype=np.int8) * 2 - 1))


def _lattice_bonds(c, rng):
    """Periodic hypercubic lattice: per axis the +1 neighbour of every site and the bond to it."""
    n, L = c["L"] ** c["d"], c["L"]
    idx = np.arange(n, dtype=np.int64)
    nb, w = [], []
    for a in range(c["d"]):
        x = idx // L**a % L
        nb.append(idx + ((x + 1) % L - x) * L**a)
        w.append(_draw_J(rng, c["J"], n))
    return nb, w


def _field(c, rng, n):
    if not c["field"]:
        return None
    if c["J"] == "gauss":
        return rng.standard_normal(n, dtype=np.float32)
    return (rng.integers(0, 3, size=n, dtype=np.int8) - 1).astype(np.int8)


def _lattice(c, rng):
    n, L, d = c["L"] ** c["d"], c["L"], c["d"]
    nb, w = _lattice_bonds(c, rng)
    h = _field(c, rng, n)
    idx = np.arange(n, dtype=np.int64)
    cols, vals = np.empty((n, 2 * d), np.int64), np.empty((n, 2 * d), w[0].dtype)
    for a in range(d):
        cols[:, 2 * a], vals[:, 2 * a] = nb[a], w[a]
        cols[nb[a], 2 * a + 1], vals[nb[a], 2 * a + 1] = idx, w[a]
    order = np.argsort(cols, axis=1, kind="stable")
    col = np.take_along_axis(cols, order, 1).reshape(-1).astype(np.int32)
    J = np.take_along_axis(vals, order, 1).reshape(-1)
    colour = None
    if L % 2 == 0:  # checkerboard
        colour = np.zeros(n, np.int32)
        for a in range(d):
            colour += (idx // L**a % L).astype(np.int32)
        colour &= 1
    return _instance(n, np.arange(n + 1, dtype=np.int64) * (2 * d), col, J, h, colour=colour)


def _chimera(side, rng):
    """side x side grid of K4,4 cells, 8 side^2 spins, N(0,1) couplings, N(0,0.1)
    fields, one 3-spin term N(0,0.5) per cell on a random triple of its spins."""
    n = 8 * side * side
    cell = np.arange(side * side, dtype=np.int64).reshape(side, side)
    k = np.arange(4)
    a, b = np.meshgrid(k, k, indexing="ij")
    u = [(cell.reshape(-1, 1) * 8 + a.reshape(1, -1)).ravel(),
         (cell[:-1].reshape(-1, 1) * 8 + k).ravel(), (cell[:, :-1].reshape(-1, 1) * 8 + 4 + k).ravel()]
    v = [(cell.reshape(-1, 1) * 8 + 4 + b.reshape(1, -1)).ravel(),
         (cell[1:].reshape(-1, 1) * 8 + k).ravel(), (cell[:, 1:].reshape(-1, 1) * 8 + 4 + k).ravel()]
    u, v = np.concatenate(u), np.concatenate(v)
    row_ptr, col, J = _csr(n, u, v, rng.standard_normal(len(u), dtype=np.float32))
    h = rng.standard_normal(n, dtype=np.float32) * np.float32(0.1)
    triple = np.sort(np.argsort(rng.random((side * side, 8)), axis=1)[:, :3], axis=1)
    members = (cell.reshape(-1, 1) * 8 + triple).reshape(-1).astype(np.int32)
    hJ = rng.standard_normal(side * side, dtype=np.float32) * np.float32(0.5)
    return _instance(n, row_ptr, col, J, h, (np.arange(0, 3 * side * side + 1, 3, dtype=np.int64), members, hJ))


def _random(c, rng):
    """Sparse random graph with fields and `hyper` terms of 3 or 4 spins."""
    n, m = c["n"], c["n"] * c["degree"] // 2
    u, v = rng.integers(0, n, size=2 * m), rng.integers(0, n, size=2 * m)
    keep = u != v
    key = np.unique(np.minimum(u, v)[keep] * np.int64(n) + np.maximum(u, v)[keep])
    key = np.sort(rng.permutation(key)[:m])
    row_ptr, col, J = _csr(n, key // n, key % n, _draw_J(rng, c["J"], len(key)))
    h = rng.standard_normal(n, dtype=np.float32) if c["J"] == "gauss" else rng.integers(-3, 4, size=n, dtype=np.int8)
    hyper = None
    if c["hyper"]:
        base = rng.integers(0, n, size=c["hyper"])
        size = rng.integers(3, 5, size=c["hyper"])
        step = np.cumsum(rng.integers(1, max(2, n // 8), size=(c["hyper"], 3)), axis=1)  # distinct modulo n
        mem = np.concatenate([base[:, None], (base[:, None] + step) % n], axis=1)
        ptr = np.zeros(c["hyper"] + 1, np.int64)
        np.cumsum(size, out=ptr[1:])
        hyper = (ptr, mem[np.arange(4)[None, :] < size[:, None]].astype(np.int32), _draw_J(rng, c["J"], c["hyper"]))
    return _instance(n, row_ptr, col, J, h, hyper)


def _instances(c, seed):
    rng = np.random.default_rng([seed, 0x15])
    if c["graph"] == "lattice":
        return [_lattice(c, rng)]
    if c["graph"] == "chimera":
        # the sizes are the case's (uniform in lo..hi), the values the seed's
        sides = np.random.default_rng([c["count"], c["lo"], c["hi"]]).integers(c["lo"], c["hi"] + 1, size=c["count"])
        return [_chimera(int(s), rng) for s in sides]
    if c["graph"] == "random":
        return [_random(c, rng)]
    n = c["n"]  # Sherrington-Kirkpatrick: J_ij ~ N(0,1) / sqrt(n)
    up = np.triu(rng.standard_normal((n, n), dtype=np.float32) / np.float32(np.sqrt(n)), 1)
    return [_instance(n, None, None, None, J_dense=up + up.T)]


def _seeds(seed, count):
    return np.random.default_rng([seed, 0x5EED]).integers(0, 1 << 63, size=count, dtype=np.uint64)


def _configurations(c, seed, total):
    """Random +/-1 configurations [instance][replica][spin]."""
    g = torch.Generator(device="cuda").manual_seed(int(seed) + 77)
    return torch.randint(0, 2, (c["R"] * total,), generator=g, device="cuda", dtype=torch.int8) * 2 - 1


def prepare(case, seed):
    insts = _instances(case, seed)
    h = isg.Handle(insts)
    state = SimpleNamespace(case=case, handle=h, seeds=_seeds(seed, len(insts)))
    if case["op"] == "energy":
        state.spins = _configurations(case, seed, h.total_spins)
    return state


def run(state):
    c, h = state.case, state.handle
    if c["op"] == "energy":
        return {"energy": h.energy(state.spins, c["R"])}
    if c["op"] == "passes":
        spins, energy, passes, _ = h.fm_search(state.seeds, c["R"], restarts=c["restarts"], stats=False)
        return {"spins": spins, "energy": energy, "passes": passes}
    schedule = isg.SCHED_SEQUENTIAL if c["graph"] == "sk" else isg.SCHED_COLOUR
    r = h.local_search(state.seeds, c["R"], max_sweeps=c["max_sweeps"], restarts=c["restarts"],
                       sweep_budget=c["budget"], schedule=schedule, stats=False)
    return {"spins": r.spins, "energy": r.energy, "minima": r.minima}


def work(case):
    """Bytes: the instance's couplings (value and column), fields and hyper-edges
    read once, the outputs (or the given spins) once.  Operations: for an energy
    a multiply and an add per term; for a descent the sweeps it makes (a budget's,
    else about 10 per descent), one gain (2) per visit; for passes about six
    passes of n moves, each updating a row's gains."""
    c = case
    if c["graph"] == "lattice":
        n, jb = c["L"] ** c["d"], 1 if c["J"] == "pm1" else 4
        deg, hyper, field = 2 * c["d"], 0, c["field"]
    elif c["graph"] == "chimera":
        sides = range(c["lo"], c["hi"] + 1)
        n, jb = int(c["count"] * 8 * sum(s * s for s in sides) / len(sides)), 4
        deg, hyper, field = 5.75, n // 8, True
    elif c["graph"] == "random":
        n, jb = c["n"], 4 if c["J"] == "gauss" else 1
        deg, hyper, field = c["degree"], c["hyper"], True
    else:
        n, jb, deg, hyper, field = c["n"], 4, c["n"], 0, False
    R = c["R"]
    inst = n * deg * (jb + (0 if c["graph"] == "sk" else 4)) + n * jb * field + hyper * (jb + 14)
    out = n * R
    terms = n * deg / 2 + n * field + hyper
    if c["op"] == "energy":
        return {"bytes": inst + out + 8 * R, "flops": 2.0 * terms * R}
    if c["op"] == "passes":
        return {"bytes": inst + out + 12 * R, "flops": 6.0 * 2 * deg * n * R * c["restarts"]}
    sweeps = c["budget"] or 10 * c["restarts"]
    return {"bytes": inst + out + 12 * R, "flops": 2.0 * sweeps * n * R + 2.0 * terms * R}


# ------------------------------------------------------- 64-bit expectations
def _philox(c0, c1, c2, c3, k0, k1):
    """Philox4x32-10 (Salmon et al. 2011) on uint64 arrays holding 32-bit words."""
    m = np.uint64(0xFFFFFFFF)
    s = np.uint64(32)
    for _ in range(10):
        p0, p1 = c0 * np.uint64(0xD2511F53), c2 * np.uint64(0xCD9E8D57)
        c0, c1, c2, c3 = (p1 >> s) ^ c1 ^ k0, p1 & m, (p0 >> s) ^ c3 ^ k1, p0 & m
        k0, k1 = (k0 + np.uint64(0x9E3779B9)) & m, (k1 + np.uint64(0xBB67AE85)) & m
    return c0, c1, c2, c3


def _starts(seed, n, R, k):
    """Random starts of descents (or pass searches) k of all replicas: int8 [R, n]."""
    u = np.uint64
    w, r = np.meshgrid(np.arange((n + 127) // 128, dtype=u), np.arange(R, dtype=u))
    x = _philox(w, r, np.full_like(w, k), np.zeros_like(w), u(int(seed) & 0xFFFFFFFF), u(int(seed) >> 32))
    bits = np.stack(x, axis=-1)[..., None] >> np.arange(32, dtype=u) & u(1)
    return (bits.reshape(R, -1)[:, :n].astype(np.int8) * 2 - 1)


def _tables(inst):
    """Neighbours and couplings [n, deg] of a regular graph, and the fields, in 64 bits on the GPU."""
    nb = torch.from_numpy(inst.col.reshape(inst.n, -1).astype(np.int64)).cuda()
    J = torch.from_numpy(inst.J.reshape(inst.n, -1).astype(np.float64)).cuda()
    h = np.zeros(inst.n) if inst.h is None else inst.h.astype(np.float64)
    return nb, J, torch.from_numpy(h).cuda()


def _lattice_energy(nb, J, h, s):
    e = torch.zeros(s.shape[0], dtype=torch.float64, device="cuda")
    for r in range(s.shape[0]):
        x = s[r].double()
        f = (J * x[nb]).sum(1)
        e[r] = -(x * (0.5 * f + h)).sum()
    return e


def _exact_descent(c, inst, seed):
    nb, J, h = _tables(inst)
    nb_T, J8, h8 = nb.t().contiguous(), J.t().contiguous().to(torch.int8), h.to(torch.int8)
    n, R = inst.n, c["R"]
    classes = [torch.from_numpy(np.flatnonzero(inst.colour == k)).cuda() for k in (0, 1)]
    best = torch.full((R,), float("inf"), dtype=torch.float64, device="cuda")
    for k in range(c["restarts"]):
        s = torch.from_numpy(_starts(seed, n, R, k)).cuda().t().contiguous()  # [n, R]
        done = torch.zeros(R, dtype=torch.bool, device="cuda")
        for _ in range(c["max_sweeps"]):
            flipped = torch.zeros(R, dtype=torch.bool, device="cuda")
            for idx in classes:
                f = h8[idx][:, None].expand(-1, R).contiguous()
                for a in range(nb_T.shape[0]):
                    f += J8[a][idx][:, None] * s[nb_T[a][idx]]
                x = s[idx]
                flip = (x * f < 0) & ~done
                flipped |= flip.any(0)
                s[idx] = torch.where(flip, -x, x)
            done |= ~flipped
            if bool(done.all()):
                break
        e = _lattice_energy(nb, J, h, s.t())
        best = torch.where(done & (e < best), e, best)
    last = torch.where(torch.isinf(best), e, best)
    return {"spins": None, "energy": last.view(1, R), "minima": None}


def _exact_passes(c, inst, seed):
    nb, J, h = _tables(inst)
    n, R, S = inst.n, c["R"], c["R"] * c["restarts"]
    s = np.stack([_starts(seed, n, R, k) for k in range(c["restarts"])], axis=1).reshape(S, n)
    s = torch.from_numpy(s.astype(np.float64)).cuda()
    rows = torch.arange(S, device="cuda")
    margin = 1e-9 if c["J"] == "gauss" else 0.0
    E = _lattice_energy(nb, J, h, s)
    active = torch.ones(S, dtype=torch.bool, device="cuda")
    while bool(active.any()):
        x = s.clone()
        f = torch.stack([(J * x[q][nb]).sum(1) + h for q in range(S)])
        gain = -2.0 * x * f
        cur, low = E.clone(), E.clone()
        order = torch.empty((n, S), dtype=torch.int64, device="cuda")
        best_len = torch.zeros(S, dtype=torch.int64, device="cuda")
        free = torch.ones((S, n), dtype=torch.bool, device="cuda")
        for step in range(n):
            g = torch.where(free, gain, -torch.inf)
            top = g.max(1).values
            i = (g == top[:, None]).to(torch.int8).argmax(1)  # ties: the lowest index
            cur = cur - top
            better = cur < low
            low = torch.where(better, cur, low)
            best_len = torch.where(better, step + 1, best_len)
            order[step] = i
            free[rows, i] = False
            old = x[rows, i]
            x[rows, i] = -old
            j = nb[i]
            d = 4.0 * J[i] * old[:, None] * x[rows[:, None], j]
            gain.scatter_add_(1, j, d)
        moved = torch.zeros((S, n), dtype=torch.bool, device="cuda")
        moved.scatter_(1, order.t(), torch.arange(n, device="cuda")[None, :] < best_len[:, None])
        new = torch.where(moved, -s, s)
        E_new = _lattice_energy(nb, J, h, new)
        better = active & (E_new < E - margin * (1.0 + E.abs()))
        s = torch.where(better[:, None], new, s)
        E = torch.where(better, E_new, E)
        active = better
    return {"spins": None, "energy": E.view(R, -1).min(1).values.view(1, R), "passes": None}


def _exact_energy(c, insts, seed):
    spins = _configurations(c, seed, sum(i.n for i in insts))
    out, at = [], 0
    for inst in insts:
        s = spins[at:at + c["R"] * inst.n].view(c["R"], inst.n).double()
        at += c["R"] * inst.n
        row = torch.from_numpy(np.repeat(np.arange(inst.n), np.diff(inst.row_ptr))).cuda()
        col, J = torch.from_numpy(inst.col.astype(np.int64)).cuda(), torch.from_numpy(inst.J.astype(np.float64)).cuda()
        e = torch.stack([-0.5 * (J * x[row] * x[col]).sum() for x in s])
        if inst.h is not None:
            e -= s @ torch.from_numpy(inst.h.astype(np.float64)).cuda()
        if inst.hyper_ptr is not None:
            size = np.diff(inst.hyper_ptr)
            at4 = inst.hyper_ptr[:-1, None] + np.minimum(np.arange(4)[None, :], size[:, None] - 1)
            mem = torch.from_numpy(inst.hyper_members.astype(np.int64)[at4]).cuda()
            pad = torch.from_numpy(np.arange(4)[None, :] >= size[:, None]).cuda()
            hJ = torch.from_numpy(inst.hyper_J.astype(np.float64)).cuda()
            for r in range(c["R"]):
                e[r] -= (torch.where(pad, 1.0, s[r][mem]).prod(1) * hJ).sum()
        out.append(e)
    return {"energy": torch.stack(out)}


def exact(case, seed):
    c = case
    if c["op"] == "energy":
        return _exact_energy(c, _instances(c, seed), seed)
    if c["graph"] != "lattice":
        return None
    inst = _instances(c, seed)[0]
    s0 = _seeds(seed, 1)[0]
    if c["op"] == "passes":
        return _exact_passes(c, inst, s0)
    if c["J"] == "pm1" and c["L"] % 2 == 0 and not c["budget"]:
        return _exact_descent(c, inst, s0)
    return None
