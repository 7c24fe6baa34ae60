"""Performance cases: the work a user of the library has it do, one public call (or one
short sequence of calls) per pass, over the sizes of the test systems, the batched set and
the benchmark.

A case names a system (an open Hubbard chain without point group, or random ab initio-like
integrals with a point group of 8 irreps), a bond dimension D (reduced multiplets), a pair
of sites and what is done there.  The MPS of a case has block sizes like those a sweep
leaves (many small sectors, a few large ones around the mean particle number and low spin)
and random isometries in mixed canonical form around the pair, drawn from the seed, as are
the integrals' values and the two-site vector.  Every state owns its context.
"""
import functools
import math
import struct

import numpy as np
import torch

from paper_1312_2415_gb300 import Batch, Context

# local states of an orbital: (electrons, doubled spin); the singly occupied one carries
# the orbital's irrep
_LN, _LT = (0, 1, 2), (0, 1, 0)
# occupation states of an orbital by local state: (index, doubled m)
_OCC = {0: ((0, 0),), 1: ((1, 1), (2, -1)), 2: ((3, 0),)}


# ---------------------------------------------------------------- the cases

def listed():
    def case(name, do, **kw):
        c = dict(name=name, do=do, system="random", L=12, N=12, two_S=0, D=500, site=5)
        c.update(kw)
        return c
    return [
        # H_eff x on the smallest system in use (a few thousand elements, blocks of a few
        # rows): what a caller's own eigensolver pays per application, launch latency
        case("matvec_hubbard8_d64", "matvec", system="hubbard", L=8, N=8, D=64, site=3),
        # the same on the D2h system of the tests, FP64
        case("matvec_random12_d500", "matvec"),
        # the same at the benchmark's orbitals (28, 12 electrons): thousands of blocks
        # of up to ~100 rows, operators of several hundred MB
        case("matvec_random28_d1500", "matvec", L=28, N=12, D=1500, site=13),
        # one micro-iteration's energy x^T H x / x^T x, always FP64, at half filling
        case("energy_random16_d600", "energy", L=16, N=16, D=600, site=7),
        # Davidson to convergence on a small problem: vector kernels and launches
        case("davidson_hubbard8_d64", "davidson", system="hubbard", L=8, N=8, D=64, site=3, iters=100),
        # mixed-precision Davidson with its FP64 finish, open shell, iteration cap of a sweep
        case("davidson_mixed12_d350", "davidson_mixed", two_S=2, D=350, site=4, iters=12),
        # decomposition of a two-site vector, both directions: a small and a large one
        case("truncate_left_hubbard16_d200", "truncate", system="hubbard", L=16, N=16, D=200, site=8, dir=-1),
        case("truncate_right_random28_d1500", "truncate", L=28, N=12, D=1500, site=13, dir=1),
        # the turn of a sweep: a mixed-precision step to the right and one to the left at
        # the same pair (Davidson, FP64 energy, decomposition, operator update)
        case("turn_random28_d700", "turn", L=28, N=12, D=700, site=13, iters=12),
        # 1- and 2-RDMs (the gradient of the energy) in one pass over the chain
        case("rdm_random10_d120", "rdm", L=10, N=10, D=120, site=4),
        # matvecs of several independent problems in one launch sequence
        case("batch6_hubbard_d48", "batch", system="hubbard", L=8, N=8, D=48, site=3, count=6),
        # a whole solve of the smallest system, two macro-iterations from a given MPS
        case("solve_hubbard8_d32", "solve", system="hubbard", L=8, N=8, D=32, site=0, iters=40),
    ]


def draw(rng):
    def between(lo, hi):
        return int(round(math.exp(rng.uniform(math.log(lo), math.log(hi)))))
    do = rng.choice(["matvec", "matvec", "energy", "davidson", "davidson_mixed", "truncate", "turn", "rdm", "batch",
                     "solve"])
    system = rng.choice(["hubbard", "random"])
    L = {"rdm": rng.randint(6, 10), "batch": rng.randint(6, 12), "solve": rng.randint(6, 8)}.get(do)
    L = L or rng.choice([8, 9, 10, 11, 12, 13, 14, 16])
    N = L if rng.random() < 0.5 else max(4, L - rng.randint(1, 3))
    two_S = (N & 1) + (2 if rng.random() < 0.3 else 0)
    top = {"rdm": 120, "solve": 40, "truncate": 900, "batch": 100, "turn": 350, "matvec": 800}.get(do, 400)
    c = dict(do=do, system=system, L=L, N=N, two_S=two_S, D=between(24, top), site=L // 2 - 1 + rng.randint(-1, 1))
    if do in ("davidson", "davidson_mixed", "turn", "solve"):
        c["iters"] = rng.randint(8, 16)
    if do == "truncate":
        c["dir"] = rng.choice([-1, 1])
    if do == "batch":
        c["count"] = rng.randint(2, 8)
    if do == "solve":
        c["site"] = 0
    return c


# ---------------------------------------------------------------- the problem of a case

def _irreps(case):
    """Orbital irreps: none for the Hubbard chain; the benchmark's D2h counts at 28
    orbitals, otherwise round robin."""
    L = case["L"]
    if case["system"] == "hubbard":
        return [0] * L
    if L == 28:
        return [i for i, c in enumerate((8, 3, 3, 2, 6, 2, 2, 2)) for _ in range(c)]
    return [i % 8 for i in range(L)]


def _integrals(case, seed):
    L, irr = case["L"], np.array(_irreps(case))
    rng = np.random.default_rng([seed, 1])
    if case["system"] == "hubbard":
        h = np.zeros((L, L))
        i = np.arange(L - 1)
        h[i, i + 1] = h[i + 1, i] = -1.0 - 0.1 * rng.random(L - 1)
        V = np.zeros((L, L, L, L))
        V[np.arange(L), np.arange(L), np.arange(L), np.arange(L)] = 4.0 + 0.2 * rng.random(L)
        return h, V
    off = np.triu(rng.normal(0.0, 0.5, (L, L)), 1)
    h = np.where(irr[:, None] == irr[None, :], off + off.T, 0.0)
    np.fill_diagonal(h, np.linspace(-2.0, 0.0, L))
    pair = irr[:, None] ^ irr[None, :]
    rank = 3 * L
    g = rng.normal(0.0, 0.3, (rank, L, L))
    g = np.triu(g) + np.triu(g, 1).transpose(0, 2, 1)
    g *= pair[None] == (np.arange(rank) % 8)[:, None, None]
    V = (g.reshape(rank, -1).T @ g.reshape(rank, -1)).reshape(L, L, L, L).transpose(0, 2, 1, 3)
    V = 0.5 * (V + V.transpose(1, 0, 3, 2))  # the eightfold symmetry holds to the last bit
    V = 0.5 * (V + V.transpose(2, 1, 0, 3))
    V = 0.5 * (V + V.transpose(0, 3, 2, 1))
    return h, np.ascontiguousarray(0.5 * (V + V.transpose(1, 0, 3, 2)))


def _steps(sec, irrep):
    """(local state, sector) reached from a sector (2j, N, irrep) through an orbital."""
    for ls in range(3):
        for tj in ((sec[0],) if ls != 1 else (sec[0] - 1, sec[0] + 1)):
            if tj >= 0:
                yield ls, (tj, sec[1] + _LN[ls], sec[2] ^ (irrep if ls == 1 else 0))


def _bonds(L, N, two_S, irr, D, site):
    """Sector dimensions of every bond: D multiplets spread like the spectrum of a swept
    state, no sector larger than its number of multiplets or than what isometries towards
    the pair (site, site + 1) allow."""
    left = [{(0, 0, 0): 1}]
    for k in range(L):
        new = {}
        for s, d in left[k].items():
            for _, t in _steps(s, irr[k]):
                if t[1] <= N:
                    new[t] = new.get(t, 0) + d
        left.append(new)
    right = [None] * L + [{(two_S, N, 0): 1}]
    for k in range(L - 1, -1, -1):
        right[k] = {}
        for s in left[k]:
            d = sum(right[k + 1].get(t, 0) for _, t in _steps(s, irr[k]))
            if d:
                right[k][s] = d
    cap = [{s: min(left[k][s], right[k][s]) for s in right[k]} for k in range(L + 1)]
    want = []
    for k in range(L + 1):
        mean, sigma = N * k / L, 1.3
        w = {s: math.exp(-0.5 * ((s[1] - mean) / sigma) ** 2 - 0.45 * s[0]) for s in cap[k]}
        dims, rest, open_ = {s: 0 for s in w}, D, dict(w)
        while open_ and rest > 0:  # proportional shares, the overflow of full sectors shared again
            tot, given = sum(open_.values()), 0
            for s in sorted(open_):
                a = min(cap[k][s] - dims[s], max(1, int(rest * open_[s] / tot)))
                dims[s] += a
                given += a
            rest -= given
            open_ = {s: v for s, v in open_.items() if dims[s] < cap[k][s]}
            if given == 0:
                break
        want.append({s: d for s, d in dims.items() if d > 0})
    out = [None] * (L + 1)
    out[0], out[L] = {(0, 0, 0): 1}, {(two_S, N, 0): 1}
    for k in range(site + 1):  # isometries from the left up to the middle bond
        room = {}
        for s, d in out[k].items():
            for _, t in _steps(s, irr[k]):
                room[t] = room.get(t, 0) + d
        out[k + 1] = {s: min(d, room[s]) for s, d in want[k + 1].items() if s in room}
    for k in range(L - 1, site + 1, -1):  # and from the right down to the pair's right bond
        out[k] = {}
        for s, d in want[k].items():
            room = sum(out[k + 1].get(t, 0) for _, t in _steps(s, irr[k]))
            if room:
                out[k][s] = min(d, room)
    return [sorted(b.items(), key=lambda q: (q[0][1], q[0][0], q[0][2])) for b in out]


@functools.lru_cache(maxsize=8)
def _bonds_of(key):
    L, N, two_S, irr, D, site = key
    return _bonds(L, N, two_S, list(irr), D, site)


def _shape(case):
    return _bonds_of((case["L"], case["N"], case["two_S"], tuple(_irreps(case)), case["D"], case["site"]))


def _mps(case, seed):
    """Bonds and reduced tensors {(local state, left, right): block} of every site:
    left-normalised up to site `site`, right-normalised right of site + 1, and a pair of
    unit norm.  A case that replaces the pair at once (truncate) or that normalises the
    whole chain first (solve, rdm) needs no isometries."""
    L, irr, site = case["L"], _irreps(case), case["site"]
    bonds = _shape(case)
    rng = np.random.default_rng([seed, 2])
    plain = case["do"] in ("truncate", "solve", "rdm")
    sites = []
    for k in range(L):
        idx = {s: i for i, (s, _) in enumerate(bonds[k + 1])}
        blk = [(ls, l, idx[t]) for l, (s, _) in enumerate(bonds[k]) for ls, t in _steps(s, irr[k]) if t in idx]
        T = {}
        groups = {}
        for b in blk:  # the blocks that are normalised together
            groups.setdefault(b[2] if k <= site else b[1], []).append(b)
        for q, bs in groups.items():
            dl = [bonds[k][b[1]][1] for b in bs]
            dr = [bonds[k + 1][b[2]][1] for b in bs]
            if k <= site:
                m = rng.standard_normal((sum(dl), dr[0]))
                if not plain:
                    m = np.linalg.qr(m)[0]
                parts = np.split(m, np.cumsum(dl)[:-1], axis=0)
            else:
                m = rng.standard_normal((sum(dr), dl[0]))
                if not plain and k > site + 1:
                    m = np.linalg.qr(m)[0]
                parts = [p.T for p in np.split(m, np.cumsum(dr)[:-1], axis=0)]
            for b, p in zip(bs, parts):
                if k > site:  # Eq. 6: the weighted tensor has orthonormal rows
                    p = p * math.sqrt((bonds[k][b[1]][0][0] + 1) / (bonds[k + 1][b[2]][0][0] + 1))
                T[b] = p
        if k == site + 1 and not plain:  # the norm of the state sits in this site
            n2 = sum((bonds[k + 1][b[2]][0][0] + 1) * float((p * p).sum()) for b, p in T.items())
            T = {b: p / math.sqrt(n2) for b, p in T.items()}
        sites.append(T)
    return bonds, sites


def _serialise(case, bonds, sites):
    out = [struct.pack("<6i", 0x444D5247, 1, case["L"], case["N"], case["two_S"], 0)]
    for b in bonds:
        out.append(struct.pack("<i", len(b)))
        out += [struct.pack("<4i", s[0], s[1], s[2], d) for s, d in b]
    for T in sites:
        out.append(struct.pack("<i", len(T)))
        for (ls, l, r), p in T.items():
            out.append(struct.pack("<3i", ls, l, r) + np.ascontiguousarray(p).tobytes())
    return b"".join(out)


def _layout(case):
    """Blocks (l, ls1, ls2, 2j, r, rows, cols, offset) of the two-site vector: right
    sectors in order, then left sectors, local states and 2j; and its length."""
    bonds, irr, i = _shape(case), _irreps(case), case["site"]
    left, right = bonds[i], bonds[i + 2]
    out, off = [], 0
    by = {}
    for l, (s, _) in enumerate(left):
        for ls1 in range(3):
            for ls2 in range(3):
                key = (s[1] + _LN[ls1] + _LN[ls2], s[2] ^ (irr[i] if ls1 == 1 else 0) ^ (irr[i + 1] if ls2 == 1 else 0))
                by.setdefault(key, []).append((l, ls1, ls2))
    for r, (t, dr) in enumerate(right):
        for l, ls1, ls2 in by.get((t[1], t[2]), []):
            s, dl = left[l]
            for tj in range(abs(_LT[ls1] - _LT[ls2]), _LT[ls1] + _LT[ls2] + 1, 2):
                if abs(s[0] - tj) <= t[0] <= s[0] + tj:
                    out.append((l, ls1, ls2, tj, r, dl, dr, off))
                    off += dl * dr
    return out, off


def _vector(case, seed):
    """The two-site vector: unit norm, its blocks with singular values falling over five
    orders of magnitude where it is decomposed, as an optimised vector's do."""
    blocks, n = _layout(case)
    rng = np.random.default_rng([seed, 3])
    x = rng.standard_normal(n)
    if case["do"] == "truncate":
        bonds, i = _shape(case), case["site"]
        fall = {}
        for side, b in ((0, bonds[i]), (1, bonds[i + 2])):
            for q, (_, d) in enumerate(b):
                fall[side, q] = np.exp(-6.0 * rng.permutation(d) / max(d, 1))
        for l, _, _, _, r, dl, dr, off in blocks:
            x[off:off + dl * dr] *= (fall[0, l][:, None] * fall[1, r][None, :]).ravel()
    return x / np.linalg.norm(x)


# ---------------------------------------------------------------- prepare / run / work

def _context(case, seed):
    c = Context(case["L"], _irreps(case), case["N"], case["two_S"], 0, group=0 if case["system"] == "hubbard" else 7)
    c.set_integrals(*_integrals(case, seed))
    c.set_mps(_serialise(case, *_mps(case, seed)))
    D = case["D"]
    iters = case.get("iters", 100)
    if case["do"] == "solve":
        c.set_schedule([D], [0.0], [2], [0.0], davidson_tol=1e-10, davidson_max_iter=iters)
    else:
        c.set_schedule([D], [1e-8], [2], [0.0], davidson_tol=1e-10, davidson_max_iter=iters)
    return c


def prepare(case, seed):
    do, site = case["do"], case["site"]
    st = {"do": do, "site": site, "D": case["D"], "dir": case.get("dir", 1)}
    if do == "batch":
        # independent problems of neighbouring sizes, as in a scan over geometries
        subs = [dict(case, D=case["D"] + 8 * q) for q in range(case["count"])]
        st["ctxs"] = [_context(s, seed + 7919 * q) for q, s in enumerate(subs)]
        st["xs"] = [torch.tensor(_vector(s, seed + 7919 * q), device="cuda") for q, s in enumerate(subs)]
        st["ys"] = [torch.empty_like(x) for x in st["xs"]]
        st["batch"] = Batch(st["ctxs"], [site] * len(subs), autotune=False)
        return st
    c = st["ctx"] = _context(case, seed)
    if do == "davidson_mixed":
        c.set_precision(1)
    if do == "turn":
        c.set_precision(1, 1)
    if do == "solve":
        st["mps"] = c.get_mps()
    elif do == "rdm":
        c.canonicalize(0)
    elif do != "turn":
        st["x"] = torch.tensor(_vector(case, seed), device="cuda")
        st["y"] = torch.empty_like(st["x"])
    if do in ("matvec", "energy", "davidson", "davidson_mixed"):
        c.matvec(site, st["x"], st["y"])  # the tables of this pair, made once
    if do == "energy":
        c.energy(site, st["x"])
    return st


def run(state):
    do, site, c = state["do"], state["site"], state.get("ctx")
    if do == "matvec":
        return c.matvec(site, state["x"], state["y"])
    if do == "energy":
        return c.energy(site, state["x"])
    if do in ("davidson", "davidson_mixed"):
        v = state["y"].copy_(state["x"])
        e, _, _ = c.davidson(site, v)
        return e, v
    if do == "truncate":
        w = c.truncate(site, state["dir"], state["D"], state["x"])
        return w, c.tt_to_x(site, state["y"])
    if do == "turn":
        out = []
        for d in (1, -1):
            c.set_next_site(site)
            e, w, _, _ = c.sweep_step(site, d, state["D"])
            out += [e, w]
        return out, c.tt_to_x(site)
    if do == "rdm":
        return c.rdm()
    if do == "batch":
        state["batch"].run(state["xs"], state["ys"])
        return state["ys"]
    c.set_mps(state["mps"])
    e_min, e_last = c.solve()
    D, E, w = c.solve_history()
    return e_min, e_last, D, E


def _ops(L, k, irr):
    """(dN, irrep, 2K) of the renormalised operators a block of k orbitals holds: the
    identity and the Hamiltonian, single operators inside and complementary ones outside,
    and pairs a+a+, aa, a+a coupled to spin 0 and 1 inside."""
    ops = [(0, 0, 0)] * 2
    for p in range(L):
        ops += [(1, irr[p], 1), (-1, irr[p], 1)]
    for p in range(k):
        for q in range(p, k):
            g = irr[p] ^ irr[q]
            for K in (0, 2):
                if p < q or K == 0:
                    ops += [(2, g, K), (-2, g, K)]
                ops.append((0, g, K))
                if p < q:
                    ops.append((0, g, K))
    return ops


def _count_blocks(bond, ops):
    """Elements of the operators' blocks at a bond, and 2 m k n summed over the products
    of each block with the right factor of `width` columns per row of its source."""
    dim = dict(bond)
    size, per = 0, {}
    for op in ops:
        if op not in per:
            per[op] = [(d * dim[t], s) for s, d in bond
                       for t in ((tj, s[1] + op[0], s[2] ^ op[1]) for tj in range(abs(s[0] - op[2]), s[0] + op[2] + 1, 2))
                       if t in dim]
        size += sum(a for a, _ in per[op])
    return size, per


def _one(case):
    """bytes and flops of one H_eff x: the operators of both blocks read once, x read and
    y written; every operator block times the part of x it acts on."""
    bonds, irr, i, L = _shape(case), _irreps(case), case["site"], case["L"]
    blocks, n = _layout(case)
    hub = case["system"] == "hubbard"
    rows, cols = {}, {}
    for l, _, _, _, r, dl, dr, _ in blocks:
        cols[l] = cols.get(l, 0) + dr
        rows[r] = rows.get(r, 0) + dl
    nbytes, flops = 16.0 * n, 0.0
    for bond, k, width in ((bonds[i], i, cols), (bonds[i + 2], L - i - 2, rows)):
        order = irr if bond is bonds[i] else irr[::-1]
        ops = [(0, 0, 0)] * 2 + [(s, 0, 1) for s in (1, -1)] * 2 if hub else _ops(L, k, order)
        pos = {s: q for q, (s, _) in enumerate(bond)}
        size, per = _count_blocks(bond, ops)
        nbytes += 8.0 * size
        for op in ops:
            flops += sum(2.0 * a * width.get(pos[s], 0) for a, s in per[op]) / 2  # half: the pairs of one side only
    return nbytes, flops


def work(case):
    do, L = case["do"], case["L"]
    n = _layout(case)[1]
    if do == "truncate":
        # reduced matrices of the middle sectors: Gram product, eigenvectors, projection
        b = _shape(case)[case["site"] if case["dir"] > 0 else case["site"] + 2]
        f = sum(2.0 * n * 2 * d for _, d in b) / max(1, len(b)) * 3
        return {"bytes": 16.0 * n, "flops": f}
    if do in ("rdm", "solve"):
        tot_b = tot_f = 0.0
        for i in range(L - 1):
            b, f = _one(dict(case, site=i, do="matvec"))
            tot_b, tot_f = tot_b + b, tot_f + f
        k = 2 if do == "rdm" else 4 * 10  # adjoint products; two macro-iterations of some ten products per step
        return {"bytes": tot_b * (1 if do == "rdm" else 4), "flops": tot_f * k}
    if do == "batch":
        parts = [_one(dict(case, D=case["D"] + 8 * q)) for q in range(case["count"])]
        return {"bytes": sum(p[0] for p in parts), "flops": sum(p[1] for p in parts)}
    b, f = _one(case)
    if do == "energy":
        return {"bytes": b, "flops": 0.5 * f}
    if do in ("davidson", "davidson_mixed", "turn"):
        # one product per iteration; a turn also updates the operators of both blocks
        it = min(case["iters"], 25)
        return {"bytes": b * (2 if do == "turn" else 1), "flops": f * (2 * it + 4 if do == "turn" else it)}
    return {"bytes": b, "flops": f}


# ---------------------------------------------------------------- exact values
#
# H_eff = P^T H P written out in the determinants of the whole chain: the two-site vector
# is expanded with Clebsch-Gordan coefficients (spin projections explicit), H acts through
# single excitations of alpha and beta strings, and the result is projected back.

@functools.lru_cache(maxsize=None)
def _cg(j1, m1, j2, m2, j, m):
    """<j1 m1 j2 m2 | j m>, all arguments doubled (Racah's formula)."""
    if m1 + m2 != m or not abs(j1 - j2) <= j <= j1 + j2 or (j1 + j2 + j) & 1 or abs(m) > j or abs(m1) > j1 or abs(m2) > j2:
        return 0.0
    f = lambda a: math.factorial(a // 2)  # noqa: E731
    pre = (j + 1) * f(j1 + j2 - j) * f(j1 - j2 + j) * f(-j1 + j2 + j) / f(j1 + j2 + j + 2)
    pre *= f(j + m) * f(j - m) * f(j1 + m1) * f(j1 - m1) * f(j2 + m2) * f(j2 - m2)
    s = 0.0
    for k in range(0, j1 + j2 - j + 1, 2):
        d = (k, j1 + j2 - j - k, j1 - m1 - k, j2 + m2 - k, j - j2 + m1 + k, j - j1 - m2 + k)
        if min(d) >= 0:
            s += (-1) ** (k // 2) / math.prod(f(a) for a in d)
    return math.sqrt(pre) * s


@functools.lru_cache(maxsize=None)
def _sixj(a, b, c, d, e, f):
    """{a b c; d e f}, all arguments doubled (Racah's formula)."""
    tri = ((a, b, c), (a, e, f), (d, b, f), (d, e, c))
    if any(not abs(x - y) <= z <= x + y or (x + y + z) & 1 for x, y, z in tri):
        return 0.0
    g = lambda v: math.factorial(v // 2)  # noqa: E731
    pre = math.prod(g(x + y - z) * g(x - y + z) * g(-x + y + z) / g(x + y + z + 2) for x, y, z in tri)
    s = 0.0
    lo = [sum(t) for t in tri]
    hi = (a + b + d + e, b + c + e + f, c + a + f + d)
    for t in range(max(lo), min(hi) + 1, 2):
        s += (-1) ** (t // 2) * g(t + 2) / (math.prod(g(t - v) for v in lo) * math.prod(g(v - t) for v in hi))
    return math.sqrt(pre) * s


def _dev():
    return "cuda" if torch.cuda.is_available() else "cpu"


def _grow(case, bonds, sites):
    """Left and right renormalised states of the pair's outer bonds in occupation states:
    {sector index: (states, dim, 2j + 1)} and {sector index: (dim, 2j + 1, states)}."""
    irr, i, L, dev = _irreps(case), case["site"], case["L"], _dev()
    A = {0: torch.ones(1, 1, 1, dtype=torch.float64, device=dev)}
    for k in range(i):
        A = _step_left(A, bonds, sites, k)
    S = case["two_S"]
    B = {0: torch.zeros(1, S + 1, 1, dtype=torch.float64, device=dev)}
    B[0][0, S, 0] = 1.0  # the component m = S of the target multiplet
    for k in range(L - 1, i + 1, -1):
        B = _step_right(B, bonds, sites, k)
    return A, B


def _step_left(A, bonds, sites, k):
    out = {}
    for (ls, l, r), T in sites[k].items():
        if l not in A:
            continue
        jl, jr = bonds[k][l][0][0], bonds[k + 1][r][0][0]
        F = A[l].shape[0]
        Y = torch.einsum("fam,ab->fbm", A[l], torch.tensor(np.ascontiguousarray(T), device=A[l].device))
        if r not in out:
            out[r] = torch.zeros(F, 4, bonds[k + 1][r][1], jr + 1, dtype=torch.float64, device=Y.device)
        for occ, ms in _OCC[ls]:
            for im in range(jl + 1):
                m = 2 * im - jl + ms
                if abs(m) <= jr:
                    out[r][:, occ, :, (m + jr) // 2] += _cg(jl, 2 * im - jl, _LT[ls], ms, jr, m) * Y[:, :, im]
    return {r: v.reshape(-1, v.shape[2], v.shape[3]) for r, v in out.items()}


def _step_right(B, bonds, sites, k):
    out = {}
    for (ls, l, r), T in sites[k].items():
        if r not in B:
            continue
        jl, jr = bonds[k][l][0][0], bonds[k + 1][r][0][0]
        G = B[r].shape[2]
        Y = torch.einsum("ab,bmg->amg", torch.tensor(np.ascontiguousarray(T), device=B[r].device), B[r])
        if l not in out:
            out[l] = torch.zeros(bonds[k][l][1], jl + 1, 4, G, dtype=torch.float64, device=Y.device)
        for occ, ms in _OCC[ls]:
            for im in range(jl + 1):
                m = 2 * im - jl + ms
                if abs(m) <= jr:
                    out[l][:, im, occ, :] += _cg(jl, 2 * im - jl, _LT[ls], ms, jr, m) * Y[:, (m + jr) // 2, :]
    return {l: v.reshape(v.shape[0], v.shape[1], -1) for l, v in out.items()}


def _terms(case, bonds):
    """(block, m index of the left state, occupations, m index of the right state,
    coefficient) of the expansion of every block of the two-site vector."""
    i = case["site"]
    for b in _layout(case)[0]:
        l, ls1, ls2, tj, r = b[:5]
        jl, jr = bonds[i][l][0][0], bonds[i + 2][r][0][0]
        for o1, m1 in _OCC[ls1]:
            for o2, m2 in _OCC[ls2]:
                c = _cg(_LT[ls1], m1, _LT[ls2], m2, tj, m1 + m2)
                for im in range(jl + 1):
                    m = 2 * im - jl + m1 + m2
                    v = c * _cg(jl, 2 * im - jl, tj, m1 + m2, jr, m) / math.sqrt(jr + 1)
                    if v != 0.0:
                        yield b, im, o1 * 4 + o2, (m + jr) // 2, v


def _expand(case, bonds, A, B, x):
    """P x: amplitudes over the occupation states of the chain (left, pair, right)."""
    F, G = next(iter(A.values())).shape[0], next(iter(B.values())).shape[2]
    psi = torch.zeros(F, 16, G, dtype=torch.float64, device=x.device)
    per = {}
    for b, im, o, jm, v in _terms(case, bonds):
        l, r, dl, dr, off = b[0], b[4], b[5], b[6], b[7]
        if l in A and r in B:
            y = v * (A[l][:, :, im] @ x[off:off + dl * dr].view(dl, dr))
            key = (r, jm, o)
            per[key] = per[key] + y if key in per else y
    for (r, jm, o), y in per.items():
        psi[:, o, :] += y @ B[r][:, jm, :]
    return psi.reshape(-1)


def _project(case, bonds, A, B, psi, n):
    """P^T psi."""
    F, G = next(iter(A.values())).shape[0], next(iter(B.values())).shape[2]
    psi = psi.view(F, 16, G)
    y = torch.zeros(n, dtype=torch.float64, device=psi.device)
    per = {}
    for b, im, o, jm, v in _terms(case, bonds):
        l, r, dl, dr, off = b[0], b[4], b[5], b[6], b[7]
        if l in A and r in B:
            if (r, jm, o) not in per:
                per[r, jm, o] = psi[:, o, :] @ B[r][:, jm, :].T
            y[off:off + dl * dr] += v * (A[l][:, :, im].T @ per[r, jm, o]).reshape(-1)
    return y * (case["two_S"] + 1)  # the other spin projections contribute the same


class _Strings:
    """Determinants with N electrons and spin projection S, and the single excitations of
    their alpha and beta strings."""

    def __init__(self, L, N, two_S):
        self.L, na, nb = L, (N + two_S) // 2, (N - two_S) // 2
        dev = _dev()
        bits = np.arange(1 << L)
        pop = np.array([bin(b).count("1") for b in bits])
        self.str = [bits[pop == na], bits[pop == nb]]
        pos = np.full((2, 1 << L), -1)
        for s in (0, 1):
            pos[s, self.str[s]] = np.arange(len(self.str[s]))
        self.exc = [[None] * (L * L) for _ in (0, 1)]
        for s in (0, 1):
            S = self.str[s]
            for p in range(L):
                for q in range(L):
                    ok = (S >> q) & 1 == 1
                    T = S ^ (1 << q)
                    ok &= (T >> p) & 1 == 0
                    src = np.nonzero(ok)[0]
                    t = T[src]
                    sg = (pop[S[src] & ((1 << q) - 1)] + pop[t & ((1 << p) - 1)]) & 1
                    dst = pos[s, t | (1 << p)]
                    self.exc[s][p * L + q] = tuple(torch.tensor(v, device=dev) for v in (src, dst, 1.0 - 2.0 * sg))
        # occupation index (base 4, orbital 0 first: empty, up, down, both) of every
        # determinant, and the sign of moving the alpha operators left of the beta ones
        a, b = self.str[0][:, None], self.str[1][None, :]
        occ = np.zeros((len(self.str[0]), len(self.str[1])), dtype=np.int64)
        par = np.zeros_like(occ)
        for k in range(L):
            occ = occ * 4 + ((a >> k) & 1) + 2 * ((b >> k) & 1)
            par += ((b >> k) & 1) * pop[a >> (k + 1)]
        self.occ = torch.tensor(occ.ravel(), device=dev)
        self.sign = torch.tensor(1.0 - 2.0 * (par.ravel() & 1), device=dev)
        self.shape = occ.shape

    def read(self, psi):
        return (psi[self.occ] * self.sign).view(self.shape)

    def write(self, v, size):
        psi = torch.zeros(size, dtype=torch.float64, device=v.device)
        psi[self.occ] = v.reshape(-1) * self.sign
        return psi

    def excite(self, pq, v, out):
        """out += E_pq v."""
        src, dst, sg = self.exc[0][pq]
        out.index_add_(0, dst, v[src] * sg[:, None])
        src, dst, sg = self.exc[1][pq]
        out.index_add_(1, dst, v[:, src] * sg[None, :])

    def all_excitations(self, v):
        out = torch.zeros((self.L ** 2,) + self.shape, dtype=torch.float64, device=v.device)
        for pq in range(self.L ** 2):
            self.excite(pq, v, out[pq])
        return out

    def apply(self, h, V, v):
        """H v with H = sum h E + 1/2 sum V_ijkl (E_ik E_jl - delta_jk E_il)."""
        L = self.L
        dev = v.device
        E = self.all_excitations(v).view(L * L, -1)
        h1 = torch.tensor(h - 0.5 * np.einsum("ijjl->il", V), device=dev).reshape(1, -1)
        G = torch.tensor(0.5 * np.ascontiguousarray(V.transpose(0, 2, 1, 3)).reshape(L * L, L * L), device=dev)
        out = (h1 @ E).view(self.shape).clone()
        M = (G @ E).view((L * L,) + self.shape)
        for pq in range(L * L):
            self.excite(pq, M[pq], out)
        return out


@functools.lru_cache(maxsize=4)
def _strings(L, N, two_S):
    return _Strings(L, N, two_S)


def _heff(case, seed):
    """x -> P^T H P x of the case's problem."""
    bonds, sites = _mps(case, seed)
    h, V = _integrals(case, seed)
    A, B = _grow(case, bonds, sites)
    D = _strings(case["L"], case["N"], case["two_S"])
    n = _layout(case)[1]

    def apply(x):
        psi = _expand(case, bonds, A, B, x)
        return _project(case, bonds, A, B, D.write(D.apply(h, V, D.read(psi)), psi.numel()), n)
    return apply


def _exact_truncate(case, seed):
    """The D largest reduced singular values kept over all middle sectors; the discarded
    weight and the two-site vector of the truncated, rescaled state."""
    bonds, irr, i, x = _shape(case), _irreps(case), case["site"], _vector(case, seed)
    left, right = bonds[i], bonds[i + 2]
    mats = {}
    for l, ls1, ls2, tj, r, dl, dr, off in _layout(case)[0]:
        (jl, nl, il), jr = left[l][0], right[r][0][0]
        t1, t2 = _LT[ls1], _LT[ls2]
        ph = -1.0 if ((jl + jr + t1 + t2) // 2) & 1 else 1.0
        for jm in range(abs(jl - t1), jl + t1 + 1, 2):
            c = ph * _sixj(jl, jr, tj, t2, t1, jm) * math.sqrt(tj + 1)
            if c != 0.0:
                s = (jm, nl + _LN[ls1], il ^ (irr[i] if ls1 == 1 else 0))
                mats.setdefault(s, []).append(((l, ls1), (r, ls2), c, off, dl, dr))
    svd = {}
    for s, parts in mats.items():
        ro, co, R, C = {}, {}, 0, 0
        for a, b, _, _, dl, dr in sorted(parts, key=lambda q: (q[0], q[1])):
            if a not in ro:
                ro[a], R = R, R + dl
            if b not in co:
                co[b], C = C, C + dr
        M = np.zeros((R, C))
        for a, b, c, off, dl, dr in parts:
            M[ro[a]:ro[a] + dl, co[b]:co[b] + dr] += c * x[off:off + dl * dr].reshape(dl, dr)
        svd[s] = np.linalg.svd(M, full_matrices=False) + (ro, co)
    lam = sorted(((v, s) for s in svd for v in svd[s][1]), reverse=True, key=lambda q: q[0])
    kept = [q for q in lam[:case["D"]] if q[0] > 3e-8 * lam[0][0]]
    norm2 = sum((s[0] + 1) * v * v for v, s in lam)
    w = sum((s[0] + 1) * v * v for v, s in lam[len(kept):]) / norm2
    count = {}
    for _, s in kept:
        count[s] = count.get(s, 0) + 1
    out = np.zeros_like(x)
    for s, k in count.items():
        U, sv, Vt, ro, co = svd[s]
        M = (U[:, :k] * sv[:k]) @ Vt[:k]
        for a, b, c, off, dl, dr in mats[s]:
            out[off:off + dl * dr] += (s[0] + 1) * c * M[ro[a]:ro[a] + dl, co[b]:co[b] + dr].ravel()
    return float(w), torch.tensor(out / math.sqrt(norm2))


def _exact_rdm(case, seed):
    """Spin-summed RDMs of the state, the two-particle one averaged over the eight index
    permutations that leave V unchanged."""
    bonds, sites = _mps(case, seed)
    L, S = case["L"], case["two_S"]
    A = {0: torch.ones(1, 1, 1, dtype=torch.float64, device=_dev())}
    half = L // 2
    for k in range(half):
        A = _step_left(A, bonds, sites, k)
    B = {0: torch.zeros(1, S + 1, 1, dtype=torch.float64, device=_dev())}
    B[0][0, S, 0] = 1.0
    for k in range(L - 1, half - 1, -1):
        B = _step_right(B, bonds, sites, k)
    psi = sum(A[q].reshape(A[q].shape[0], -1) @ B[q].reshape(-1, B[q].shape[2]) for q in A if q in B).reshape(-1)
    D = _strings(L, case["N"], S)
    v = D.read(psi)
    v = v / v.norm()
    E = D.all_excitations(v).view(L * L, -1)
    gamma = (E @ v.reshape(-1)).view(L, L)
    two = (E @ E.T).view(L, L, L, L)  # <(E_pq v), (E_rs v)> = <E_qp E_rs>
    two = two.permute(1, 2, 0, 3).clone()  # [i = q, j = r, k = p, l = s]: <E_ik E_jl>
    for j in range(L):
        two[:, j, j, :] -= gamma
    g8 = two
    for p in ((1, 0, 3, 2), (2, 1, 0, 3), (0, 3, 2, 1)):
        g8 = 0.5 * (g8 + g8.permute(p))
    return 0.5 * (gamma + gamma.T), g8


def exact(case, seed):
    do = case["do"]
    if do == "truncate":
        return _exact_truncate(case, seed)
    if case["L"] > 12:
        return None
    if do == "rdm":
        return _exact_rdm(case, seed)
    if do == "matvec":
        return _heff(case, seed)(torch.tensor(_vector(case, seed), device=_dev()))
    if do == "energy":
        x = torch.tensor(_vector(case, seed), device=_dev())
        return float(x @ _heff(case, seed)(x))
    if do == "batch":
        return [exact(dict(case, do="matvec", D=case["D"] + 8 * q), seed + 7919 * q) for q in range(case["count"])]
    if do == "davidson" and _layout(case)[1] <= 2000 and case["iters"] >= 100:
        f = _heff(case, seed)
        eye = torch.eye(_layout(case)[1], dtype=torch.float64, device=_dev())
        H = torch.stack([f(e) for e in eye])
        w, U = torch.linalg.eigh(0.5 * (H + H.T))
        u = U[:, 0]
        s = float(u @ torch.tensor(_vector(case, seed), device=u.device))
        return float(w[0]), u if s >= 0 else -u
    return None
