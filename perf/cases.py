"""Performance cases: the calls that a user of the library makes, over the range of sizes.

A case names a problem (integral type, orbitals, electrons, layout), a precision and a call
(one sigma build, a Davidson solve, a compressed sigma, a batch of sigma builds).  listed()
gives fixed cases, draw(rng) one more of the same ranges, prepare(case, seed) what a program
holds before the call, run(state) the call, work(case) the bytes and operations that the
result cannot do without, and exact(case, seed) the result in 64 bits by plain torch.
"""
from __future__ import annotations

import itertools
import math

import numpy as np
import torch

from paper_2505_20375_gb300 import fci

E_CORE = 0.75


# ---------------------------------------------------------------------------- cases

def _fci(n, na, nb, precision, slices=0, **more):
    return dict(kind="fci", n=n, na=na, nb=nb, precision=precision, slices=slices, **more)


def _das(spaces, ref, transfer, precision, slices=0, **more):
    return dict(kind="das", spaces=",".join(map(str, spaces)), ref=",".join(map(str, ref)), transfer=transfer,
                precision=precision, slices=slices, **more)


def _spinor(n, ne, precision, slices=0, **more):
    return dict(kind="spinor", n=n, ne=ne, precision=precision, slices=slices, **more)


def listed():
    return [
        # the smallest space worth a solve: launches and latency count
        _fci(8, 4, 4, "oz_bf16", 6, name="fci_8e8o_s6"),
        # an FP64 sigma of a medium FCI space, the reference precision of every solve
        _fci(12, 6, 6, "fp64", name="fci_12e12o_fp64"),
        # an open-shell space (odd orbital count, unequal spins) at the highest slice count
        _fci(13, 7, 6, "oz_bf16", 7, name="fci_13e13o_s7"),
        # the benchmark's headline: FP64-class split sigma of FCI(14e,14o)
        _fci(14, 7, 7, "oz_bf16", 6, name="fci_14e14o_s6"),
        # the long FP64 request of the serving mix
        _das((4, 4, 4, 4), (1, 1, 1, 1), 1, "fp64", name="das_16o_8e_t1_fp64"),
        # the FP64-class phase of a mixed-precision solve on the DAS layout
        _das((4, 4, 4, 4), (2, 2, 1, 1), 1, "oz_bf16", 6, name="das_16o_12e_t1_s6"),
        # the first phase of a mixed-precision solve on the largest DAS space
        _das((4, 4, 4, 4), (2, 2, 2, 2), 2, "oz_bf16", 3, name="das_16o_16e_t2_s3"),
        # two-spinor (complex) CI: plain complex FP64, and the largest space at FP64 class
        _spinor(20, 10, "fp64", name="spinor_20s10e_fp64"),
        _spinor(24, 12, "oz_bf16", 8, name="spinor_24s12e_s8"),
        # a whole mixed-precision Davidson solve
        dict(kind="davidson", n=10, na=5, nb=5, first=3, final=6, name="davidson_10e10o_mixed"),
        # categorically compressed sigma on the literal 4 x 6 space (1.9e12 determinants)
        dict(kind="compressed", nnz=400, name="compressed_24o_400"),
        # the grouped sigma build of a serving step: several small solves of one slice count
        dict(kind="grouped", jobs=10, low=6, high=12, slices=3, name="grouped_serving_s3"),
    ]


def draw(rng):
    kind = rng.choice(["fci", "fci", "fci", "das", "das", "spinor", "spinor", "davidson", "compressed", "grouped"])
    if kind == "fci":
        n = rng.randint(6, 14)
        na, nb = (max(1, min(n - 1, n // 2 + rng.randint(-2, 1))) for _ in range(2))
        s = rng.choice([0, 0, 2, 3, 4, 5, 6, 6, 7])
        return _fci(n, na, nb, "oz_bf16" if s else "fp64", s)
    if kind == "spinor":
        s = rng.choice([0, 3, 3, 6, 8])
        n = rng.randint(10, 24 if s else 20)
        return _spinor(n, rng.randint(max(2, n // 4), n // 2 + 1), "oz_bf16" if s else "fp64", s)
    if kind == "das":
        while True:
            spaces = [rng.randint(2, 5) for _ in range(rng.randint(3, 4))]
            ref = [rng.randint(1, (m + 1) // 2) for m in spaces]
            t, s = rng.randint(0, 2), rng.choice([0, 0, 2, 3, 3, 6, 6])
            if not 8 <= sum(spaces) <= 16:
                continue
            size = _intermediate_size(spaces, ref, t)
            if 2000 <= size <= (6_000_000 if s == 0 else 60_000_000 if s <= 3 else 22_000_000):
                return _das(spaces, ref, t, "oz_bf16" if s else "fp64", s)
    if kind == "davidson":
        n = rng.randint(6, 10)
        k = n // 2
        return dict(kind="davidson", n=n, na=k, nb=k - rng.randint(0, 1), first=rng.choice([0, 3, 4]), final=6)
    if kind == "compressed":
        return dict(kind="compressed", nnz=int(round(20 * 20 ** rng.random())))
    low = rng.randint(6, 8)
    return dict(kind="grouped", jobs=rng.randint(3, 16), low=low, high=low + rng.randint(1, 3),
                slices=rng.choice([3, 3, 4, 6]))


# --------------------------------------------------------------------------- inputs

LITERAL = dict(spaces=[6, 6, 6, 6], ref=[3, 3, 3, 3], transfer=2)


def _ints(text):
    return [int(v) for v in text.split(",")]


def _integrals(n, complex_, seed):
    """One- and two-electron integrals: orbital energies spread over [-2, 1], small couplings,
    (pq|rs) from 2 n Cholesky-like vectors (positive semidefinite, full permutation symmetry)."""
    r = np.random.default_rng([seed, n, int(complex_)])

    def matrices(count, scale):
        x = r.normal(size=(count, n, n)) * scale
        if complex_:
            x = (x + 1j * r.normal(size=(count, n, n)) * scale) / math.sqrt(2)
        x = np.triu(x, 1)
        return x + x.conj().transpose(0, 2, 1) + np.eye(n) * (r.normal(size=(count, 1, n)) * scale)

    h = matrices(1, 0.05)[0]
    h[np.diag_indices(n)] = np.sort(r.uniform(-2, 1, n))
    L = matrices(2 * n, 0.1).reshape(2 * n, n * n)
    return h, (L.T @ L).reshape(n, n, n, n)


def _vector(count, complex_, seed):
    g = torch.Generator(device="cuda").manual_seed(seed)
    v = torch.randn(count, dtype=torch.complex128 if complex_ else torch.float64, device="cuda", generator=g)
    return v / torch.linalg.vector_norm(v)


def _coefficients(case, seed):
    """Ascending addresses over the literal space and their normalised values.  The addresses
    follow from the case, as the support of a vector outlives its values in a solve."""
    r = np.random.default_rng([case["nnz"], 24])
    total = _target_size(**LITERAL)
    addr = np.unique((r.random(2 * case["nnz"]) * total).astype(np.int64))
    addr = np.sort(r.choice(addr, case["nnz"], replace=False))
    val = np.random.default_rng([seed, 24]).normal(size=case["nnz"])
    return torch.from_numpy(addr).cuda(), torch.from_numpy(val / np.linalg.norm(val)).cuda()


def _handle(h, g, na, nb, das=None):
    f = fci.FCI(0).setup_integrals(h, g, E_CORE).build_strings(na, nb)
    return f.build_das(das[0], das[1], das[1], das[2]) if das else f


def _das_of(case):
    if case["kind"] == "compressed":
        return LITERAL["spaces"], LITERAL["ref"], LITERAL["transfer"]
    return _ints(case["spaces"]), _ints(case["ref"]), case["transfer"]


def _group(case):
    """(orbitals, alpha, beta) of the batch's problems, sizes in turn from low to high."""
    span = case["high"] - case["low"] + 1
    sizes = [case["low"] + j % span for j in range(case["jobs"])]
    return [(n, n // 2, n // 2) for n in sizes]


def prepare(case, seed):
    kind = case["kind"]
    if kind == "grouped":
        jobs = []
        for j, (n, na, nb) in enumerate(_group(case)):
            f = _handle(*_integrals(n, False, seed + 1000 * j), na, nb)
            C = _vector(f.n_det, False, seed + 1000 * j)
            size = f.sigma_workspace_bytes("oz_bf16", case["slices"])
            ws = torch.empty(size + 256, dtype=torch.uint8, device="cuda")
            jobs.append((f, C, torch.empty_like(C), "oz_bf16", case["slices"], (ws.data_ptr() + 255) & ~255, size, ws))
        return dict(case=case, jobs=jobs)
    if kind == "spinor":
        f = _handle(*_integrals(case["n"], True, seed), case["ne"], -1)
        return dict(case=case, f=f, C=_vector(f.n_det, True, seed))
    if kind in ("das", "compressed"):
        das = _das_of(case)
        f = _handle(*_integrals(sum(das[0]), False, seed), sum(das[1]), sum(das[1]), das)
        if kind == "compressed":
            addr, val = _coefficients(case, seed)
            return dict(case=case, f=f, addr=addr, val=val)
        return dict(case=case, f=f, C=_vector(f.n_det, False, seed))
    f = _handle(*_integrals(case["n"], False, seed), case["na"], case["nb"])
    return dict(case=case, f=f, C=_vector(f.n_det, False, seed) if kind == "fci" else None)


def run(state):
    case = state["case"]
    kind = case["kind"]
    if kind == "grouped":
        fci.sigma_grouped([j[:7] for j in state["jobs"]])
        return [j[2] for j in state["jobs"]]
    if kind == "compressed":
        addr, val = state["f"].sigma_compressed(state["addr"], state["val"])
        return dict(addr=addr, val=val)
    if kind == "davidson":
        first = dict(precision="oz_bf16", n_slices=case["first"], switch_residual=1e-3) if case["first"] else {}
        final = dict(final_precision="oz_bf16", final_slices=case["final"]) if case["first"] else {}
        r = state["f"].davidson(max_iter=200, tol_residual=1e-6, tol_energy=1e-10, **first, **final)
        return dict(energy=r.energy, vector=r.vector)
    return state["f"].sigma(state["C"], precision=case["precision"], n_slices=case["slices"])


# ----------------------------------------------------------------------------- work

def _patterns(spaces, ref, limit):
    """Electron counts per space of one spin with excess over the reference <= limit."""
    ne = sum(ref)
    for p in itertools.product(*[range(m + 1) for m in spaces]):
        e = sum(max(0, a - b) for a, b in zip(p, ref))
        if sum(p) == ne and e <= limit:
            yield p, e, math.prod(math.comb(m, k) for m, k in zip(spaces, p))


def _size(spaces, ref, limit):
    by = {}
    for _, e, count in _patterns(spaces, ref, limit):
        by[e] = by.get(e, 0) + count
    return sum(a * b for e, a in by.items() for f, b in by.items() if e + f <= limit)


def _target_size(spaces, ref, transfer):
    return _size(spaces, ref, transfer)


def _intermediate_size(spaces, ref, transfer):
    return _size(spaces, ref, transfer + 1)


def _connections(pattern, spaces, ref, moves):
    """{excess after: count} of the same-spin replacements of `moves` electrons of one string."""
    out = {}
    S = range(len(spaces))
    for taken in itertools.combinations_with_replacement(S, moves):
        for put in itertools.combinations_with_replacement(S, moves):
            ways, q = 1, list(pattern)
            for s in S:
                ways *= math.comb(pattern[s], taken.count(s)) * math.comb(spaces[s] - pattern[s], put.count(s))
                q[s] += put.count(s) - taken.count(s)
            if ways:
                e = sum(max(0, a - b) for a, b in zip(q, ref))
                out[e] = out.get(e, 0) + ways
    return out


def _elements(spaces, ref_a, ref_b, transfer):
    """Nonzero matrix elements of H over the whole space: the multiply-adds of one sigma."""
    def spin(ref):
        by = {}  # (excess, per-move connection counts) summed over strings
        for p, e, count in _patterns(spaces, ref, transfer):
            c = [{e: 1}, _connections(p, spaces, ref, 1), _connections(p, spaces, ref, 2)]
            key = (e, str(c))
            by[key] = (by.get(key, (0, c))[0] + count, c)
        return [(e, n, c) for (e, _), (n, c) in by.items()]

    total = 0
    beta = spin(ref_b) if ref_b is not None else [(0, 1, [{0: 1}, {}, {}])]
    for ea, na, ca in spin(ref_a):
        for eb, nb, cb in beta:
            if ea + eb > transfer:
                continue
            for i, j in ((0, 0), (1, 0), (0, 1), (2, 0), (0, 2), (1, 1)):
                total += na * nb * sum(x * y for e, x in ca[i].items() for f, y in cb[j].items() if e + f <= transfer)
    return total


def work(case):
    kind = case["kind"]
    if kind == "grouped":
        parts = [work(_fci(n, na, nb, "oz_bf16", 3)) for n, na, nb in _group(case)]
        return {k: sum(p[k] for p in parts) for k in ("bytes", "flops")}
    if kind == "spinor":
        size, n_el = math.comb(case["n"], case["ne"]), _elements([case["n"]], [case["ne"]], None, 0)
        return {"bytes": 32 * size, "flops": 8 * n_el}
    if kind == "das":
        spaces, ref, t = _das_of(case)
        return {"bytes": 16 * _target_size(spaces, ref, t), "flops": 2 * _elements(spaces, ref, ref, t)}
    if kind == "compressed":
        per_row = _elements(**{"spaces": LITERAL["spaces"], "ref_a": LITERAL["ref"], "ref_b": LITERAL["ref"],
                               "transfer": LITERAL["transfer"]}) / _target_size(**LITERAL)
        return {"bytes": 16 * case["nnz"] * (1 + per_row), "flops": 2 * case["nnz"] * per_row}
    size = math.comb(case["n"], case["na"]) * math.comb(case["n"], case["nb"])
    n_el = _elements_fci(case["n"], case["na"], case["nb"])
    if kind == "davidson":  # about 30 products, each with one pass over the subspace
        return {"bytes": 30 * 16 * size, "flops": 30 * 2 * n_el}
    return {"bytes": 16 * size, "flops": 2 * n_el}


def _elements_fci(n, na, nb):
    single = [k * (n - k) for k in (na, nb)]
    double = [math.comb(k, 2) * math.comb(n - k, 2) for k in (na, nb)]
    return math.comb(n, na) * math.comb(n, nb) * (1 + sum(single) + sum(double) + single[0] * single[1])


# ---------------------------------------------------------------------------- exact

def _strings(n, k):
    s = np.arange(1 << n, dtype=np.int64)
    return s[np.bitwise_count(s) == k]


def _move(strings, rank, a, b):
    """(target index, sign) of a+_b a_a applied to each string; sign 0 where it vanishes."""
    ok = ((strings >> a) & 1 == 1) & ((a == b) | ((strings >> b) & 1 == 0))
    lo, hi = min(a, b), max(a, b)
    between = strings & (((1 << hi) - 1) & ~((2 << lo) - 1))
    odd = between
    for shift in (16, 8, 4, 2, 1):
        odd = odd ^ (odd >> shift)
    target = torch.where(ok, rank[(strings & ~(1 << a)) | ((1 << b) * ok)], 0)
    return target, torch.where(ok, 1.0 - 2.0 * (odd & 1), 0.0)


def _ranked(n, k):
    s = torch.from_numpy(_strings(n, k)).cuda()
    rank = torch.zeros(1 << n, dtype=torch.int64, device="cuda")
    rank[s] = torch.arange(len(s), device="cuda")
    return s, rank


def _one_electron(h, g):
    return h - 0.5 * np.einsum("prrq->pq", g)


def _exact_ab(h, g, na, nb, C):
    """H C over alpha x beta strings, C of shape (N_alpha, N_beta)."""
    n = h.shape[0]
    pairs = [(p, q) for p in range(n) for q in range(p + 1)]
    P, Q = (np.array(v) for v in zip(*pairs))
    G = torch.from_numpy(0.5 * g[P, Q][:, P, Q]).cuda()
    one = torch.from_numpy(_one_electron(h, g)[P, Q]).cuda()

    def table(k):
        s, rank = _ranked(n, k)
        rows = []
        for p, q in pairs:
            t, x = _move(s, rank, p, q)
            if p != q:
                t2, x2 = _move(s, rank, q, p)
                t, x = torch.where(x2 != 0, t2, t), x + x2
            rows.append((t, x))
        return torch.stack([r[0] for r in rows]), torch.stack([r[1] for r in rows])

    (ta, xa), (tb, xb) = table(na), table(nb)
    out = E_CORE * C
    step = max(1, int(1.5e9 / (len(pairs) * C.shape[1])))
    for r0 in range(0, C.shape[0], step):
        r1 = min(C.shape[0], r0 + step)
        own = C[r0:r1]
        D = torch.empty(len(pairs), r1 - r0, C.shape[1], dtype=C.dtype, device=C.device)
        for i in range(len(pairs)):
            D[i] = xa[i, r0:r1, None] * C[ta[i, r0:r1]] + xb[i] * own[:, tb[i]]
        W = (G @ D.view(len(pairs), -1)).view_as(D)
        del D
        for i in range(len(pairs)):
            w = W[i] + one[i] * own
            out.index_add_(0, ta[i, r0:r1], xa[i, r0:r1, None] * w)
            out[r0:r1] += xb[i] * w[:, tb[i]]
    return out


def _exact_spinor(h, g, ne, C):
    n = h.shape[0]
    s, rank = _ranked(n, ne)
    G = torch.from_numpy(0.5 * g.reshape(n * n, n * n)).cuda()
    one = torch.from_numpy(_one_electron(h, g)).cuda()
    out = E_CORE * C
    step = max(1, int(4e8 / n**2))
    for k0 in range(0, len(s), step):
        part = s[k0:k0 + step]
        moves = {(a, b): _move(part, rank, a, b) for a in range(n) for b in range(n)}
        D = torch.stack([moves[a, b][1] * C[moves[a, b][0]] for a in range(n) for b in range(n)])
        W = G @ D
        del D
        for a in range(n):
            for b in range(n):  # <I|E_ab|K>: I = K - b + a
                t, x = moves[b, a]
                torch.view_as_real(out).index_add_(0, t, torch.view_as_real(x * (W[a * n + b] + one[a, b] * C[k0:k0 + step])))
    return out


def _das_blocks(spaces, ref, transfer):
    """Per spin pattern its strings' masks in local order, and the target (alpha, beta) pairs."""
    offsets = np.concatenate([[0], np.cumsum(spaces)])
    pats = list(_patterns(spaces, ref, transfer))
    masks = []
    for p, _, _ in pats:
        m = np.zeros(1, dtype=np.int64)
        for s, k in enumerate(p):  # the first space varies slowest
            m = (m[:, None] | (_strings(spaces[s], k) << int(offsets[s]))[None, :]).ravel()
        masks.append(m)
    pairs = [(i, j) for i, a in enumerate(pats) for j, b in enumerate(pats) if a[1] + b[1] <= transfer]
    return pats, masks, pairs


def _exact_das(case, h, g, C):
    spaces, ref, t = _das_of(case)
    n, k = sum(spaces), sum(ref)
    _, rank = _ranked(n, k)
    _, masks, pairs = _das_blocks(spaces, ref, t)
    index = [rank[torch.from_numpy(m).cuda()] for m in masks]
    size = math.comb(n, k)
    at = torch.cat([(index[i][:, None] * size + index[j][None, :]).reshape(-1) for i, j in pairs])
    full = torch.zeros(size * size, dtype=C.dtype, device=C.device)
    full[at] = C
    return _exact_ab(h, g, k, k, full.view(size, size)).view(-1)[at]


def _exact_compressed(case, h, g, addr, val):
    spaces, ref, t = _das_of(case)
    n = sum(spaces)
    pats, masks, pairs = _das_blocks(spaces, ref, t)
    pat_of = {p: i for i, (p, _, _) in enumerate(pats)}
    base = torch.full((len(pats) + 1, len(pats) + 1), -1, dtype=torch.int64)
    starts, order, o = [], [], 0
    for i, j in pairs:
        base[i, j] = o
        starts.append(o)
        order.append((i, j))
        o += len(masks[i]) * len(masks[j])
    base = base.cuda()
    width = torch.tensor([len(m) for m in masks] + [0]).cuda()
    offsets = np.concatenate([[0], np.cumsum(spaces)])
    # pattern and local index of a string from its sub-strings
    sub_rank, sub_count = [], []
    for m in spaces:
        r = np.zeros(1 << m, dtype=np.int64)
        for k in range(m + 1):
            r[_strings(m, k)] = np.arange(math.comb(m, k))
        sub_rank.append(torch.from_numpy(r).cuda())
        sub_count.append(torch.from_numpy(np.bitwise_count(np.arange(1 << m)).astype(np.int64)).cuda())
    key_of = torch.full((math.prod(m + 1 for m in spaces),), len(pats), dtype=torch.int64)
    for p, i in pat_of.items():
        key = 0
        for m, k in zip(spaces, p):
            key = key * (m + 1) + k
        key_of[key] = i
    key_of = key_of.cuda()
    combs = [torch.tensor([math.comb(m, k) for k in range(m + 1)]).cuda() for m in spaces]

    def locate(mask):
        key, loc = torch.zeros_like(mask), torch.zeros_like(mask)
        for s, m in enumerate(spaces):
            sub = (mask >> int(offsets[s])) & ((1 << m) - 1)
            c = sub_count[s][sub]
            key, loc = key * (m + 1) + c, loc * combs[s][c] + sub_rank[s][sub]
        return key_of[key], loc

    # the nonzero determinants' strings
    c = np.searchsorted(np.array(starts), addr.cpu().numpy(), side="right") - 1
    a0, b0 = [], []
    for x, k in zip(addr.cpu().numpy(), c):
        i, j = order[k]
        la, lb = divmod(int(x) - starts[k], len(masks[j]))
        a0.append(masks[i][la])
        b0.append(masks[j][lb])
    A, B = torch.tensor(a0).cuda(), torch.tensor(b0).cuda()

    def moves(A, B):
        """Every replacement E_ba of every determinant: rows, new strings, sign, a, b."""
        a, b = (v.reshape(-1).cuda() for v in torch.meshgrid(torch.arange(n), torch.arange(n), indexing="ij"))
        lo, hi = torch.minimum(a, b), torch.maximum(a, b)
        window = ((1 << hi) - 1) & ~((2 << lo) - 1)
        found = []
        for spin, S in enumerate((A, B)):
            ok = ((S[:, None] >> a) & 1 == 1) & ((a == b) | ((S[:, None] >> b) & 1 == 0))
            row, m = ok.nonzero(as_tuple=True)
            T = (S[row] & ~(1 << a[m])) | (1 << b[m])
            odd = S[row] & window[m]
            for shift in (16, 8, 4, 2, 1):
                odd = odd ^ (odd >> shift)
            found.append((row, T if spin == 0 else A[row], B[row] if spin == 0 else T, 1.0 - 2.0 * (odd & 1), a[m], b[m]))
        return [torch.cat(v) for v in zip(*found)]

    r1, A1, B1, x1, a1, b1 = moves(A, B)
    r2, A2, B2, x2, a2, b2 = moves(A1, B1)
    gd, hd = torch.from_numpy(g).cuda(), torch.from_numpy(_one_electron(h, g)).cuda()
    source = r1[r2]
    two = 0.5 * x1[r2] * x2 * gd[b2, a2, b1[r2], a1[r2]] * val[source]
    A3, B3 = torch.cat([A2, A1, A]), torch.cat([B2, B1, B])
    v3 = torch.cat([two, x1 * hd[b1, a1] * val[r1], E_CORE * val])
    (pa, la), (pb, lb) = locate(A3), locate(B3)
    start = base[pa, pb]
    ok = start >= 0
    place = (start + la * width[pb] + lb)[ok]
    where, inverse = torch.unique(place, return_inverse=True)
    return where, torch.zeros(len(where), dtype=torch.float64, device="cuda").index_add_(0, inverse, v3[ok])


def _lowest(apply, size, steps=160):
    """Lowest eigenvalue by Lanczos with full reorthogonalisation."""
    v = torch.randn(size, dtype=torch.float64, device="cuda", generator=torch.Generator(device="cuda").manual_seed(1))
    V, alpha, beta = [v / v.norm()], [], []
    for _ in range(min(steps, size)):
        w = apply(V[-1])
        alpha.append(float(w @ V[-1]))
        basis = torch.stack(V)
        for _ in range(2):
            w = w - basis.T @ (basis @ w)
        beta.append(float(w.norm()))
        if beta[-1] < 1e-12:
            break
        V.append(w / beta[-1])
    k = len(alpha)
    return float(np.linalg.eigvalsh(np.diag(alpha) + np.diag(beta[:k - 1], 1) + np.diag(beta[:k - 1], -1))[0])


def exact(case, seed):
    kind = case["kind"]
    if kind == "grouped":
        return [exact(_fci(n, na, nb, "fp64"), seed + 1000 * j) for j, (n, na, nb) in enumerate(_group(case))]
    if kind == "spinor":
        h, g = _integrals(case["n"], True, seed)
        return _exact_spinor(h, g, case["ne"], _vector(math.comb(case["n"], case["ne"]), True, seed))
    if kind in ("das", "compressed"):
        spaces, ref, t = _das_of(case)
        h, g = _integrals(sum(spaces), False, seed)
        if kind == "das":
            return _exact_das(case, h, g, _vector(_target_size(spaces, ref, t), False, seed))
        addr, val = _exact_compressed(case, h, g, *_coefficients(case, seed))
        return dict(addr=addr, val=val)
    h, g = _integrals(case["n"], False, seed)
    shape = [math.comb(case["n"], case[k]) for k in ("na", "nb")]
    if kind == "davidson":  # the vector's sign is free
        H = lambda v: _exact_ab(h, g, case["na"], case["nb"], v.view(shape)).view(-1)  # noqa: E731
        return dict(energy=_lowest(H, math.prod(shape)), vector=None)
    return _exact_ab(h, g, case["na"], case["nb"], _vector(math.prod(shape), False, seed).view(shape)).view(-1)
