"""Performance cases of the annealer: what a program of this library has it do, over the
sizes, bond dimensions, graph degrees, precisions and entry points that are used in earnest.

A case is a dict of plain values; `prepare` makes its inputs from a seed, `run` is one pass
through the public entry points, `work` is the work the pass cannot do without and `exact` is
the value of its outputs in plain 64-bit torch, written from the method alone.

Kinds of pass:

  anneal   one whole (coarse) anneal: create the state from the host arrays of the instance,
           layers 1..K, marginals, bond weights, destroy.  Every pass starts from |+>, so a
           repeated pass does the same work;
  bp       a fixed number of flooding sweeps from the warm start on a resident state;
  static   the same through the allocation-free entry point, on the caller's device arrays;
  circuit  rounds of arbitrary one- and two-qubit gates, each followed by BP and the regauge;
  sample   a short anneal, then a BP-guided measurement sampling of some qubits.

A vertex tensor is defined only up to a unitary on each of its bonds (a phase per bond index
where the bond weights differ), so the outputs of a pass that moves the state are the things
that do not depend on that choice and that a program reads: the bond weights lambda and the
marginals rho of every vertex.  The states of the mixed and complex64 precisions hold their
tensors in complex64, and a program keeps their results at that precision.
"""
import concurrent.futures
import math

import numpy as np
import torch

from paper_2409_12240_gb300 import gtqa as G

PRECISION = {"fp64": G.GTQA_FP64, "mixed": G.GTQA_MIXED, "c64": G.GTQA_C64}


# ---------------------------------------------------------------------------------------------
# the cases
# ---------------------------------------------------------------------------------------------
def listed():
    return [
        # the smallest: one small instance in FP64 (the size a user checks against exact
        # simulation); launches, barriers and the set-up are what it costs
        {"name": "anneal_n16_fp64", "kind": "anneal", "n": 16, "degree": 3, "chi": 4, "precision": "fp64",
         "K": 20, "dt": 0.1, "tol": 1e-12, "h": 0.1, "instances": 1},
        # the headline workload's instance size, bond dimension and precision
        {"name": "anneal_n1000_mixed", "kind": "anneal", "n": 1000, "degree": 3, "chi": 4, "precision": "mixed",
         "K": 16, "dt": 0.2, "tol": 1e-8, "h": 0.1, "instances": 1},
        # the same instance in FP64, the reference precision of a study
        {"name": "anneal_n1000_fp64", "kind": "anneal", "n": 1000, "degree": 3, "chi": 4, "precision": "fp64",
         "K": 12, "dt": 0.2, "tol": 1e-8, "h": 0.1, "instances": 1},
        # a batch of uneven instances in one state: the throughput mode
        {"name": "anneal_batch32_mixed", "kind": "anneal", "n": 1000, "degree": 3, "chi": 4, "precision": "mixed",
         "K": 8, "dt": 0.2, "tol": 1e-8, "h": 0.1, "instances": 32},
        # larger bond dimension in FP64, odd number of vertices (one vertex of lower degree)
        {"name": "anneal_n401_chi8_fp64", "kind": "anneal", "n": 401, "degree": 3, "chi": 8, "precision": "fp64",
         "K": 8, "dt": 0.2, "tol": 1e-8, "h": 0.1, "instances": 1},
        # the largest: a big graph at chi = 8 in the mixed precision
        {"name": "anneal_n12000_chi8_mixed", "kind": "anneal", "n": 12000, "degree": 3, "chi": 8, "precision": "mixed",
         "K": 5, "dt": 0.2, "tol": 1e-8, "h": 0.1, "instances": 1},
        # the largest bond dimension of a bond-dimension sweep
        {"name": "anneal_n200_chi16_fp64", "kind": "anneal", "n": 200, "degree": 3, "chi": 16, "precision": "fp64",
         "K": 6, "dt": 0.2, "tol": 1e-8, "h": 0.1, "instances": 1},
        # random 4-regular graphs
        {"name": "anneal_n200_degree4_mixed", "kind": "anneal", "n": 200, "degree": 4, "chi": 4, "precision": "mixed",
         "K": 10, "dt": 0.2, "tol": 1e-10, "h": 0.1, "instances": 1},
        # every step in complex64, the lowest precision of a precision study
        {"name": "anneal_n1000_c64", "kind": "anneal", "n": 1000, "degree": 3, "chi": 4, "precision": "c64",
         "K": 8, "dt": 0.2, "tol": 1e-6, "h": 0.1, "instances": 1},
        # BP to its sweep limit, as most layers of a long anneal with weak fields run it
        {"name": "bp100_n1000_mixed", "kind": "bp", "n": 1000, "degree": 3, "chi": 4, "precision": "mixed",
         "sweeps": 100},
        # a random circuit of arbitrary gates, FP64
        {"name": "circuit_n300_fp64", "kind": "circuit", "n": 300, "degree": 3, "chi": 4, "precision": "fp64",
         "rounds": 2, "tol": 1e-10},
        # measurement sampling of a degenerate instance (no fields): many small dependent launches
        {"name": "sample_n120_fp64", "kind": "sample", "n": 120, "degree": 3, "chi": 4, "precision": "fp64",
         "K": 6, "dt": 0.2, "tol": 1e-9, "qubits": 30},
    ]


def _logint(rng, lo, hi):
    return int(round(math.exp(rng.uniform(math.log(lo), math.log(hi)))))


def draw(rng):
    kind = rng.choice(["anneal", "anneal", "anneal", "batch", "plain", "plain", "bp", "static", "circuit", "sample"])
    h = rng.choice([0.1, 0.1, 1.0])
    if kind == "anneal":
        chi = rng.choice([2, 3, 4, 4, 6, 8])
        prec = rng.choice(["fp64", "mixed", "mixed"])
        top = {2: 4000, 3: 2500, 4: 2500}.get(chi, 500 if prec == "fp64" else 1500)
        return {"kind": "anneal", "n": _logint(rng, 10, top), "degree": 3, "chi": chi, "precision": prec,
                "K": rng.randint(4, 12), "dt": rng.choice([0.1, 0.2]), "tol": rng.choice([1e-8, 1e-10]), "h": h,
                "instances": 1}
    if kind == "batch":
        return {"kind": "anneal", "n": _logint(rng, 60, 800), "degree": 3, "chi": 4,
                "precision": rng.choice(["fp64", "mixed"]), "K": rng.randint(4, 8), "dt": 0.2, "tol": 1e-8, "h": h,
                "instances": rng.randint(2, 20)}
    if kind == "plain":
        form = rng.choice(["degree4", "degree4", "chi16", "c64"])
        if form == "degree4":
            return {"kind": "anneal", "n": _logint(rng, 10, 500), "degree": 4, "chi": rng.choice([2, 3, 4]),
                    "precision": rng.choice(["fp64", "mixed"]), "K": rng.randint(4, 10), "dt": rng.choice([0.1, 0.2]),
                    "tol": 1e-9, "h": h, "instances": 1}
        if form == "chi16":
            return {"kind": "anneal", "n": _logint(rng, 12, 160), "degree": 3, "chi": rng.choice([12, 16]),
                    "precision": rng.choice(["fp64", "mixed", "c64"]), "K": rng.randint(4, 6), "dt": 0.2, "tol": 1e-6,
                    "h": h, "instances": 1}
        return {"kind": "anneal", "n": _logint(rng, 10, 1500), "degree": rng.choice([3, 3, 4]),
                "chi": rng.choice([2, 4]), "precision": "c64", "K": rng.randint(4, 8), "dt": 0.2, "tol": 1e-6, "h": h,
                "instances": 1}
    if kind == "bp":
        chi = rng.choice([2, 4, 4, 8])
        return {"kind": "bp", "n": _logint(rng, 12, 5000 if chi < 8 else 600), "degree": 3, "chi": chi,
                "precision": rng.choice(["fp64", "mixed", "mixed"]), "sweeps": rng.randint(5, 100)}
    if kind == "static":
        return {"kind": "static", "n": _logint(rng, 12, 2000), "degree": 3, "chi": 4, "precision": "fp64",
                "sweeps": rng.randint(5, 60)}
    if kind == "circuit":
        return {"kind": "circuit", "n": _logint(rng, 12, 400), "degree": rng.choice([3, 3, 4]), "chi": rng.choice([2, 4]),
                "precision": rng.choice(["fp64", "mixed"]), "rounds": rng.randint(1, 2), "tol": 1e-10}
    n = _logint(rng, 16, 150)
    return {"kind": "sample", "n": n, "degree": 3, "chi": rng.choice([2, 4]), "precision": "fp64",
            "K": rng.randint(4, 8), "dt": 0.2, "tol": 1e-9, "qubits": rng.randint(4, min(n, 30))}


# ---------------------------------------------------------------------------------------------
# inputs
# ---------------------------------------------------------------------------------------------
def _graph(n, d, rng):
    """A random simple graph of degree d by the pairing model, bad pairs re-drawn; with n odd some
    edges are left out, so that vertices of lower degree occur and d colours still suffice.
    Sorted (m, 2) int32 edges, u < v."""
    stubs = rng.permutation(np.repeat(np.arange(n), d))
    p = stubs[: len(stubs) // 2 * 2].reshape(-1, 2)
    for _ in range(1000):
        a, b = p.min(1), p.max(1)
        key = a * n + b
        order = np.argsort(key, kind="stable")
        bad = a == b
        bad[order[1:]] |= key[order[1:]] == key[order[:-1]]
        if not bad.any():
            break
        mix = np.nonzero(bad)[0]
        mix = np.unique(np.concatenate([mix, rng.integers(0, len(p), 3 * len(mix) + 4)]))
        p[mix] = rng.permutation(p[mix].ravel()).reshape(-1, 2)
    else:
        raise RuntimeError("no simple graph found")
    e = np.stack([p.min(1), p.max(1)], 1)
    if n % 2:
        e = rng.permutation(e)[: len(e) - max(3, len(e) // 40)]
    return e[np.lexsort((e[:, 1], e[:, 0]))].astype(np.int32)


def _instances(case, seed):
    """The problem instances of a case: (n, edges, colour, J, h) each."""
    rng = np.random.default_rng([int(seed), 2409])
    out, B = [], case.get("instances", 1)
    for b in range(B):
        n = case["n"]
        if B > 1:   # uneven sizes spread over n / 20 .. n, even numbers of vertices
            n = 2 * (max(n // 40, 4) + (n // 2 - max(n // 40, 4)) * (b * 7 % B) // max(B - 1, 1))
        e = _graph(n, case["degree"], rng)
        J = rng.standard_normal(len(e))
        h = rng.standard_normal(n) * case.get("h", 0.0)
        out.append((n, e, G.gtqa_edge_colouring(n, e)[0], J, h))
    return out


def _storage(chi):
    return next(c for c in (2, 4, 8, 16) if c >= chi)


def _slots(n, edges):
    """Edge at every bond slot of every vertex (-1: none), and each edge's slot at its ends; a
    vertex's slots are its edges in ascending id."""
    deg = np.zeros(n, dtype=np.int64)
    D = 4 if len(edges) and np.bincount(edges.ravel(), minlength=n).max() > 3 else 3
    at = np.full((n, D), -1, dtype=np.int64)
    sl = np.zeros((len(edges), 2), dtype=np.int64)
    for e, (u, v) in enumerate(edges.tolist()):
        for x, w in ((0, u), (1, v)):
            at[w, deg[w]] = e
            sl[e, x] = deg[w]
            deg[w] += 1
    return D, at, sl


def _resident(case, seed):
    """A state in the middle of an anneal as host arrays: bond weights that fall off by a random
    factor per index, tensors near the Vidal gauge (unit columns on every bond)."""
    n, e, colour, J, h = _instances(case, seed)[0]
    rng = np.random.default_rng([int(seed), 77])
    C = _storage(case["chi"])
    D, at, _ = _slots(n, e)
    lam = np.exp(-np.arange(case["chi"]) * rng.uniform(0.7, 1.5, (len(e), 1)))
    lam = np.pad(lam / np.linalg.norm(lam, axis=1, keepdims=True), ((0, 0), (0, C - case["chi"])))
    g = rng.standard_normal((n, 2) + (C,) * D) + 1j * rng.standard_normal((n, 2) + (C,) * D)
    for k in range(D):
        keep = np.where(at[:, k, None] >= 0, lam[at[:, k]] > 0, np.arange(C) == 0)
        g *= keep.reshape((n, 1) + (1,) * k + (C,) + (1,) * (D - 1 - k))
    g /= math.sqrt(4.0)
    msg = np.zeros((2 * len(e), C, C), dtype=np.complex128)
    i = np.arange(C)
    msg[:, i, i] = np.repeat(lam / lam.sum(1, keepdims=True), 2, axis=0)
    return n, e, colour, J, h, g, lam, msg


def _gates(case, m, n, seed):
    """Haar-random two-qubit gates on every edge (in a random order) and one-qubit gates on every
    vertex, per round."""
    rng = np.random.default_rng([int(seed), 5])

    def haar(count, k):
        a = rng.standard_normal((count, k, k)) + 1j * rng.standard_normal((count, k, k))
        q, r = np.linalg.qr(a)
        d = np.diagonal(r, axis1=1, axis2=2)
        return q * (d / np.abs(d))[:, None, :]

    return [(rng.permutation(m).astype(np.int32), haar(m, 4), np.arange(n, dtype=np.int32), haar(n, 2))
            for _ in range(case["rounds"])]


def _sampling(case, seed):
    rng = np.random.default_rng([int(seed), 6])
    return rng.permutation(case["n"])[: case["qubits"]].astype(np.int32), rng.uniform(0.02, 0.98, case["qubits"])


class State:
    """What a program has in hand before the call; gives the handle it keeps back."""

    def __init__(self, **kw):
        self.handle = 0
        self.__dict__.update(kw)

    def __del__(self):
        if self.handle:
            G.gtqa_destroy(self.handle)
            self.handle = 0


def _options(case):
    return G.gtqa_options_init(precision=PRECISION[case["precision"]])


def prepare(case, seed):
    if case["kind"] in ("anneal", "circuit", "sample"):
        s = State(case=case, inst=_instances(case, seed), opt=_options(case))
        if case["kind"] == "circuit":
            s.gates = _gates(case, len(s.inst[0][1]), s.inst[0][0], seed)
        if case["kind"] == "sample":
            s.order, s.u = _sampling(case, seed)
        return s
    n, e, colour, J, h, g, lam, msg = _resident(case, seed)
    if case["kind"] == "bp":
        s = State(case=case, n=n, m=len(e), C=lam.shape[1],
                  handle=G.gtqa_create(n, e, J, h, case["chi"], colour, _options(case)))
        G.gtqa_set_state(s.handle, g, lam, msg)
        return s
    D, at, sl = _slots(n, e)
    deg = (at >= 0).sum(1, keepdims=True)
    dev = lambda a, t: torch.from_numpy(np.ascontiguousarray(a).astype(t)).cuda()  # noqa: E731
    return State(case=case, n=n, m=len(e), vert=dev(np.concatenate([at, deg], 1), np.int32),
                 edge=dev(np.concatenate([e, sl], 1), np.int32), g=dev(g, np.complex128), lam=dev(lam, np.float64),
                 out=torch.empty((2 * len(e), 4, 4), dtype=torch.complex128, device="cuda"))


# ---------------------------------------------------------------------------------------------
# one pass
# ---------------------------------------------------------------------------------------------
def _create(s):
    if len(s.inst) == 1:
        n, e, colour, J, h = s.inst[0]
        return G.gtqa_create(n, e, J, h, s.case["chi"], colour, s.opt)
    ns, es, cs, Js, hs = zip(*s.inst)
    return G.gtqa_create_batch(ns, es, Js, hs, s.case["chi"], cs, s.opt)


def _read(s, handle):
    """Marginals, bond weights and (FP64) the read-out signs.  In the lower precisions the sign
    of a vertex whose two outcomes are equal to rounding is not defined, so rho alone is read."""
    n, m, C, _ = G.gtqa_sizes(handle)
    rho = torch.empty((n, 2, 2), dtype=torch.complex128, device="cuda")
    lam = torch.empty((m, C), dtype=torch.float64, device="cuda")
    _, sign = G.gtqa_marginals(handle, rho)
    G._check(G.load().gtqa_get_state(handle, None, lam.data_ptr(), None), "gtqa_get_state")
    if s.case["precision"] == "fp64":
        return {"rho": rho, "lam": lam, "sign": sign} if s.case.get("h", 0.0) else {"rho": rho, "lam": lam}
    return {"rho": rho.to(torch.complex64), "lam": lam.to(torch.float32)}


def run(s):
    c = s.case
    if c["kind"] == "static":
        G.gtqa_bp_static(s.n, s.m, s.vert, s.edge, s.g, s.lam, s.out, 0.0, c["sweeps"])
        return {"messages": s.out}
    if c["kind"] == "bp":
        G.gtqa_bp_sweep(s.handle, 0.0, c["sweeps"], G.GTQA_BP_WARM_START)
        msg = np.empty((2 * s.m, s.C, s.C), dtype=np.complex128)
        G._check(G.load().gtqa_get_state(s.handle, None, None, msg.ctypes.data), "gtqa_get_state")
        return {"messages": msg if c["precision"] == "fp64" else msg.astype(np.complex64)}
    handle = _create(s)
    try:
        if c["kind"] == "circuit":
            for edge, U, vertex, W in s.gates:
                G.gtqa_apply_single_qubit_gates(handle, vertex, W)
                G.gtqa_apply_gates(handle, edge, U)
                G.gtqa_bp_sweep(handle, c["tol"], 100, G.GTQA_BP_DEFAULT)
            return _read(s, handle)
        G.gtqa_anneal(handle, 1, c["K"], c["K"], c["dt"], c["tol"], 100)
        if c["kind"] == "anneal":
            return _read(s, handle)
        x, p = G.gtqa_sample(handle, s.order, s.u, c["tol"], 100)
        return {**_read(s, handle), "x": x, "p": p}
    finally:
        G.gtqa_destroy(handle)


# ---------------------------------------------------------------------------------------------
# the work of a pass
# ---------------------------------------------------------------------------------------------
def work(case):
    """Bytes: the instance or state read once and the results written once.  Flops: the method's
    steps per edge, directed message and sweep (two Householder QRs and an SVD of the 2 chi core
    per gate, three contractions per message, two eigen-decompositions and an SVD per regauged
    edge), with two sweeps for a BP run that stops by itself."""
    chi, D = case["chi"], case["degree"]
    B = case.get("instances", 1)
    n = case["n"] * (0.525 if B > 1 else 1.0) * B
    m = n * D / 2
    NR, N = chi ** (D - 1), 2 * chi
    qr = 4 * 8 * NR * chi * chi
    gate = qr + 8 * N ** 3 + 7.5 * 11 * N * N * (N - 1) / 2 + 2 * qr
    msg = 8 * D * 2 * chi ** (D + 1)
    edge = 3 * (7.5 * 11 * chi * chi * (chi - 1) / 2) + 6 * 8 * chi ** 3 + 2 * 8 * 2 * chi ** (D + 1)
    item = 16 if case["precision"] == "fp64" else 8
    results = n * 4 * item + m * chi * item / 2
    if case["kind"] in ("bp", "static"):
        return {"bytes": n * 2 * chi ** D * item + m * chi * 8 + 2 * m * chi * chi * item,
                "flops": case["sweeps"] * 2 * m * msg}
    if case["kind"] == "circuit":
        big = 4 * chi
        general = 2 * 8 * NR * N * N + 8 * 4 * N ** 3 + 7.5 * 11 * big * big * (big - 1) / 2 + 4 * 8 * NR * N * chi
        return {"bytes": case["rounds"] * (m * 260 + n * 68) + m * 20 + results,
                "flops": case["rounds"] * (m * (general + edge) + 2 * 2 * m * msg)}
    runs = case["K"] + case.get("qubits", 0)
    return {"bytes": m * 20 + n * 8 + results,
            "flops": case["K"] * m * gate + runs * (m * edge + 2 * 2 * m * msg)}


# ---------------------------------------------------------------------------------------------
# the same in plain 64-bit torch
# ---------------------------------------------------------------------------------------------
def _svd(a):
    """LAPACK's divide-and-conquer SVD stops the process on some rank-deficient matrices of order
    above 25, so those are decomposed on the GPU."""
    if a.shape[-1] <= 25:
        return _chunked(torch.linalg.svd, a)
    return tuple(x.cpu() for x in torch.linalg.svd(a.cuda()))


def _chunked(f, a, size=512):
    """f over the leading axis of a in chunks on the host's cores (LAPACK runs one matrix at a time)."""
    if len(a) <= size:
        return f(a)
    with concurrent.futures.ThreadPoolExecutor(max_workers=16) as pool:
        return tuple(torch.cat(x) for x in zip(*pool.map(f, a.split(size))))


class _Network:
    """The state and the steps of the method (App. B, C, D, E) in complex128 on the CPU, batched
    over the edges of a colour and over the vertices; bonds padded to chi with zero weight."""

    SVD_CUT, EIG_CUT = 1e-14, 1e-13

    def __init__(self, n, edges, chi):
        self.n, self.m, self.chi = n, len(edges), chi
        self.D, at, sl = _slots(n, edges)
        self.at, self.sl, self.e = torch.from_numpy(at), torch.from_numpy(sl), torch.from_numpy(edges.astype(np.int64))
        self.g = torch.zeros((n, 2) + (chi,) * self.D, dtype=torch.complex128)
        self.g[(slice(None), slice(None)) + (0,) * self.D] = math.sqrt(0.5)
        self.lam = torch.zeros((self.m, chi), dtype=torch.float64)
        self.lam[:, 0] = 1.0

    def weights(self):
        """lambda on every slot of every vertex; a missing slot has dimension 1."""
        one = torch.zeros(self.chi, dtype=torch.float64)
        one[0] = 1.0
        return torch.where(self.at[:, :, None] >= 0, self.lam[self.at.clamp(min=0)], one)

    def along(self, v, k):
        return v.reshape((self.n, 1) + (1,) * k + (self.chi,) + (1,) * (self.D - 1 - k))

    def side(self, idx, x):
        """(q, 2, chi^(D-1), chi) tensors of the x ends of edges idx, bond last, and the weights
        of the other slots."""
        v, s = self.e[idx, x], self.sl[idx, x]
        NR = self.chi ** (self.D - 1)
        A = torch.empty((len(idx), 2, NR, self.chi), dtype=torch.complex128)
        w = torch.empty((len(idx), NR), dtype=torch.float64)
        W = self.weights()[v]
        for k in range(self.D):
            q = s == k
            if not q.any():
                continue
            A[q] = self.g[v[q]].movedim(2 + k, -1).reshape(-1, 2, NR, self.chi)
            t = torch.ones((int(q.sum()), 1), dtype=torch.float64)
            for o in range(self.D):
                if o != k:
                    t = (t[:, :, None] * W[q][:, None, o]).reshape(len(t), -1)
            w[q] = t
        return A, w

    def put(self, idx, x, A):
        v, s = self.e[idx, x], self.sl[idx, x]
        for k in range(self.D):
            q = s == k
            if not q.any():
                continue
            B = A[q].reshape((-1, 2) + (self.chi,) * self.D)
            self.g[v[q]] = B.movedim(-1, 2 + k)

    def gate(self, idx, U, diagonal):
        """The simple update of edges idx (disjoint) with the matrices U, and the truncation."""
        chi, N = self.chi, len(idx)
        (A, wa), (B, wb) = self.side(idx, 0), self.side(idx, 1)
        wA, wB = wa[:, None, :, None] * A, wb[:, None, :, None] * B
        l = self.lam[idx]
        if diagonal:   # block by block of the physical index: a 2 chi x 2 chi core
            Qa, Ra = _chunked(torch.linalg.qr, wA)
            Qb, Rb = _chunked(torch.linalg.qr, wB)
            M = torch.einsum("qabab,qarj,qj,qbsj->qarbs", U.reshape(N, 2, 2, 2, 2), Ra, l.to(A.dtype), Rb)
            r = chi
        else:          # both physical components of a side together
            flat = lambda t: t.movedim(1, 2).reshape(N, t.shape[2], 2 * chi)  # noqa: E731
            Qa, Ra = torch.linalg.qr(flat(wA))
            Qb, Rb = torch.linalg.qr(flat(wB))
            r = Ra.shape[1]
            Ra, Rb = Ra.reshape(N, r, 2, chi), Rb.reshape(N, r, 2, chi)
            K = torch.einsum("qrcj,qj,qsdj->qcrds", Ra, l.to(A.dtype), Rb)
            M = torch.einsum("qabcd,qcrds->qarbs", U.reshape(N, 2, 2, 2, 2), K)
            Qa, Qb = Qa[:, None], Qb[:, None]
        u, s, vh = _svd(M.reshape(N, 2 * r, 2 * r))
        u, s, v = u[:, :, :chi], s[:, :chi], vh[:, :chi].transpose(1, 2)
        keep = s > self.SVD_CUT * s[:, :1]
        keep[:, 0] = True
        s = s * keep
        self.lam[idx] = s / torch.linalg.norm(s, dim=1, keepdim=True)
        for x, Q, t, w in ((0, Qa, u, wa), (1, Qb, v, wb)):
            new = Q @ (t * keep[:, None]).reshape(N, 2, r, chi)
            self.put(idx, x, new * torch.where(w > 0, 1.0 / w, 0.0)[:, None, :, None])

    def one_qubit(self, W):
        self.g = torch.einsum("nab,nbj->naj", W, self.g.reshape(self.n, 2, -1)).reshape(self.g.shape)

    def ising(self, classes, J, h, tZ, tX):
        deg = (self.at >= 0).sum(1)
        z = torch.tensor([1.0, -1.0], dtype=torch.float64)
        f = h / deg.clamp(min=1)
        for idx in classes:
            a, b = self.e[idx, 0], self.e[idx, 1]
            E = J[idx, None, None] * z[:, None] * z[None] + f[a, None, None] * z[:, None] + f[b, None, None] * z[None]
            U = torch.diag_embed(torch.exp(-1j * tZ * E).reshape(-1, 4))
            self.gate(idx, U, True)
        c, s = math.cos(tX), -1j * math.sin(tX)
        self.one_qubit(torch.tensor([[c, s], [s, c]], dtype=torch.complex128).expand(self.n, 2, 2))

    def bp(self, tol, limit, parts, exact_sweeps=False):
        """Flooding BP from the warm start; `parts`: (first edge, end, first vertex, end) of every
        instance, each of which stops by itself.  Leaves T and the messages (2m, chi, chi)."""
        chi, D, at = self.chi, self.D, self.at
        T = self.g
        for k, w in enumerate(self.weights().sqrt().unbind(1)):
            T = T * self.along(w, k)
        self.T = T
        m0 = self.lam / self.lam.sum(1, keepdim=True)
        self.msg = torch.diag_embed(m0).repeat_interleave(2, 0).to(torch.complex128)
        first = self.e[at.clamp(min=0), 0] == torch.arange(self.n)[:, None]
        out = 2 * at + torch.where(first, 0, 1)
        inn = 2 * at + torch.where(first, 1, 0)
        phantom = torch.zeros((chi, chi), dtype=torch.complex128)
        phantom[0, 0] = 1.0
        real = at >= 0
        open_ = [m1 > m_0 for m_0, m1, _, _ in parts]
        for _ in range(limit):
            min_ = torch.where(real[:, :, None, None], self.msg[inn.clamp(min=0)], phantom)
            new = torch.zeros_like(self.msg)
            for s in range(D):
                X = T.reshape(self.n, 2, -1)
                for o in range(D):
                    if o != s:
                        Y = X.reshape(self.n, 2 * chi ** o, chi, chi ** (D - 1 - o))
                        X = torch.einsum("nlqr,nqx->nlxr", Y, min_[:, o])
                Xs = X.reshape(self.n, 2 * chi ** s, chi, -1).movedim(2, 1).reshape(self.n, chi, -1)
                Ts = T.reshape(self.n, 2 * chi ** s, chi, -1).movedim(2, 1).reshape(self.n, chi, -1)
                F = Xs @ Ts.conj().transpose(1, 2)
                F = F / torch.diagonal(F, dim1=1, dim2=2).sum(1)[:, None, None]
                new[out[real[:, s], s]] = F[real[:, s]]
            for b, (e0, e1, _, _) in enumerate(parts):
                if not open_[b]:
                    new[2 * e0:2 * e1] = self.msg[2 * e0:2 * e1]
                elif not exact_sweeps:
                    d = new[2 * e0:2 * e1] - self.msg[2 * e0:2 * e1]
                    # the Frobenius norm bounds the trace norm from below
                    if float(torch.linalg.matrix_norm(d).sum()) < tol * (e1 - e0):
                        open_[b] = not float(torch.linalg.svdvals(d).sum()) < tol * (e1 - e0)
            self.msg = new
            if not any(open_):
                break

    def regauge(self):
        M = (self.msg + self.msg.mH) / 2
        w, V = _chunked(torch.linalg.eigh, M)
        keep = w > self.EIG_CUT * w[:, -1:]
        root = torch.where(keep, w, 0.0).sqrt()
        sq = (V * root[:, None].to(V.dtype)) @ V.mH
        isq = (V * torch.where(keep, 1.0 / root.clamp(min=1e-300), 0.0)[:, None].to(V.dtype)) @ V.mH
        u, s, vh = _svd(sq[0::2].mT @ sq[1::2])
        keep = s > self.SVD_CUT * s[:, :1]
        nrm = torch.linalg.norm(s, dim=1)
        Xa = isq[0::2].conj() @ (u * keep[:, None])
        Xb = isq[1::2].conj() @ (vh.mT * keep[:, None])
        X = torch.stack([Xa, Xb], 1) * nrm.sqrt()[:, None, None, None]
        self.lam = s * keep / nrm[:, None]
        g, one = self.T, torch.eye(self.chi, dtype=torch.complex128)
        for k in range(self.D):
            ek = self.at[:, k]
            side = torch.where(self.e[ek.clamp(min=0), 0] == torch.arange(self.n), 0, 1)
            Xk = torch.where((ek >= 0)[:, None, None], X[ek.clamp(min=0), side], one)
            g = torch.einsum("nlqr,nqx->nlxr", g.reshape(self.n, 2 * self.chi ** k, self.chi, -1), Xk)
        self.g = g.reshape(self.T.shape)

    def rho(self):
        A = self.g
        for k, w in enumerate(self.weights().unbind(1)):
            A = A * self.along(w, k)
        A = A.reshape(self.n, 2, -1)
        r = A @ A.mH
        return r / torch.diagonal(r, dim1=1, dim2=2).sum(1).real[:, None, None]


def _joined(inst, chi):
    """One network over all instances (disjoint), its colour classes, couplings and parts."""
    es, parts, n0, e0 = [], [], 0, 0
    for n, e, _, _, _ in inst:
        es.append(e.astype(np.int64) + n0)
        parts.append((e0, e0 + len(e), n0, n0 + n))
        n0, e0 = n0 + n, e0 + len(e)
    net = _Network(n0, np.concatenate(es), chi)
    col = np.concatenate([i[2] for i in inst])
    classes = [torch.from_numpy(np.nonzero(col == k)[0]) for k in range(int(col.max()) + 1)]
    J, h = (torch.from_numpy(np.concatenate([i[k] for i in inst])) for k in (3, 4))
    return net, classes, J, h, parts


def exact(case, seed):
    chi, C = case["chi"], _storage(case["chi"])
    if case["kind"] in ("bp", "static"):
        n, e, _, _, _, g, lam, _ = _resident(case, seed)
        net = _Network(n, e, C)
        net.g, net.lam = torch.from_numpy(g), torch.from_numpy(lam)
        net.bp(0.0, case["sweeps"], [(0, len(e), 0, n)], True)
        return {"messages": net.msg}
    inst = _instances(case, seed)
    net, classes, J, h, parts = _joined(inst, chi)
    extra = {}
    if case["kind"] == "circuit":
        for edge, U, _, W in _gates(case, net.m, net.n, seed):
            net.one_qubit(torch.from_numpy(W))
            # a gate goes one batch after the last earlier gate that shares a vertex with it
            free, layer = [0] * net.n, np.zeros(len(edge), dtype=np.int64)
            for q, (a, b) in enumerate(inst[0][1][edge].tolist()):
                layer[q] = max(free[a], free[b])
                free[a] = free[b] = layer[q] + 1
            for q in range(int(layer.max()) + 1):
                sel = layer == q
                net.gate(torch.from_numpy(edge[sel].astype(np.int64)), torch.from_numpy(U[sel]), False)
            net.bp(case["tol"], 100, parts)
            net.regauge()
    else:
        for k in range(1, case["K"] + 1):
            tau = k / case["K"]
            net.ising(classes, J, h, case["dt"] * tau, case["dt"] * (1.0 - tau))
            net.bp(case["tol"], 100, parts)
            net.regauge()
    if case["kind"] == "sample":
        order, u = _sampling(case, seed)
        x, p = np.zeros(net.n, dtype=np.int8), np.zeros(len(order))
        for q, a in enumerate(order.tolist()):
            p0 = float(net.rho()[a, 0, 0].real)
            up = u[q] < p0
            x[a], p[q] = (1, p0) if up else (-1, 1.0 - p0)
            net.g[a, 1 if up else 0] = 0.0
            net.bp(case["tol"], 100, parts)
            net.regauge()
        extra = {"x": x, "p": p}
    rho = net.rho()
    lam = torch.nn.functional.pad(net.lam, (0, C - chi))
    out = {"rho": rho, "lam": lam, **extra}
    if case["precision"] == "fp64" and case.get("h", 0.0):
        out["sign"] = torch.where(rho[:, 0, 0].real > 0.5, 1, -1).to(torch.int8)
    return out
