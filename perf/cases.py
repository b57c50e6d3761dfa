"""The work that a user of the optimal-cycle-mean solver has it do, as cases to
be timed: whole calls of the public entry points (``solve``, ``solve_batch``,
``solve_scc``, ``backward``, ``backward_batch``, ``OCMFunction``) on the graph
families of ``synth/``, generated on the GPU from a seed.

A case names a family and its sizes; the families are

========  ==================================================================
ring      ring i -> i+1 plus U{0..4} uniform extra edges, w in U[1,100]
product   P processes x S-state ring with 2 chords a state, all interleavings,
          states numbered in the order a breadth-first search finds them,
          w in U[0,1000] (a model checker's state space)
locality  out-degree 4/16/64, targets i + 1 + floor|N(0,4096)|,
          w in U[-1000,1000], minimum
resolve   the locality graph solved again from the last policy after one
          weight in 64 changed, with the optimality certificate
diff      ring plus U{0..7} extras, forward and backward through autograd
ratio     ring plus U{0..7} extras with transit times U[1,8], optimal cycle
          ratio and its gradient
single    the product family in the single-lambda form
batch     G graphs, n_g log-uniform in [100, nmax], ring plus U{0..7} extras,
          w in U[1,10000], one batched solve and its gradient
hub       ring plus 3 extras and one vertex with many more out-edges
scc       a random digraph, out-degree Poisson(1.5), 5% sinks: its components
          and the optimum of each
========  ==================================================================
"""
from __future__ import annotations

import math

import torch

import paper_1111_0627_gb300 as ocm

INT32_MAX = 2**31 - 1


def listed():
    return [
        # the smallest call: one small system (a marked graph, a controller), where launches count
        {"name": "ring_257", "family": "ring", "n": 257},
        # the repository's small benchmark graph
        {"name": "ring_10k", "family": "ring", "n": 10_000},
        # a model checker's state space, the paper's own use (38^4 = 2,085,136 states)
        {"name": "product_4x38", "family": "product", "P": 4, "S": 38},
        # the largest single graph: 2^25 vertices, 2.7e8 edges, the benchmark's default
        {"name": "locality_32m", "family": "locality", "n": 1 << 25},
        # a system that changed a little is solved again, with its certificate; an odd size
        {"name": "resolve_3m", "family": "resolve", "n": 3_000_017},
        # lambda* inside a training loop: one forward and one backward
        {"name": "diff_1m", "family": "diff", "n": 1 << 20},
        # cost over time instead of cost over steps, and its gradient
        {"name": "ratio_400k", "family": "ratio", "n": 400_009},
        # the paper's own form of the iteration, on a smaller state space (331,776 states)
        {"name": "single_4x24", "family": "single", "P": 4, "S": 24},
        # many independent systems at once: 4,096 of up to 20,000 vertices
        {"name": "batch_4096_20k", "family": "batch", "G": 4096, "nmax": 20_000},
        # fewer and larger ones, up to 200,000 vertices
        {"name": "batch_1024_200k", "family": "batch", "G": 1024, "nmax": 200_000},
        # skewed degrees: one vertex with four million out-edges
        {"name": "hub_4m", "family": "hub", "n": 1 << 20, "hub": 4_000_000},
        # a graph that is not strongly connected: every component's own optimum
        {"name": "scc_10m", "family": "scc", "n": 10_000_000},
    ]


def _log_int(rng, lo, hi):
    return int(round(math.exp(rng.uniform(math.log(lo), math.log(hi)))))


def draw(rng):
    f = rng.choice(["ring", "product", "locality", "resolve", "diff", "ratio", "single", "batch",
                    "batch", "hub", "scc"])
    if f == "ring":
        return {"family": f, "n": _log_int(rng, 100, 200_000)}
    if f in ("product", "single"):
        P = rng.choice([3, 4])
        top = 38 if f == "product" else 24
        return {"family": f, "P": P, "S": rng.randint(8, top) if P == 4 else rng.randint(20, 100)}
    if f == "locality":
        return {"family": f, "n": _log_int(rng, 1 << 16, 1 << 25)}
    if f == "resolve":
        return {"family": f, "n": _log_int(rng, 1 << 16, 1 << 22)}
    if f == "diff":
        return {"family": f, "n": _log_int(rng, 1 << 10, 1 << 20)}
    if f == "ratio":
        return {"family": f, "n": _log_int(rng, 1 << 10, 1 << 20)}
    if f == "batch":
        nmax = _log_int(rng, 1000, 200_000)
        most = min(4096, 1024 * 200_000 // nmax)
        return {"family": f, "G": _log_int(rng, 64, most), "nmax": nmax}
    if f == "hub":
        return {"family": f, "n": _log_int(rng, 1 << 16, 1 << 20),
                "hub": _log_int(rng, 50_000, 4_000_000)}
    return {"family": f, "n": _log_int(rng, 100_000, 10_000_000)}


# ----------------------------------------------------------------- inputs --

def _gen(seed):
    g = torch.Generator(device="cuda")
    g.manual_seed(1_111_062_700 + int(seed))
    return g


def _ints(g, lo, hi, size):
    """Uniform integers in [lo, hi], int32."""
    return torch.randint(lo, hi + 1, (size,), generator=g, device="cuda", dtype=torch.int32)


def _row_ptr(deg):
    rp = torch.zeros(deg.numel() + 1, dtype=torch.int64, device="cuda")
    torch.cumsum(deg, 0, out=rp[1:])
    assert int(rp[-1]) <= INT32_MAX
    return rp


def _spread(g, n, k):
    """Uniform in [0, k), every value equally often (so that a size has one
    edge count), in random order."""
    return torch.randperm(n, generator=g, device="cuda") % k


def _ring(g, n, xhi, wlo, whi):
    rp = _row_ptr(1 + _spread(g, n, xhi + 1))
    m = int(rp[-1])
    col = _ints(g, 0, n - 1, m)
    col[rp[:-1]] = (torch.arange(1, n + 1, device="cuda") % n).to(torch.int32)
    return rp.to(torch.int32), col, _ints(g, wlo, whi, m)


def _locality(g, n):
    u = _spread(g, n, 30)
    deg = torch.where(u == 0, 64, torch.where(u <= 5, 16, 4))
    del u
    rp = _row_ptr(deg)
    m = int(rp[-1])
    col = torch.randn(m, generator=g, device="cuda").mul_(4096.0).abs_().floor_().to(torch.int32)
    col[rp[:-1]] = 0
    src = torch.repeat_interleave(torch.arange(1, n + 1, device="cuda", dtype=torch.int32), deg,
                                  output_size=m)
    col += src
    del src, deg
    col.remainder_(n)   # (i + 1 + offset stays far below 2^31)
    return rp.to(torch.int32), col, _ints(g, -1000, 1000, m)


def _product(g, P, S):
    """Interleaving product of P processes, each a ring of S states with two
    chords a state (a chord to the state itself, to its ring successor or equal
    to the other chord is dropped)."""
    C, N = 2, S**P
    s = torch.arange(S, device="cuda")
    ring = (s + 1) % S
    code = torch.arange(N, device="cuda")
    moves = []
    for p in range(P):
        ch = torch.randint(0, S, (C, S), generator=g, device="cuda")
        for k in range(C):
            drop = (ch[k] == s) | (ch[k] == ring)
            for j in range(k):
                drop |= ch[k] == ch[j]
            ch[k][drop] = -1
        unit = S**p
        mine = (code // unit) % S
        for local in (ring, ch[0], ch[1]):
            to = local[mine]
            moves.append(torch.where(to < 0, -1, code + (to - mine) * unit))
    adj = torch.stack(moves, 1)     # [N, 3 P] targets by code, -1: none
    # breadth-first numbering from the all-zero state, in the order of discovery
    ident = torch.full((N,), -1, dtype=torch.int64, device="cuda")
    first = torch.empty(N, dtype=torch.int64, device="cuda")
    front = torch.zeros(1, dtype=torch.int64, device="cuda")
    ident[0] = 0
    order, found = [front], 1
    while front.numel():
        t = adj[front].reshape(-1)
        t = t[t >= 0]
        t = t[ident[t] < 0]
        pos = torch.arange(t.numel(), device="cuda")
        first[t] = t.numel()
        first.scatter_reduce_(0, t, pos, "amin")
        front = t[first[t] == pos]
        ident[front] = found + torch.arange(front.numel(), device="cuda")
        found += front.numel()
        order.append(front)
    order = torch.cat(order)
    rows = adj[order]
    keep = rows >= 0
    rp = _row_ptr(keep.sum(1))
    col = ident[rows[keep]].to(torch.int32)
    return rp.to(torch.int32), col, _ints(g, 0, 1000, col.numel())


def _batch(g, G, nmax):
    u = (torch.randperm(G, generator=g, device="cuda").double() + 0.5) / G
    sizes = (100.0 * torch.exp(u * math.log(nmax / 100.0))).floor().to(torch.int64)
    vp = _row_ptr(sizes)
    N = int(vp[-1])
    gid = torch.repeat_interleave(torch.arange(G, device="cuda"), sizes, output_size=N)
    deg = 1 + _spread(g, N, 8)
    rp = _row_ptr(deg)
    m = int(rp[-1])
    # (an edge's graph from its source; targets uniform in the graph)
    first = torch.repeat_interleave(vp[gid].to(torch.int32), deg, output_size=m)
    size = torch.repeat_interleave(sizes[gid].to(torch.int32), deg, output_size=m)
    col = (torch.rand(m, generator=g, device="cuda", dtype=torch.float64) * size).to(torch.int32)
    col += first
    del first, size
    v = torch.arange(N, device="cuda")
    nxt = v + 1
    col[rp[:-1]] = torch.where(nxt == vp[gid + 1], vp[gid], nxt).to(torch.int32)
    return vp.to(torch.int32), rp.to(torch.int32), col, _ints(g, 1, 10_000, m)


def _hub(g, n, hub_deg):
    deg = torch.full((n,), 4, dtype=torch.int64, device="cuda")
    deg[int(torch.randint(0, n, (1,), generator=g, device="cuda"))] += hub_deg
    rp = _row_ptr(deg)
    m = int(rp[-1])
    col = _ints(g, 0, n - 1, m)
    col[rp[:-1]] = (torch.arange(1, n + 1, device="cuda") % n).to(torch.int32)
    return rp.to(torch.int32), col, _ints(g, -1000, 1000, m)


def _digraph(g, n):
    deg = torch.poisson(torch.full((n,), 1.5, device="cuda"), generator=g).to(torch.int64)
    deg[torch.rand(n, generator=g, device="cuda") < 0.05] = 0
    rp = _row_ptr(deg)
    m = int(rp[-1])
    return rp.to(torch.int32), _ints(g, 0, n - 1, m), _ints(g, -50, 50, m)


def prepare(case, seed):
    g, f = _gen(seed), case["family"]
    s = {"family": f}
    if f == "ring":
        s["graph"] = _ring(g, case["n"], 4, 1, 100)
    elif f in ("product", "single"):
        s["graph"] = _product(g, case["P"], case["S"])
    elif f == "locality":
        s["graph"] = _locality(g, case["n"])
    elif f == "resolve":
        rp, col, w = _locality(g, case["n"])
        s["workspace"] = ocm.make_workspace(rp.numel() - 1, col.numel())
        before = ocm.solve(rp, col, w, "min", workspace=s["workspace"], certificate=True)
        s["policy"] = before.policy
        moved = torch.randint(0, 64, (w.numel(),), generator=g, device="cuda") == 0
        w = torch.where(moved, _ints(g, -1000, 1000, w.numel()), w)
        s["graph"] = (rp, col, w)
    elif f == "diff":
        # (weights wide enough for one optimal cycle, where the gradient is one)
        rp, col, w = _ring(g, case["n"], 7, 0, 1_000_000)
        s["graph"] = (rp, col, w)
        s["w_float"] = w.to(torch.float32).requires_grad_(True)
    elif f == "ratio":
        rp, col, w = _ring(g, case["n"], 7, -100_000, 100_000)
        s["graph"] = (rp, col, w)
        s["transit"] = _ints(g, 1, 8, col.numel())
        s["grad"] = torch.ones(1, device="cuda")
    elif f == "batch":
        s["batch"] = _batch(g, case["G"], case["nmax"])
        s["grad"] = torch.ones(case["G"], device="cuda")
    elif f == "hub":
        s["graph"] = _hub(g, case["n"], case["hub"])
    elif f == "scc":
        s["graph"] = _digraph(g, case["n"])
    if f in ("product", "locality"):   # a program that solves large graphs keeps its scratch
        rp, col, _ = s["graph"]
        s["workspace"] = ocm.make_workspace(rp.numel() - 1, col.numel())
    if f == "scc":     # each component's optimum, kept at the component's smallest vertex
        n = case["n"]
        s["num"] = torch.zeros(n, dtype=torch.int64, device="cuda")
        s["den"], s["len"] = (torch.zeros(n, dtype=torch.int32, device="cuda") for _ in range(2))
    elif f not in ("diff", "batch"):
        s["cycle"] = torch.full((s["graph"][0].numel() - 1,), -1, dtype=torch.int32,
                                device="cuda")
    return s


# -------------------------------------------------------------------- run --

def run(s):
    f = s["family"]
    if f == "batch":
        vp, rp, col, w = s["batch"]
        sol = ocm.solve_batch(vp, rp, col, w, "max")
        return [sol.num, sol.den, sol.cycle_len, ocm.backward_batch(sol, s["grad"], col.numel())]
    rp, col, w = s["graph"]
    if f == "diff":
        lam = ocm.OCMFunction.apply(s["w_float"], rp, col, w, "max", None)
        (grad,) = torch.autograd.grad(lam, s["w_float"])
        return [lam, grad]
    if f == "scc":
        sol = ocm.solve_scc(rp, col, w, "min")
        root = sol.root.long()
        s["num"][root], s["den"][root], s["len"][root] = sol.num, sol.den, sol.cycle_len
        return [sol.labels, s["num"], s["den"], s["len"]]
    cycle = s["cycle"]
    if f in ("ring", "hub"):
        sol = ocm.solve(rp, col, w, "max", cycle_out=cycle)
    elif f == "product":
        sol = ocm.solve(rp, col, w, "max", cycle_out=cycle, workspace=s["workspace"])
    elif f == "locality":
        sol = ocm.solve(rp, col, w, "min", cycle_out=cycle, workspace=s["workspace"])
    elif f == "single":
        sol = ocm.solve(rp, col, w, "max", cycle_out=cycle, single_lambda=True)
    elif f == "resolve":
        sol = ocm.solve(rp, col, w, "min", cycle_out=cycle, workspace=s["workspace"],
                        certificate=True, init_policy=s["policy"])
        return [sol.num, sol.den, cycle, sol.eta_num, sol.eta_den, sol.potential, sol.policy]
    else:
        sol = ocm.solve(rp, col, w, "min", cycle_out=cycle, transit=s["transit"])
        grad = ocm.backward(sol.cycle, s["grad"], col.numel(), transit=s["transit"])
        return [sol.num, sol.den, cycle, grad]
    return [sol.num, sol.den, cycle]


def work(case):
    """The CSR read once and the outputs written once; one multiply-add an
    edge (a policy that is optimal from the start needs no more)."""
    f = case["family"]
    extra = 0.0
    if f in ("product", "single"):
        n = float(case["S"] ** case["P"])
        # three moves a process, less the chords that are dropped
        S = case["S"]
        m = n * case["P"] * (1 + (1 - 2 / S) + (1 - 2 / S) ** 2)
    elif f == "batch":
        lg = math.log(case["nmax"] / 100.0)
        n = case["G"] * (case["nmax"] - 100.0) / lg
        m = 4.5 * n
        extra = 4 * m + 24 * case["G"]          # the gradient; offsets in, results out
    else:
        n = float(case["n"])
        m = n * {"ring": 3.0, "locality": 8.0, "resolve": 8.0, "diff": 4.5, "ratio": 4.5,
                 "hub": 4.0, "scc": 1.5 * 0.95}[f]
        if f == "hub":
            m += case["hub"]
        if f == "resolve":
            extra = 4 * n + 24 * n              # the start policy; the certificate
        if f == "diff":
            extra = 4 * m
        if f == "ratio":
            extra = 8 * m                       # transit times; the gradient
        if f == "scc":
            extra = 4 * n                       # the labels
    return {"bytes": 4 * (n + 1) + 8 * m + extra, "flops": 2 * m}


# ------------------------------------------------------------------ exact --

def _howard(rp, col, w, gid, G, t=None):
    """Howard's policy iteration in plain torch, 64-bit integers: maximum cycle
    mean (or ratio w/t) of each of G graphs given as one union.  Returns per
    graph the numerator and denominator, and the optimal cycles' edge mask."""
    n, m = rp.numel() - 1, col.numel()
    rp, col, w = rp.long(), col.long(), w.long()
    t = torch.ones_like(w) if t is None else t.long()
    src = torch.repeat_interleave(torch.arange(n, device=w.device), rp[1:] - rp[:-1],
                                  output_size=m)
    eid = torch.arange(m, device=w.device)
    low = torch.iinfo(torch.int64).min

    def best_edge(keys):
        on = torch.ones(m, dtype=torch.bool, device=w.device)
        for k in keys:
            top = torch.full((n,), low, device=w.device).scatter_reduce(
                0, src[on], k[on], "amax")
            on &= k == top[src]
        return torch.full((n,), m, device=w.device).scatter_reduce(0, src[on], eid[on], "amin")

    pi = best_edge([w])
    rounds = max(1, n.bit_length())
    while True:
        succ = col[pi]
        # the smallest vertex of the cycle that each vertex reaches
        J, M = succ, torch.arange(n, device=w.device)
        for _ in range(rounds):
            M, J = torch.minimum(M, M[J]), J[J]
        root = J                       # on the cycle by now
        M, J = torch.arange(n, device=w.device), succ
        for _ in range(rounds):
            M, J = torch.minimum(M, M[J]), J[J]
        root = M[root]                 # smallest vertex ahead of a cycle vertex
        # path weight and time to it
        term = root == torch.arange(n, device=w.device)
        J = torch.where(term, torch.arange(n, device=w.device), succ)
        S, T, L = (torch.where(term, 0, x) for x in (w[pi], t[pi], torch.ones_like(pi)))
        for _ in range(rounds):
            S, T, L, J = S + S[J], T + T[J], L + L[J], J[J]
        r = torch.nonzero(term).reshape(-1)
        W, Q = w[pi[r]] + S[succ[r]], t[pi[r]] + T[succ[r]]
        d = torch.gcd(W, Q).clamp_(min=1)
        p, q = W // d, Q // d
        whole = torch.div(p, q, rounding_mode="floor")
        # fractions of short cycles differ by far more than 2^-52
        frac = (p - whole * q).double() / q.double()
        _, a = torch.unique(whole, return_inverse=True)
        _, b = torch.unique(frac, return_inverse=True)
        _, rank = torch.unique(a * (b.max() + 1) + b, return_inverse=True)
        at = torch.empty(n, dtype=torch.int64, device=w.device)
        at[r] = torch.arange(r.numel(), device=w.device)
        mine = at[root]
        P, Qv, R = p[mine], q[mine], rank[mine]
        V = Qv * S - P * T
        rk, key = R[col], Qv[col] * w - P[col] * t + V[col]
        e = best_edge([rk, key])
        better = (rk[e] > rk[pi]) | ((rk[e] == rk[pi]) & (key[e] > key[pi]))
        if not bool(better.any()):
            break
        pi = torch.where(better, e, pi)
    # per graph the best cycle, ties to the smallest root
    gr = gid[r]
    top = torch.full((G,), -1, device=w.device).scatter_reduce(0, gr, rank, "amax")
    on = rank == top[gr]
    first = torch.full((G,), n, device=w.device).scatter_reduce(0, gr[on], r[on], "amin")
    k = at[first]
    mask = torch.zeros(m, dtype=torch.bool, device=w.device)
    v = first.clone()
    while True:
        mask[pi[v]] = True
        v = succ[v]
        going = v != first[gid[v]]
        if not bool(going.any()):
            break
        v = v[going]
    return p[k], q[k], mask, t


def exact(case, seed):
    f = case["family"]
    if f not in ("diff", "ratio", "batch"):
        return None    # whole numbers only
    s = prepare(case, seed)
    if f == "batch":
        vp, rp, col, w = s["batch"]
        if col.numel() > 150_000_000:
            return None
        G, n = case["G"], rp.numel() - 1
        vp = vp.long()
        gid = torch.repeat_interleave(torch.arange(G, device="cuda"), vp[1:] - vp[:-1],
                                      output_size=n)
        _, _, mask, _ = _howard(rp, col, w, gid, G)
        e = torch.nonzero(mask).reshape(-1)
        eg = gid[torch.searchsorted(rp.long(), e, right=True) - 1]
        length = torch.bincount(eg, minlength=G)
        grad = torch.zeros(col.numel(), dtype=torch.float64, device="cuda")
        grad[e] = 1.0 / length[eg].double()
        return [None, None, None, grad]
    rp, col, w = s["graph"]
    gid = torch.zeros(rp.numel() - 1, dtype=torch.int64, device="cuda")
    sign = -1 if f == "ratio" else 1
    p, q, mask, t = _howard(rp, col, sign * w, gid, 1, s.get("transit"))
    grad = mask.double() / t[mask].sum().double()
    if f == "ratio":
        return [None, None, None, grad]
    return [p[0].double() / q[0].double(), grad]
