"""The work that users of this framework have it do, as measurable cases.

A case is a dict of plain values: which call is made (`call`), the graph it is made on (`graph`,
`n`, `m`, `gamma`, `weighted`) and the call's options.  `prepare` makes what a program has in hand
before the call, on the GPU and from the seed alone; `run` makes the call through the binding's
public entry points; `exact` is the same in float64 with plain torch operations.

Calls:
  run       erc_run: the whole path on a device-resident edge list
  run_host  erc_run_host: the same from and to pinned host memory, copies included
  cg, pcg   erc_batched_cg / erc_batched_pcg on one batch of projected right-hand sides
  build     erc_build_laplacian on a shuffled edge list with some repeated pairs
  rhs       erc_jl_rhs: one batch of right-hand sides
  finish    what follows a batch's solve: edge distances, curvature, sampling probabilities
  sample    erc_sample_subgraph and erc_saint_counts: one training subgraph and its counts
The outputs are what a call computes: solutions, resistances, curvature, probabilities, graphs.
`relres` (the float32 rounding that is left of a solution near its attainable accuracy) and the
iteration counts of the long solves (where the residual crosses the threshold at rounding level)
are the stop test's diagnostics and are left out; the short solves return their counts.
"""
import math

import torch

from paper_2609_27209_gb300 import erc

EPS = 1e-3
SEED_Q = 0xE2C1  # Philox key of the projection, as in the repository's workloads
DEV = "cuda"
L2_BYTES = 126 << 20


def listed():
    return [
        # the smallest whole run: a 2,000-node sanity graph, K = 64 in one batch; launches,
        # synchronisations and the single-launch solver's latency
        dict(name="run_ring_2k", call="run", graph="ring", n=2000, m=10000, gamma=0.0,
             weighted=False, K=64, kc=64, tol=1e-6, iterations=20),
        # an ordinary community graph with weights, K = 128 in one batch
        dict(name="run_sbm_20k", call="run", graph="sbm", n=20000, m=104945, gamma=0.0,
             weighted=True, K=128, kc=128, tol=1e-6, iterations=42),
        # a program that keeps its edge list on the host, odd sizes: 100 columns in ragged
        # batches of 36, with the optional preconditioner
        dict(name="run_host_60k_ragged", call="run_host", graph="power_law", n=60013, m=411007,
             gamma=2.6, weighted=True, K=100, kc=36, tol=1e-6, precond=1, iterations=20),
        # one wide batch on a citation-network-sized power-law graph, unit weights
        dict(name="cg_169k", call="cg", graph="power_law", n=169343, m=1339252, gamma=2.5,
             weighted=False, K=256, kc=256, tol=1e-6, iterations=286),
        # a dense power-law graph (mean degree 492) streamed in narrow batches
        dict(name="cg_dense_233k", call="cg", graph="power_law", n=232965, m=57500000, gamma=2.1,
             weighted=False, K=128, kc=32, tol=1e-5, iterations=64),
        # the largest graph, plain CG, a narrow batch
        dict(name="cg_2449k", call="cg", graph="power_law", n=2449029, m=64348144, gamma=2.3,
             weighted=True, K=1024, kc=32, tol=1e-5, iterations=353),
        # the largest graph, preconditioned, the full batch width
        dict(name="pcg_2449k", call="pcg", graph="power_law", n=2449029, m=64348144, gamma=2.3,
             weighted=True, K=1024, kc=128, tol=1e-5, iterations=7),
        # the largest graph's Laplacian from its edge list
        dict(name="build_2449k", call="build", graph="power_law", n=2449029, m=64348144,
             gamma=2.3, weighted=True, repeats=0.02),
        # the largest graph: one batch of right-hand sides in the middle of the projection
        dict(name="rhs_2449k", call="rhs", graph="power_law", n=2449029, m=64348144, gamma=2.3,
             weighted=True, K=1024, kc=128, c0=256),
        # the largest graph: a batch's edge distances, then curvature and probabilities
        dict(name="finish_2449k", call="finish", graph="power_law", n=2449029, m=64348144,
             gamma=2.3, weighted=True, K=1024, kc=128),
        # one training step's subgraph by nodes on the citation-network-sized graph
        dict(name="sample_nodes_169k", call="sample", graph="power_law", n=169343, m=1339252,
             gamma=2.5, weighted=False, kind=0, budget=16934, induced=True),
        # one subgraph by edges on the largest graph
        dict(name="sample_edges_2449k", call="sample", graph="power_law", n=2449029, m=64348144,
             gamma=2.3, weighted=True, kind=1, budget=6434814, induced=True),
    ]


def _log(rng, lo, hi):
    return int(round(math.exp(rng.uniform(math.log(lo), math.log(hi)))))


def draw(rng):
    """One more case: sizes from 2 thousand to 2.4 million nodes, mean degrees from 6 to 400."""
    call = rng.choice(["run", "run", "run_host", "cg", "cg", "pcg", "build", "rhs", "finish",
                       "sample"])
    n = _log(rng, 2000, 2400000) | 1
    m = min(n * _log(rng, 3, 200), 60000000)
    m = max(2 * n, min(m, n * (n - 1) // 40))
    graph = rng.choice(["power_law", "power_law", "power_law", "sbm"])
    if graph == "sbm":
        n = n // 10 * 10
        m = min(m, 20 * n)
    case = dict(call=call, graph=graph, n=n, m=m, gamma=round(rng.uniform(2.1, 2.9), 3),
                weighted=rng.random() < 0.5)
    if call in ("run", "run_host", "cg", "pcg", "rhs", "finish"):
        cap = 4e8 if call in ("run", "run_host", "cg") else 8e9  # edges x columns
        top = max(4, min(256, int(cap / m)))
        kc = rng.choice([4, 7, 16, 30, 32, 50, 64, 100, 128, 200, 256])
        kc = min(kc, top)
        batches = rng.choice([1, 1, 2, 3]) if call in ("run", "run_host") else 1
        batches = max(1, min(batches, int(cap / (m * kc))))
        if batches > 1:
            kc = max(4, kc // 4 * 4)
        case.update(K=kc * batches - (rng.randrange(4) if batches > 1 else 0), kc=kc)
        if call in ("cg", "pcg", "rhs", "finish"):
            case["K"] = max(case["K"], rng.choice([64, 128, 256, 1024]))
    if call in ("run", "run_host", "cg", "pcg"):
        case.update(tol=rng.choice([1e-6, 1e-5]))
        case.update(precond=int(call == "pcg" or (call != "cg" and rng.random() < 0.5)))
        case.update(iterations=20 if case["precond"] else 150)
    if call == "rhs":
        case.update(c0=4 * rng.randrange((case["K"] - case["kc"]) // 4 + 1))
    if call == "build":
        case.update(repeats=rng.choice([0.0, 0.02, 0.2]))
    if call == "sample":
        kind = rng.randrange(2)
        case.update(kind=kind, budget=max(1, (m if kind else n) // _log(rng, 5, 200)),
                    induced=rng.random() < 0.7)
    return case


# ------------------------------------------------------------------------------------ inputs
def _sorted_unique(keys):
    keys = torch.sort(keys).values
    keep = torch.ones_like(keys, dtype=torch.bool)
    keep[1:] = keys[1:] != keys[:-1]
    return keys[keep]


def _pair_keys(u, v, n):
    return torch.minimum(u, v) * n + torch.maximum(u, v)


def _power_law_cdf(n, gamma, mean_deg):
    """Expected degrees ~ (i + 1)^(-1 / (gamma - 1)), capped at the square root of their sum."""
    base = torch.arange(1, n + 1, dtype=torch.float64, device=DEV) ** (-1.0 / (gamma - 1.0))
    s = mean_deg / base.mean()
    for _ in range(40):
        w = (s * base).clamp(max=math.sqrt(mean_deg * n))
        s = s * (mean_deg / w.mean())
    return w.cpu().cumsum(0).to(DEV)  # summed on the host: the same on every run


def _edges(case, seed):
    """The case's edge list: int64 endpoints in a shuffled order and orientation, m distinct pairs
    (a ring over all nodes and m - n others), and float32 weights or None."""
    n, m = case["n"], case["m"]
    gen = torch.Generator(DEV).manual_seed(seed)
    i = torch.arange(n, device=DEV)
    ring = _pair_keys(i, (i + 1) % n, n)
    cdf = _power_law_cdf(n, case["gamma"], 2.0 * m / n) if case["graph"] == "power_law" else None

    def ids(k):
        if cdf is None:
            return torch.randint(0, n, (k,), device=DEV, generator=gen)
        r = torch.rand(k, dtype=torch.float64, device=DEV, generator=gen) * cdf[-1]
        return torch.searchsorted(cdf, r).clamp_(max=n - 1)

    need = m - n
    keys = torch.empty(0, dtype=torch.int64, device=DEV)
    while keys.numel() < need:
        k = int((need - keys.numel()) * 1.12) + 64
        u = ids(k)
        v = ids(k)
        if case["graph"] == "sbm":  # ten contiguous blocks, 16 of 17 edges inside one
            size = n // 10
            inside = torch.rand(k, device=DEV, generator=gen) < 16.0 / 17.0
            v = torch.where(inside, u // size * size + v % size, v)
        gap = (u - v).abs()
        ok = (gap > 1) & (gap < n - 1)  # neither a loop nor a ring pair
        keys = _sorted_unique(torch.cat([keys, _pair_keys(u[ok], v[ok], n)]))
        del u, v, gap, ok
    order = torch.randperm(keys.numel(), device=DEV, generator=gen)
    keys = torch.cat([keys[order[:need]], ring])
    del order
    keys = keys[torch.randperm(keys.numel(), device=DEV, generator=gen)]
    a, b = keys // n, keys % n
    del keys
    if case.get("repeats"):  # some pairs given twice
        k = int(a.numel() * case["repeats"])
        a, b = torch.cat([a, a[:k]]), torch.cat([b, b[:k]])
    flip = torch.rand(a.numel(), device=DEV, generator=gen) < 0.5
    src, dst = torch.where(flip, b, a), torch.where(flip, a, b)
    w = None
    if case["weighted"]:
        if case["graph"] == "sbm":
            w = torch.empty(a.numel(), device=DEV).log_normal_(0.0, 0.5, generator=gen)
        else:
            w = torch.empty(a.numel(), device=DEV).uniform_(0.5, 2.0, generator=gen)
    return src, dst, w, gen


def _graph(case, seed):
    src, dst, w, gen = _edges(case, seed)
    return erc.erc_build_laplacian(case["n"], src.int(), dst.int(), w), gen


def _params(case):
    return erc.Params(K=case["K"], kc=case["kc"], eps=EPS, tol=case["tol"], seed=SEED_Q,
                      precond=case.get("precond", 0))


def _solution_like(case, deg, gen):
    """A block with the spread that solutions have: a row's size falls with its degree."""
    n, kc = case["n"], case["kc"]
    X = torch.zeros(n, (kc + 3) // 4 * 4, device=DEV)
    X[:, :kc] = torch.randn(n, kc, device=DEV, generator=gen)
    return X.mul_((1.0 / (case["K"] * (deg + EPS))).sqrt()[:, None])


def _degree_probabilities(case, g, kind):
    """Eq. 7 / Eq. 8 of the curvature that R_uv ~ 1/d_u + 1/d_v gives, in float64."""
    inv = 1.0 / (g.deg.double() + EPS)
    eu, ev = g.eu.long(), g.ev.long()
    R = inv[eu] + inv[ev]
    eid = g.csr_eid.long()
    rows = dict(reduce="sum", offsets=g.row_ptr, unsafe=True)
    w = g.val.double()
    p = 1.0 - 0.5 * torch.segment_reduce(w * R[eid], **rows)
    kappa = 2.0 * (p[eu] + p[ev]) / R
    if kind:
        q = (2.0 * kappa.max() - kappa).clamp(min=0.0).sqrt() + 1.0
    else:
        q = torch.segment_reduce((kappa - kappa.min())[eid], **rows)
    return (q / q.sum()).float()


def prepare(case, seed):
    call = case["call"]
    if call in ("run", "run_host"):
        src, dst, w, _ = _edges(case, seed)
        src, dst, prm = src.int(), dst.int(), _params(case)
        if call == "run":
            return dict(case=case, src=src, dst=dst, w=w, prm=prm,
                        ws=erc.erc_run_workspace(case["n"], src.numel(), prm))
        host = [None if t is None else t.cpu().pin_memory() for t in (src, dst, w)]
        sizes = dict(eu="m", ev="m", R="m", p="n", kappa="m", prob_node="n", prob_edge="m",
                     iters="K", relres="K")
        out = {k: torch.empty(case[s], pin_memory=True,
                              dtype=torch.int32 if k in ("eu", "ev", "iters") else torch.float32)
               for k, s in sizes.items()}
        return dict(case=case, src=host[0], dst=host[1], w=host[2], prm=prm, out=out,
                    ws=erc.erc_run_host_workspace(case["n"], src.numel(), prm))
    if call == "build":
        src, dst, w, _ = _edges(case, seed)
        return dict(case=case, src=src.int(), dst=dst.int(), w=w)
    g, gen = _graph(case, seed)
    if call in ("cg", "pcg"):
        Y = erc.erc_jl_rhs(g, SEED_Q, case["K"], 0, case["kc"])
        ws = torch.empty(erc.lib().erc_batched_cg_workspace_size(case["n"], Y.shape[1]),
                         dtype=torch.uint8, device=DEV)
        return dict(case=case, g=g, Y=Y, X=torch.empty_like(Y), ws=ws)
    if call == "rhs":
        return dict(case=case, g=g)
    if call == "finish":
        return dict(case=case, g=g, X=_solution_like(case, g.deg, gen))
    if call == "sample":
        return dict(case=case, g=g, prob=_degree_probabilities(case, g, case["kind"]),
                    seed=seed + 17)
    raise ValueError(call)


# --------------------------------------------------------------------------------------- run
def run(state):
    case = state["case"]
    call = case["call"]
    if call in ("run", "run_host"):
        f = erc.erc_run if call == "run" else erc.erc_run_host
        o = f(case["n"], state["src"], state["dst"], state["w"], state["prm"], ws=state["ws"],
              out=state.get("out"))
        out = {k: o[k] for k in ("m", "status", "eu", "ev", "R", "p", "kappa", "prob_node",
                                 "prob_edge")}
        if case["iterations"] <= 50:
            out["iters"] = o["iters"]
        return out
    if call in ("cg", "pcg"):
        f = erc.erc_batched_cg if call == "cg" else erc.erc_batched_pcg
        X, iters, _, status = f(state["g"], EPS, state["Y"], case["kc"], case["tol"],
                                X=state["X"], ws=state["ws"])
        return dict(X=X, status=status, **({"iters": iters} if call == "pcg" else {}))
    if call == "build":
        g = erc.erc_build_laplacian(case["n"], state["src"], state["dst"], state["w"])
        return dict(m=g.m, unit=int(g.unit_weights), row_ptr=g.row_ptr, col=g.col, val=g.val,
                    deg=g.deg, csr_eid=g.csr_eid, eu=g.eu, ev=g.ev, ew=g.ew)
    if call == "rhs":
        return dict(Y=erc.erc_jl_rhs(state["g"], SEED_Q, case["K"], case["c0"], case["kc"]))
    if call == "finish":
        R = torch.zeros(state["g"].m, device=DEV)
        erc.erc_edge_resistance(state["g"], state["X"], case["kc"], R)
        p, kappa = erc.erc_curvature(state["g"], R)
        prob_node, prob_edge = erc.erc_sampling_probs(state["g"], kappa)
        return dict(R=R, p=p, kappa=kappa, prob_node=prob_node, prob_edge=prob_edge)
    nodes, edges = erc.erc_sample_subgraph(state["g"], case["kind"], state["prob"],
                                           case["budget"], state["seed"],
                                           induced=case["induced"])
    g = state["g"]
    node_count = torch.zeros(g.n, dtype=torch.int32, device=DEV)
    edge_count = torch.zeros(g.m, dtype=torch.int32, device=DEV)
    erc.erc_saint_counts(g, nodes, edges, node_count, edge_count)
    return dict(n_sub=nodes.numel(), m_sub=edges.numel(), node_count=node_count,
                edge_count=edge_count)


# -------------------------------------------------------------------------------------- work
def _build_bytes(n, m, weighted):
    edge_in = 12 if weighted else 8
    return edge_in * m + 12 * n + 2 * m * 12 + 12 * m  # CSR with weights, edge list with weights


def _solve_work(n, m, weighted, kc, iterations):
    csr = (8 if weighted else 4) * 2 * m + 8 * n
    once = csr + 8 * n * kc
    flops = iterations * (6.0 * m * kc + 12.0 * n * kc)
    if csr + 20 * n * kc <= L2_BYTES:  # the solve's state stays on the chip
        return once, flops
    # an iteration reads the matrix, p, r, Ap, x and writes Ap, r, x, p at least once
    return once + iterations * (csr + 36 * n * kc), flops


def work(case):
    """What a pass cannot do without (solves: at the iteration counts of `iterations`)."""
    n, m, call, wt = case["n"], case["m"], case["call"], case["weighted"]
    tail = 12 * m + 12 * n + 8 * m + 8 * 2 * m
    if call in ("run", "run_host"):
        K = case["K"]
        by, fl = _build_bytes(n, m, wt), 0.0
        for c0 in range(0, K, case["kc"]):
            k = min(case["kc"], K - c0)
            b, f = _solve_work(n, m, wt, k, case["iterations"])
            by, fl = by + b, fl + f + 2.0 * 2 * m * k + 3.0 * m * k
        return dict(bytes=by + tail, flops=fl + 10.0 * m)
    if call in ("cg", "pcg"):
        by, fl = _solve_work(n, m, wt, case["kc"], case["iterations"])
        return dict(bytes=by, flops=fl)
    if call == "build":
        return dict(bytes=_build_bytes(n, m * (1 + case["repeats"]), wt), flops=0.0)
    if call == "rhs":
        return dict(bytes=2 * m * (12 if wt else 8) + 8 * n + 4 * n * case["kc"],
                    flops=2.0 * 2 * m * case["kc"])
    if call == "finish":
        return dict(bytes=4 * n * case["kc"] + 12 * m + tail, flops=3.0 * m * case["kc"] + 10.0 * m)
    count = m if case["kind"] else n
    return dict(bytes=4 * count + 8 * m + 4 * (m + n) + 8 * case["budget"], flops=float(count))


# ------------------------------------------------------------------------ float64 restatement
class _Graph64:
    """CSR, edge list and degrees of an edge list, in float64 with torch operations."""

    def __init__(self, case, seed):
        n = case["n"]
        src, dst, w, self.gen = _edges(case, seed)
        key = torch.minimum(src, dst) * n + torch.maximum(src, dst)
        w = torch.ones(key.numel(), dtype=torch.float64, device=DEV) if w is None else w.double()
        key, order = torch.sort(key, stable=True)
        keep = torch.ones_like(key, dtype=torch.bool)
        keep[1:] = key[1:] != key[:-1]
        at = torch.cumsum(keep, 0) - 1
        key = key[keep]
        self.n, self.m = n, key.numel()
        self.ew = torch.zeros(self.m, dtype=torch.float64, device=DEV).index_add_(0, at, w[order])
        self.eu, self.ev = key // n, key % n
        del src, dst, key, order, keep, at, w
        both, order = torch.sort(torch.cat([self.eu * n + self.ev, self.ev * n + self.eu]))
        row, self.col = both // n, both % n
        self.eid = order % self.m
        del both, order
        self.val = self.ew[self.eid]
        self.row_ptr = torch.zeros(n + 1, dtype=torch.int64, device=DEV)
        self.row_ptr[1:] = torch.cumsum(torch.bincount(row, minlength=n), 0)
        self.deg = torch.zeros(n, dtype=torch.float64, device=DEV).index_add_(0, row, self.val)
        self.row = row

    def csr(self, val, cols, width):
        return torch.sparse_csr_tensor(self.row_ptr, cols, val, (self.n, width),
                                       check_invariants=False)


def _philox(e, block, seed):
    """The four 32-bit words of Philox4x32-10 at counter (block, 0, e, 0), as int64 columns."""
    lo = 0xFFFFFFFF
    x = [torch.full_like(e, block), torch.zeros_like(e), e & lo, e >> 32]
    k0, k1 = seed & lo, seed >> 32
    for _ in range(10):
        a, b = x[0] * 0xD2511F53, x[2] * 0xCD9E8D57
        x = [((b >> 32) & lo) ^ x[1] ^ k0, b & lo, ((a >> 32) & lo) ^ x[3] ^ k1, a & lo]
        k0, k1 = (k0 + 0x9E3779B9) & lo, (k1 + 0xBB67AE85) & lo
    return x


def _rhs64(g, K, c0, kc):
    """B^T W^(1/2) Q, sixteen columns at a time."""
    Y = torch.empty(g.n, kc, dtype=torch.float64, device=DEV)
    side = torch.where(g.col > g.row, 1.0, -1.0).double()
    B = g.csr(side * g.val.sqrt() / math.sqrt(K), g.eid, g.m)
    e = torch.arange(g.m, device=DEV)
    block, words = -1, None
    for c in range(0, kc, 16):
        cols = []
        for j in range(c0 + c, c0 + min(c + 16, kc)):
            if j >> 7 != block:
                block = j >> 7
                words = _philox(e, block, SEED_Q)
            cols.append((1 - 2 * ((words[(j >> 5) & 3] >> (j & 31)) & 1)).double())
        Y[:, c:c + len(cols)] = torch.sparse.mm(B, torch.stack(cols, 1))
    return Y


def _solve64(g, Y):
    """(L + eps I)^-1 Y: Jacobi-preconditioned CG, each column to a relative residual of 1e-12."""
    A = g.csr(g.val, g.col, g.n)
    d = (g.deg + EPS)[:, None]
    X, R = torch.zeros_like(Y), Y.clone()
    P = R / d
    rz, stop = (R * P).sum(0), 1e-24 * Y.square().sum(0)
    for _ in range(2000):
        AP = d * P - torch.sparse.mm(A, P)
        live = R.square().sum(0) > stop
        if not bool(live.any()):
            break
        al = torch.where(live, rz / (P * AP).sum(0), torch.zeros_like(rz))
        X += al * P
        R -= al * AP
        new = (R * R / d).sum(0)
        P = R / d + torch.where(live, new / rz, torch.zeros_like(rz)) * P
        rz = torch.where(live, new, rz)
    return X


def _resistance64(g, X):
    R = torch.zeros(g.m, dtype=torch.float64, device=DEV)
    for c in range(0, X.shape[1], 8):
        x = X[:, c:c + 8].contiguous()
        for e in range(0, g.m, 1 << 24):
            s = slice(e, e + (1 << 24))
            R[s] += (x[g.eu[s]] - x[g.ev[s]]).square().sum(1)
    return R


def _tail64(g, R):
    rows = lambda v: torch.zeros(g.n, dtype=torch.float64, device=DEV).index_add_(0, g.row, v)
    p = 1.0 - 0.5 * rows(g.val * R[g.eid])
    kappa = 2.0 * (p[g.eu] + p[g.ev]) / R
    lo, hi = kappa.min(), kappa.max()
    q = rows((kappa - lo)[g.eid]) / (hi - lo + 1e-8)
    qe = (2.0 * hi - kappa).clamp(min=0.0).sqrt() + 1.0
    return dict(R=R, p=p, kappa=kappa, prob_node=q / q.sum(), prob_edge=qe / qe.sum())


def exact(case, seed):
    call = case["call"]
    if call == "sample":
        return None  # draws and subgraphs are whole numbers
    if call in ("cg", "pcg", "rhs", "run", "run_host") and case["m"] * case["kc"] > 9e9:
        return None
    g = _Graph64(case, seed)
    if call == "build":
        return dict(val=g.val, deg=g.deg, ew=g.ew)
    if call == "finish":
        X = _solution_like(case, g.deg.float(), g.gen)
        return _tail64(g, _resistance64(g, X[:, :case["kc"]].double()))
    kc = case["kc"]
    if call in ("cg", "pcg", "rhs"):
        out = torch.zeros(g.n, (kc + 3) // 4 * 4, dtype=torch.float64, device=DEV)
        Y = _rhs64(g, case["K"], case.get("c0", 0), kc)
        out[:, :kc] = Y if call == "rhs" else _solve64(g, Y)
        return dict(Y=out) if call == "rhs" else dict(X=out)
    R = torch.zeros(g.m, dtype=torch.float64, device=DEV)
    for c0 in range(0, case["K"], kc):
        R += _resistance64(g, _solve64(g, _rhs64(g, case["K"], c0, min(kc, case["K"] - c0))))
    return _tail64(g, R)
