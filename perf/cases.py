"""The work that is timed: C = A @ B through the public entry points of the package.

A case is a call as a program makes it, with its sizes.  The kinds are the ways the library is
used; sizes come from the repository's workload generators, tests and benchmark:

* ``execute``  a kept plan, one product per pass (a static graph or mask);
* ``step``     a fresh plan and one product per pass (a new graph or mask on each call);
* ``batch``    many uneven graphs in one persistent launch;
* ``gcn``      the GCN forward, every layer on one plan;
* ``serve``    a burst of requests with host operands to a server whose plans are resident.

Matrices: ``uniform`` (fixed row degree, distinct uniform columns), ``rmat`` (relabelled
power-law graph, values 1 / degree), ``attention`` (64 x 64 block mask, causal band of 4 blocks,
3 % random blocks, one scattered nonzero per row, rows summing to 1).  ``TM`` = 0 keeps every
nonzero on the CUDA cores; otherwise the plan forms dense tiles of TM x TK.
"""
import math

import numpy as np
import torch

import paper_2606_22482_gb300 as ns
from paper_2606_22482_gb300.gcn import GCN

DEV = "cuda"


# ---------------------------------------------------------------------------------------------
# the cases
# ---------------------------------------------------------------------------------------------
def _case(kind, matrix="rmat", m=0, deg=16, K=64, bf16=False, TM=0, TK=0, tau=0, W=256, count=1):
    return {"kind": kind, "matrix": matrix, "m": m, "deg": deg, "K": K, "bf16": bf16, "TM": TM, "TK": TK,
            "tau": tau, "W": W, "count": count}


def listed():
    def c(name, *a, **k):
        return dict(_case(*a, **k), name=name)
    return [
        # the smallest configuration: launch and latency bound
        c("small_f32_k32", "execute", "uniform", 4096, 16, 32),
        # one request's graph of the serving pool's median size, planned and executed once
        c("new_graph_bf16_k64", "step", "rmat", 18433, 16, 64, bf16=True),
        # a power-law graph of a million nodes with a kept plan (a GNN's aggregation)
        c("powerlaw_f32_k128", "execute", "rmat", 1 << 20, 16, 128, W=512),
        # the same re-planned on each call, as the benchmark's step does
        c("powerlaw_step_f32_k128", "step", "rmat", 1 << 20, 16, 128, W=512),
        # BF16 features of a width that is no power of two, on an odd number of nodes
        c("graph_bf16_k96", "execute", "rmat", 300007, 16, 96, bf16=True),
        # wide features
        c("wide_f32_k512", "execute", "rmat", 100003, 12, 512),
        # a sparse-attention mask with dense tiles on the tensor cores, kept over many calls
        c("attention_bf16", "execute", "attention", 32768, 0, 128, bf16=True, TM=64, TK=32, tau=512),
        c("attention_f32", "execute", "attention", 32768, 0, 128, TM=64, TK=32, tau=512),
        # a mask that changes on each call
        c("attention_step_bf16", "step", "attention", 32768, 0, 128, bf16=True, TM=64, TK=32, tau=512),
        # 512 uneven graphs in one launch
        c("batch_f32_k64", "batch", "mix", 0, 0, 64, W=512, count=512),
        # a GNN inference: two layers on one plan
        c("gcn_f32_k128", "gcn", "rmat", 200003, 16, 128),
        # a burst of mixed requests at a server
        c("serve_burst", "serve", "rmat", 18433, 16, 0, count=32),
    ]


def _log(rng, lo, hi):
    return int(round(math.exp(rng.uniform(math.log(lo), math.log(hi)))))


def draw(rng):
    kind = rng.choice(["execute", "execute", "execute", "step", "step", "mask", "mask", "mask_step", "batch", "gcn",
                       "serve"])
    bf16 = rng.random() < 0.5
    if kind in ("mask", "mask_step"):
        TM, TK = rng.choice([(64, 32), (64, 32), (32, 32), (16, 16)])
        # BF16 masks up to K = 256 (TM 64); the tile shape bounds TM * K
        return _case("execute" if kind == "mask" else "step", "attention", _log(rng, 2000, 32768), 0,
                     rng.choice([32, 64, 72, 128, 128, 256]), bf16=bf16, TM=TM, TK=TK, tau=TM * TK // 4)
    if kind == "batch":
        return _case("batch", "mix", 0, 0, rng.choice([32, 64, 128]), bf16=bf16, W=rng.choice([256, 512]),
                     count=_log(rng, 16, 256))
    if kind == "serve":
        return _case("serve", "rmat", _log(rng, 2000, 60000), 16, 0, count=_log(rng, 4, 32))
    m = _log(rng, 4096, 1 << 20)
    deg = rng.randint(8, 32)
    if kind == "gcn":
        return _case("gcn", "rmat", min(m, 500000), min(deg, 20), rng.choice([64, 128]))
    widths = [8, 16, 24, 32, 64, 64, 96, 128, 128, 136, 256, 512]
    K = rng.choice([k for k in widths if k * m * deg <= 1 << 31])
    matrix = rng.choice(["rmat", "rmat", "uniform"]) if m <= 300000 else "rmat"
    return _case(kind, matrix, m, deg, K, bf16=bf16, W=rng.choice([256, 512]))


# ---------------------------------------------------------------------------------------------
# inputs, drawn on the GPU
# ---------------------------------------------------------------------------------------------
def _gen(seed):
    g = torch.Generator(device=DEV)
    g.manual_seed(seed)
    return g


def _rmat_pairs(g, count, scale):
    """RMAT (0.57, 0.19, 0.19, 0.05): one quadrant, hence one bit of each id, per level."""
    i = torch.zeros(count, dtype=torch.int64, device=DEV)
    j = torch.zeros_like(i)
    for _ in range(scale):
        u = torch.rand(count, generator=g, device=DEV)
        bi = u >= 0.76
        bj = ((u >= 0.57) & ~bi) | (u >= 0.95)
        i = (i << 1) | bi
        j = (j << 1) | bj
    return i, j


def _pick(g, keys, count):
    """`count` of the sorted distinct keys, at random, sorted."""
    if keys.numel() <= count:
        return keys
    at = torch.randperm(keys.numel(), generator=g, device=DEV)[:count]
    return keys[at].sort().values


def _csr(m, key, vals=None):
    """CSR of the sorted distinct keys row * m + column; vals None: 1 / row degree."""
    row = torch.div(key, m, rounding_mode="floor")
    deg = torch.bincount(row, minlength=m)
    rowptr = torch.zeros(m + 1, dtype=torch.int64, device=DEV)
    rowptr[1:] = deg.cumsum(0)
    if vals is None:
        vals = (1.0 / deg.double())[row].float()
    return {"m": m, "n": m, "rowptr": rowptr.int(), "colidx": (key - row * m).int(), "vals": vals}


def _rmat(g, m, deg):
    scale = max(1, math.ceil(math.log2(m)))
    target = m * deg
    keys = torch.empty(0, dtype=torch.int64, device=DEV)
    for _ in range(16):
        need = target - keys.numel()
        if need <= 0:
            break
        i, j = _rmat_pairs(g, int(need * 1.35) + 1024, scale)
        ok = (i < m) & (j < m)
        keys = torch.unique(torch.cat([keys, i[ok] * m + j[ok]]))
    keys = _pick(g, keys, target)
    perm = torch.randperm(m, generator=g, device=DEV)
    i, j = torch.div(keys, m, rounding_mode="floor"), keys % m
    return _csr(m, (perm[i] * m + perm[j]).sort().values)


def _uniform(g, m, deg):
    """deg distinct uniform columns per row: a random start and distinct random steps around the ring."""
    step = torch.rand(m, deg, generator=g, device=DEV, dtype=torch.float64)
    step = (step / step.sum(1, keepdim=True) * (m - deg)).long() + 1      # >= 1, sums to <= m
    col = (step.cumsum(1) + torch.randint(0, m, (m, 1), generator=g, device=DEV)) % m
    key = (torch.arange(m, device=DEV)[:, None] * m + col).reshape(-1).sort().values
    return _csr(m, key, torch.rand(m * deg, generator=g, device=DEV) * 2 - 1)


def _attention(g, n):
    nb = -(-n // 64)
    bi = torch.arange(nb, device=DEV)
    active = torch.rand(nb, nb, generator=g, device=DEV) < 0.03
    off = bi[:, None] - bi[None, :]
    active |= (off >= 0) & (off < 4)
    mask = active.repeat_interleave(64, 0).repeat_interleave(64, 1)[:n, :n].contiguous()
    # one scattered nonzero per row: the first of 16 random columns outside its active blocks
    cand = torch.randint(0, n, (n, 16), generator=g, device=DEV)
    free = ~mask.gather(1, cand)
    first = free.int().argmax(1, keepdim=True)
    mask.scatter_(1, cand.gather(1, first), True)
    deg = mask.sum(1)
    rowptr = torch.zeros(n + 1, dtype=torch.int64, device=DEV)
    rowptr[1:] = deg.cumsum(0)
    at = mask.view(-1).nonzero().view(-1)
    row = torch.div(at, n, rounding_mode="floor")
    raw = torch.rand(at.numel(), generator=g, device=DEV, dtype=torch.float64) + 1e-6
    end = raw.cumsum(0)
    total = end[rowptr[1:] - 1] - torch.where(rowptr[:-1] > 0, end[(rowptr[:-1] - 1).clamp(min=0)], 0.0)
    vals = (raw / total[row]).float()
    return {"m": n, "n": n, "rowptr": rowptr.int(), "colidx": (at - row * n).int(), "vals": vals}


def _mix(g, count):
    """`count` graphs of 1000 to 50000 nodes (spread over the logarithm), mean degree 8 to 32: half of
    each graph's edges uniform, half RMAT.  All graphs are drawn together and cut apart at the end."""
    n = torch.exp((torch.arange(count, device=DEV) + 0.5) / count * math.log(50.0) + math.log(1000.0)).round().long()
    half = (n * (torch.rand(count, generator=g, device=DEV) * 24 + 8) / 2).long()
    base = torch.cat([n.new_zeros(1), n.cumsum(0)])
    of = torch.repeat_interleave(torch.arange(count, device=DEV), half)
    nn = n[of]
    ui, uj = ((torch.rand(of.numel(), generator=g, device=DEV, dtype=torch.float64) * nn).long() for _ in range(2))
    scale = torch.ceil(torch.log2(n.double())).long()[of]
    i, j = torch.zeros_like(of), torch.zeros_like(of)
    for level in range(16):
        u = torch.rand(of.numel(), generator=g, device=DEV)
        on = level < scale
        bi = u >= 0.76
        bj = ((u >= 0.57) & ~bi) | (u >= 0.95)
        i = torch.where(on, (i << 1) | bi, i)
        j = torch.where(on, (j << 1) | bj, j)
    ok = (i < nn) & (j < nn)
    b = base[of]
    key = torch.unique(torch.cat([((b + ui) << 16) | uj, (((b + i) << 16) | j)[ok]]))  # (row of all, column in graph)
    row, col = key >> 16, (key & 0xffff).int()
    rowptr = torch.cat([row.new_zeros(1), torch.bincount(row, minlength=int(base[-1])).cumsum(0)])
    vals = torch.rand(key.numel(), generator=g, device=DEV) * 2 - 1
    cut = base.tolist()
    edge = rowptr[base].tolist()
    out = []
    for k in range(count):
        r0, r1, e0, e1 = cut[k], cut[k + 1], edge[k], edge[k + 1]
        out.append({"m": r1 - r0, "n": r1 - r0, "rowptr": (rowptr[r0:r1 + 1] - e0).int(),
                    "colidx": col[e0:e1].clone(), "vals": vals[e0:e1].clone()})
    return out


def _features(g, rows, K, bf16):
    B = torch.randn(rows, K, generator=g, device=DEV)
    return B.bfloat16() if bf16 else B


def _matrix(case, g):
    if case["matrix"] == "rmat":
        return _rmat(g, case["m"], case["deg"])
    if case["matrix"] == "uniform":
        return _uniform(g, case["m"], case["deg"])
    return _attention(g, case["m"])


def _tune(case):
    t = ns.tune_default()
    t.chunk_nnz = t.absorb_cap = case["W"]
    if case["TM"]:
        t.TM, t.TK, t.tau_tile = case["TM"], case["TK"], case["tau"]
    return t


# the server's pool: node counts as multiples of case["m"], spread as the lognormal pool's are
_SERVE_POOL = (0.1, 0.3, 0.7, 1.0, 1.6, 3.0)


def _requests(case):
    """(graph, K, bf16) of each request of a burst, in order."""
    rng = np.random.default_rng(case["count"])
    return [(int(rng.integers(0, len(_SERVE_POOL))), int(rng.choice([32, 64, 128])), bool(rng.integers(0, 2)))
            for _ in range(case["count"])]


def _inputs(case, seed):
    """(matrices, dense operands) of a case: the same for prepare() and exact()."""
    g = _gen(seed)
    if case["kind"] == "batch":
        As = _mix(g, case["count"])
        rows = sum(A["m"] for A in As)
        return As, [_features(g, rows, case["K"], case["bf16"])]
    if case["kind"] == "serve":
        As = [_rmat(g, max(64, int(case["m"] * f)), case["deg"]) for f in _SERVE_POOL]
        return As, [_features(g, As[k]["n"], K, b) for k, K, b in _requests(case)]
    A = _matrix(case, g)
    X = _features(g, A["n"], case["K"], case["bf16"])
    if case["kind"] == "gcn":
        K = case["K"]
        return [A], [X] + [torch.randn(K, K, generator=g, device=DEV) / math.sqrt(K) for _ in range(2)]
    return [A], [X]


def _pinned(t):
    """A page-locked host copy of t as a numpy array (BF16 as its 16-bit patterns)."""
    t = t.cpu()
    return (t.view(torch.int16) if t.dtype == torch.bfloat16 else t).pin_memory().numpy()


def prepare(case, seed):
    As, Bs = _inputs(case, seed)
    K, dt = case["K"], ns.NS_BF16 if case["bf16"] else ns.NS_F32
    kind = case["kind"]
    s = {"kind": kind, "dt": dt, "K": K, "tune": _tune(case)}
    if kind == "serve":
        sv = ns.Server(hbm_budget_bytes=8 << 30, max_inflight=64)
        ids = [sv.register({k: (v.cpu().numpy() if torch.is_tensor(v) else v) for k, v in A.items()}) for A in As]
        reqs = []
        for (k, _, bf16), B in zip(_requests(case), Bs):
            C = torch.empty(As[k]["m"], B.shape[1]).pin_memory().numpy()
            reqs.append((ids[k], _pinned(B), C, ns.NS_BF16 if bf16 else ns.NS_F32))
        s.update(server=sv, reqs=reqs)
        _serve(s)  # the plans of the graphs become resident
        return s
    A = As[0]
    s.update(A=A, B=Bs[0])
    if kind == "batch":
        at = np.cumsum([0] + [a["m"] for a in As]).tolist()
        s["C"] = torch.empty(at[-1], K, device=DEV)
        s["Bs"] = [Bs[0][p:q] for p, q in zip(at, at[1:])]
        s["Cs"] = [s["C"][p:q] for p, q in zip(at, at[1:])]
        s["batch"] = ns.Batch(As, [K] * len(As), dt, s["tune"])
        return s
    if kind != "gcn":
        s["C"] = torch.empty(A["m"], K, device=DEV)
    if kind != "step":
        s["plan"] = ns.spmm_plan(A, K, dt, s["tune"])
    if kind == "gcn":
        s["net"] = GCN(s["plan"], Bs[1:])
    return s


def _serve(s):
    sv = s["server"]
    waiting = [sv.submit(g, B, C, dt) for g, B, C, dt in s["reqs"]]
    while waiting:
        waiting = [t for t in waiting if not sv.poll(t)[0]]
    return [C for _, _, C, _ in s["reqs"]]


def run(state):
    kind = state["kind"]
    if kind == "execute":
        state["plan"].execute(state["B"], state["C"])
        return state["C"]
    if kind == "step":
        with ns.spmm_plan(state["A"], state["K"], state["dt"], state["tune"]) as plan:
            plan.execute(state["B"], state["C"])
        return state["C"]
    if kind == "batch":
        state["batch"].execute(state["Bs"], state["Cs"])
        return state["C"]
    if kind == "gcn":
        return state["net"].forward(state["B"])
    return _serve(state)


# ---------------------------------------------------------------------------------------------
# what a pass cannot do without, and its result in 64 bits
# ---------------------------------------------------------------------------------------------
def _nnz(case):
    """Nonzeros of a case's matrices (attention: the expected number)."""
    if case["matrix"] == "attention":
        nb = case["m"] / 64
        return int(case["m"] * 64 * (min(4, nb) + 0.03 * max(0.0, nb - 4)) + case["m"])
    if case["matrix"] == "mix":
        return int(case["count"] * 49000 / math.log(50) * 20 * 0.98)
    return case["m"] * case["deg"]


def work(case):
    K, es, kind = case["K"], 2 if case["bf16"] else 4, case["kind"]
    if kind == "serve":
        byt = flops = 0.0
        for k, K, b in _requests(case):
            rows = max(64, int(case["m"] * _SERVE_POOL[k]))
            nnz = rows * case["deg"]
            byt += 4 * (rows + 1) + 8 * nnz + K * rows * (4 + (2 if b else 4))
            flops += 2.0 * nnz * K
        return {"bytes": byt, "flops": flops}
    m = case["count"] * 49000 / math.log(50) if kind == "batch" else case["m"]
    nnz = _nnz(case)
    # an RMAT graph has about half of its columns empty: B's rows that no edge names are not read
    touched = m * 0.53 if case["matrix"] == "rmat" else m
    spmm = {"bytes": 4 * (m + 1) + 8 * nnz + es * K * touched + 4 * K * m, "flops": 2.0 * nnz * K}
    if kind == "gcn":  # per layer the dense product reads and writes m x K once more, each way
        return {"bytes": 2 * (spmm["bytes"] + 8 * K * m), "flops": 2 * (spmm["flops"] + 2.0 * m * K * K)}
    return spmm


def _product(A, B):
    """A @ B in 64 bits (torch's sparse CSR product)."""
    S = torch.sparse_csr_tensor(A["rowptr"].long(), A["colidx"].long(), A["vals"].double(), (A["m"], A["n"]))
    return S @ B.double()


def exact(case, seed):
    As, Bs = _inputs(case, seed)
    if case["kind"] == "batch":
        at = np.cumsum([0] + [a["m"] for a in As]).tolist()
        return torch.cat([_product(A, Bs[0][p:q]) for A, p, q in zip(As, at, at[1:])])
    if case["kind"] == "serve":
        return [_product(As[k], B) for (k, _, _), B in zip(_requests(case), Bs)]
    if case["kind"] == "gcn":
        H = Bs[0].double()
        for li, W in enumerate(Bs[1:]):
            H = _product(As[0], H @ W.double())
            if li == 0:
                H = H.relu()
        return H
    return _product(As[0], Bs[0])
