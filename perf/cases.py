"""The calls whose speed is tracked: SpMM, SDDMM, the condensed-tile plan and the graph
chains, through the package's public entry points, over the sizes that its configurations,
tests and benchmark use.  Inputs are drawn on the GPU from the seed alone."""
import math

import torch

import paper_2604_27985_gb300 as gb

DEV = "cuda"


def listed():
    return [
        # One layer of a small pruned model: a single short call, where launches count
        # (the 1,024^2 problem instance at 90%).
        _sparse("spmm_f32_1k", "spmm", 1024, 1024, 0.10, 64),
        _sparse("sddmm_f32_1k", "sddmm", 1024, 1024, 0.10, 64),
        # The benchmark's problem: a large 99%-sparse matrix whose dense operand stays in L2.
        _sparse("spmm_f32_65k", "spmm", 65536, 65536, 0.01, 64),
        _sparse("sddmm_f32_65k", "sddmm", 65536, 65536, 0.01, 32),
        # Skewed rows and sizes that are multiples of nothing: Zipf row lengths, width 100.
        _sparse("spmm_f32_zipf_ragged", "spmm", 30011, 41017, 0.02, 100, rows="zipf"),
        # The largest problem: 110 million entries, a dense operand past the L2 cache.
        _sparse("spmm_f32_1m", "spmm", 1048576, 1048576, 1e-4, 32),
        # A pruned layer in BF16 and, per-row scaled, in E4M3: unstructured 90% sparsity.
        _sparse("spmm_bf16_16k", "spmm", 16384, 16384, 0.10, 256, dtype="bf16"),
        _sparse("sddmm_e4m3_16k", "sddmm", 16384, 16384, 0.10, 256, dtype="e4m3"),
        # The same layer with half its entries in dense 16 x 8 blocks, through a plan that the
        # program makes once: the product, and the gradient at the stored entries.
        _sparse("tc_spmm_bf16_16k", "tc_spmm", 16384, 16384, 0.10, 256, rows="clustered", dtype="bf16"),
        _sparse("tc_sddmm_bf16_16k", "tc_sddmm", 16384, 16384, 0.10, 256, rows="clustered", dtype="bf16"),
        # Edge scores and aggregation over a batch of 512 graphs of uneven size, and the
        # attention form (softmax over each row's scores) over 128.
        {"name": "gnn_512", "op": "chain", "graphs": 512, "nmin": 1000, "nmax": 50000, "softmax": False},
        {"name": "gat_128", "op": "chain", "graphs": 128, "nmin": 1000, "nmax": 50000, "softmax": True},
    ]


def _sparse(name, op, M, K, density, N, rows="uniform", dtype="f32"):
    return {"name": name, "op": op, "M": M, "K": K, "density": density, "N": N, "rows": rows, "dtype": dtype}


def _log(rng, lo, hi):
    return math.exp(rng.uniform(math.log(lo), math.log(hi)))


def draw(rng):
    op = rng.choice(["spmm", "spmm", "sddmm", "sddmm", "tc_spmm", "tc_sddmm", "chain"])
    if op == "chain":
        return {"op": op, "graphs": int(_log(rng, 8, 300)), "nmin": int(_log(rng, 100, 1000)),
                "nmax": int(_log(rng, 5000, 50000)), "softmax": rng.random() < 0.4}
    if op in ("spmm", "sddmm"):
        M, K = int(_log(rng, 1000, 300000)), int(_log(rng, 1000, 300000))
        dtype = rng.choice(["f32", "f32", "bf16", "e4m3"])
        rows = rng.choice(["uniform", "uniform", "zipf", "clustered"])
        # mostly the usual widths, some of any size
        N = rng.choice([32, 64, 128, 256]) if rng.random() < 0.6 else rng.randint(8, 256)
        density = _log(rng, 1e-4, 0.12)
        most = 4e9
        if N % {"f32": 4, "bf16": 8, "e4m3": 16}[dtype]:
            most = 5e8
    else:
        M, K = int(_log(rng, 2000, 24000)), int(_log(rng, 2000, 24000))
        dtype = rng.choice(["bf16", "bf16", "e4m3"])
        rows = rng.choice(["clustered", "clustered", "uniform"])
        N = rng.choice([64, 128, 256]) if rng.random() < 0.7 else 16 * rng.randint(4, 20)
        if op == "tc_sddmm":  # the tiles take whole 128-byte blocks of an X or Y row
            N = {"bf16": 64, "e4m3": 128}[dtype] * rng.randint(1, 4)
        density = _log(rng, 0.01, 0.12)
        most = 6e9
    density = min(density, most / (M * K * N), 4e7 / (M * K))
    return {"op": op, "M": M, "K": K, "density": density, "N": N, "rows": rows, "dtype": dtype}


# ---- inputs ----------------------------------------------------------------------------------


def _columns(lengths, width, g):
    """Row offsets and, row after row, sorted distinct columns: row r draws lengths[r] of its
    width[r] columns (order statistics of uniforms, from normalised exponential gaps, which
    are whole numbers so that their running sums do not depend on the order of addition)."""
    rowptr = torch.zeros(lengths.numel() + 1, dtype=torch.int64, device=DEV)
    torch.cumsum(lengths, 0, out=rowptr[1:])
    n = int(rowptr[-1])
    row = torch.repeat_interleave(torch.arange(lengths.numel(), device=DEV), lengths, output_size=n)
    gaps = lambda k: (-torch.log1p(-torch.rand(k, generator=g, device=DEV)) * (1 << 24)).long() + 1
    run = torch.zeros(n + 1, dtype=torch.int64, device=DEV)
    torch.cumsum(gaps(n), 0, out=run[1:])
    before = run[rowptr[:-1]]
    total = run[rowptr[1:]] - before + gaps(lengths.numel())
    u = (run[1:] - before[row]).double() / total[row].double()
    free = (width - lengths + 1)[row]
    col = torch.minimum((u * free).long(), free - 1)
    col += torch.arange(n, device=DEV) - rowptr[row]
    return rowptr, row, col


def _sizes(seed=11):
    """The generator of row lengths and node counts, which belong to the case and not to the
    seed: two seeds' outputs have the same shape."""
    return torch.Generator(DEV).manual_seed(seed)


def _zipf(M, cap, T):
    """Row lengths ~ l^-1.5 on [1, 4096], scaled to about T entries in all, at most cap each."""
    g = _sizes()
    l = torch.arange(1, 4097, device=DEV, dtype=torch.float64)
    cdf = torch.cumsum(l ** -1.5, 0)
    u = torch.rand(M, generator=g, device=DEV, dtype=torch.float32).double() * cdf[-1]
    x = torch.searchsorted(cdf, u).clamp_(max=4095).double() + 1
    s = T / float(x.sum())
    for _ in range(8):
        s *= T / float((x * s).clamp_(max=cap).round().long().sum().clamp_(min=1))
    return (x * s).clamp_(max=cap).round().long()


def _pattern(c, g):
    """CSR pattern (int32 row offsets and column indices)."""
    M, K = c["M"], c["K"]
    T = max(1, round(c["density"] * M * K))
    if c["rows"] == "clustered":  # half in aligned 16 x 8 blocks of 51 entries, half anywhere else
        br, bc = M // 16, K // 8
        nb = max(1, round(0.5 * T / 51))
        pick = torch.randint(br * bc, (int(1.3 * nb) + 64,), generator=g, device=DEV).unique()
        pick = pick[torch.randperm(pick.numel(), generator=g, device=DEV)[:nb]].sort().values
        slot = torch.rand(nb, 128, generator=g, device=DEV).argsort(1)[:, :51]
        keys = ((pick[:, None] // bc * 16 + slot // 8) * K + pick[:, None] % bc * 8 + slot % 8).reshape(-1)
        rest = max(1, T - nb * 51)
        q = torch.randint(M * K, (int(1.5 * rest) + 64,), generator=g, device=DEV)
        b = q // K // 16 * bc + q % K // 8  # (a row or column past the whole blocks is in none of them)
        b = torch.where((q // K // 16 < br) & (q % K // 8 < bc), b, -1)
        q = q[pick[torch.searchsorted(pick, b).clamp_(max=nb - 1)] != b].unique()
        q = q[torch.randperm(q.numel(), generator=g, device=DEV)[:rest]]
        keys = torch.cat([keys, q]).sort().values
        row, col = keys // K, keys % K
        rowptr = torch.zeros(M + 1, dtype=torch.int64, device=DEV)
        torch.cumsum(torch.bincount(row, minlength=M), 0, out=rowptr[1:])
    else:
        if c["rows"] == "zipf":
            lengths = _zipf(M, min(K, max(4096, 4 * T // M)), T)
        else:
            lengths = torch.full((M,), T // M, dtype=torch.int64, device=DEV)
            lengths[torch.randperm(M, generator=g, device=DEV)[: T % M]] += 1
        rowptr, row, col = _columns(lengths, torch.full_like(lengths, K), g)
    return rowptr.int(), row, col.int()


def _e4m3_scale(amax):
    """FP32 row scales: the largest magnitude of a row takes the largest E4M3 code."""
    return torch.where(amax > 0, amax / 448.0, torch.ones_like(amax))


def _dense_inputs(x, dtype):
    """(stored tensor, row scales or None)"""
    if dtype == "bf16":
        return x.to(torch.bfloat16), None
    if dtype == "e4m3":
        s = _e4m3_scale(x.abs().amax(1))
        return (x / s[:, None]).to(torch.float8_e4m3fn).view(torch.uint8), s
    return x, None


def _inputs(c, seed):
    g = torch.Generator(DEV).manual_seed(seed)
    dtype = c["dtype"]
    rowptr, row, col = _pattern(c, g)
    vals = torch.rand(col.numel(), generator=g, device=DEV) * 2 - 1
    d = {"rowptr": rowptr, "colidx": col}
    if c["op"].endswith("spmm"):
        if dtype == "bf16":
            vals = vals.to(torch.bfloat16)
        elif dtype == "e4m3":
            amax = torch.zeros(c["M"], device=DEV).scatter_reduce_(0, row, vals.abs(), "amax")
            d["a_scale"] = _e4m3_scale(amax)
            vals = (vals / d["a_scale"][row]).to(torch.float8_e4m3fn).view(torch.uint8)
        B = torch.randn(c["K"], c["N"], generator=g, device=DEV)
        d["B"], d["b_scale"] = _dense_inputs(B, dtype)
    else:
        d["X"], d["x_scale"] = _dense_inputs(torch.randn(c["M"], c["N"], generator=g, device=DEV), dtype)
        d["Y"], d["y_scale"] = _dense_inputs(torch.randn(c["K"], c["N"], generator=g, device=DEV), dtype)
    d["vals"] = vals
    return d, row


def _graphs(c, seed):
    """A batch of graphs in a few flat arrays: node counts log-uniform, power-law degrees of
    mean about 16, no self loops, values 1 / degree; BF16 features of width 64, 128 or 256."""
    g = torch.Generator(DEV).manual_seed(seed)
    G, sizes = c["graphs"], _sizes()
    u = torch.rand(G, generator=sizes, device=DEV, dtype=torch.float64)
    ns = torch.exp(math.log(c["nmin"]) + u * (math.log(c["nmax"]) - math.log(c["nmin"]))).round().long()
    widths = torch.tensor([64, 128, 256], device=DEV)[torch.randint(3, (G,), generator=sizes, device=DEV)].tolist()
    n_of = torch.repeat_interleave(ns, ns)
    d = torch.arange(1, 2049, device=DEV, dtype=torch.float64)
    cdf = torch.cumsum(d ** -1.679, 0)
    v = torch.rand(n_of.numel(), generator=sizes, device=DEV, dtype=torch.float32).double() * cdf[-1]
    deg = torch.minimum(torch.searchsorted(cdf, v).clamp_(max=2047) + 1, n_of - 1)
    rowptr, row, col = _columns(deg, n_of - 1, g)
    starts = torch.zeros(G + 1, dtype=torch.int64, device=DEV)
    torch.cumsum(ns, 0, out=starts[1:])
    own = row - torch.repeat_interleave(starts[:-1], ns)[row]
    col += col >= own
    del own
    val = (1.0 / deg.double()).float()[row]
    edges = rowptr[starts].tolist()
    starts, ns = starts.tolist(), ns.tolist()
    pad = lambda n: -(-n // 128) * 128  # each array of a graph starts on a 512-byte boundary
    eo, fo = [0], [0]
    for k in range(G):
        eo.append(eo[-1] + pad(edges[k + 1] - edges[k]))
        fo.append(fo[-1] + pad(ns[k] * widths[k]))
    ro = [0]
    for n in ns:
        ro.append(ro[-1] + pad(n + 1))
    cols = torch.zeros(eo[-1], dtype=torch.int32, device=DEV)
    vals = torch.zeros(eo[-1], device=DEV)
    rps = torch.zeros(ro[-1], dtype=torch.int32, device=DEV)
    H = torch.randn(fo[-1], generator=g, device=DEV).to(torch.bfloat16)
    parts = []
    for k in range(G):
        m, n = edges[k + 1] - edges[k], ns[k]
        cols[eo[k]:eo[k] + m] = col[edges[k]:edges[k + 1]]
        vals[eo[k]:eo[k] + m] = val[edges[k]:edges[k + 1]]
        rps[ro[k]:ro[k] + n + 1] = rowptr[starts[k]:starts[k + 1] + 1] - edges[k]
        parts.append((slice(ro[k], ro[k] + n + 1), slice(eo[k], eo[k] + m), slice(fo[k], fo[k] + n * widths[k]), n,
                      widths[k]))
    return {"rowptr": rps, "colidx": cols, "vals": vals, "H": H, "parts": parts}


# ---- the calls -------------------------------------------------------------------------------


def prepare(case, seed):
    op = case["op"]
    if op == "chain":
        d = _graphs(case, seed)
        E, O = torch.zeros_like(d["vals"]), torch.zeros_like(d["H"])
        graphs = [(d["rowptr"][r], d["colidx"][e], d["vals"][e], d["H"][f].view(n, w), O[f].view(n, w), E[e])
                  for r, e, f, n, w in d["parts"]]
        return {"op": op, "E": E, "O": O, "plan": gb.GnnPlan(graphs, softmax=case["softmax"])}
    d, _ = _inputs(case, seed)
    d["op"] = op
    if op == "tc_spmm":
        d["plan"] = gb.TcPlan(d["rowptr"], d["colidx"], d["vals"], case["K"], row_scale=d.get("a_scale"))
    elif op == "tc_sddmm":  # a plan on the pattern; its values do not enter the SDDMM
        ones = torch.ones(d["vals"].numel(), device=DEV)
        v, s = (ones.to(torch.bfloat16), None) if case["dtype"] == "bf16" else (
            ones.to(torch.float8_e4m3fn).view(torch.uint8), torch.ones(case["M"], device=DEV))
        d["plan"] = gb.TcPlan(d["rowptr"], d["colidx"], v, case["K"], row_scale=s)
    return d


def run(state):
    s, op = state, state["op"]
    if op == "spmm":
        return gb.spmm(s["rowptr"], s["colidx"], s["vals"], s["B"], a_scale=s.get("a_scale"), b_scale=s["b_scale"])
    if op == "sddmm":
        return gb.sddmm(s["rowptr"], s["colidx"], s["vals"], s["X"], s["Y"], x_scale=s["x_scale"], y_scale=s["y_scale"])
    if op == "tc_spmm":
        return s["plan"].execute(s["B"], row_scale=s["b_scale"])
    if op == "tc_sddmm":
        return s["plan"].sddmm(s["vals"], s["X"], s["Y"], x_scale=s["x_scale"], y_scale=s["y_scale"])
    s["plan"].execute()
    return {"E": s["E"], "O": s["O"]}


def work(case):
    if case["op"] == "chain":  # each array once: CSR in, H in, E and O out; two products
        lo, hi = case["nmin"], case["nmax"]
        nodes = case["graphs"] * (hi - lo) / math.log(hi / lo)
        edges, w = 15.3 * nodes, (64 + 128 + 256) / 3
        return {"bytes": edges * 12 + nodes * (4 + 4 * w), "flops": 4 * edges * w}
    M, K, N = case["M"], case["K"], case["N"]
    nnz = round(case["density"] * M * K)
    e = {"f32": 4, "bf16": 2, "e4m3": 1}[case["dtype"]]
    scales = 4 * (M + K) if e == 1 else 0
    if case["op"].endswith("spmm"):
        return {"bytes": nnz * (4 + e) + 4 * (M + 1) + K * N * e + M * N * 4 + scales, "flops": 2 * nnz * N}
    return {"bytes": nnz * 12 + 4 * (M + 1) + (M + K) * N * e + scales, "flops": 2 * nnz * N}


# ---- 64 bits ---------------------------------------------------------------------------------


def _wide(x, scale=None):
    """A stored dense operand or value array in 64 bits."""
    if x.dtype == torch.uint8:
        x = x.view(torch.float8_e4m3fn).float()
    x = x.double()
    return x if scale is None else x * (scale.double()[:, None] if x.dim() == 2 else scale.double())


def _product(rowptr, colidx, vals, B):
    A = torch.sparse_csr_tensor(rowptr, colidx, vals, size=(rowptr.numel() - 1, B.shape[0]), check_invariants=False)
    return A @ B


def _sampled(row, col, s, X, Y):
    out = torch.empty(row.numel(), dtype=torch.float64, device=DEV)
    step = max(1, (1 << 28) // X.shape[1])
    for a in range(0, row.numel(), step):
        b = slice(a, a + step)
        out[b] = (X[row[b]] * Y[col[b].long()]).sum(1) * s[b]
    return out


def _rows(rowptr, n):
    lengths = (rowptr[1:] - rowptr[:-1]).long()
    return torch.repeat_interleave(torch.arange(lengths.numel(), device=DEV), lengths, output_size=n)


def exact(case, seed):
    if case["op"] == "chain":
        d = _graphs(case, seed)
        E = torch.zeros(d["vals"].numel(), dtype=torch.float64, device=DEV)
        O = torch.zeros(d["H"].numel(), dtype=torch.float64, device=DEV)
        for r, e, f, n, w in d["parts"]:
            rowptr, col, H = d["rowptr"][r], d["colidx"][e], d["H"][f].view(n, w).double()
            row = _rows(rowptr, col.numel())
            z = _sampled(row, col, d["vals"][e].double(), H, H)
            if case["softmax"]:
                top = torch.full((n,), -math.inf, dtype=torch.float64, device=DEV).scatter_reduce_(0, row, z, "amax")
                z = torch.exp(z - top[row])
                z = z / torch.zeros(n, dtype=torch.float64, device=DEV).index_add_(0, row, z)[row]
            E[e] = z
            O[f] = _product(rowptr, col, z, H).reshape(-1)
        return {"E": E, "O": O}
    d, row = _inputs(case, seed)
    if case["op"].endswith("spmm"):
        scale = d["a_scale"][row] if "a_scale" in d else None
        return _product(d["rowptr"], d["colidx"], _wide(d["vals"], scale), _wide(d["B"], d["b_scale"]))
    return _sampled(row, d["colidx"], d["vals"].double(), _wide(d["X"], d["x_scale"]), _wide(d["Y"], d["y_scale"]))
