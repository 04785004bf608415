"""The work that programs give to the sparse-chain executor, as cases that can be timed and compared.

A program builds the compressed tensor B once (``SparseTensor``), keeps the dense operands on the device and
evaluates a chain again and again, through ``SparseTensor.run``: one pass here is one such call with the default
schedule.  ``listed`` holds the cases (every expression of the library, from calls of a few microseconds of device
work to the headline workload), ``draw`` gives further cases of the same ranges.

Inputs follow the laws of ``workloads/configs.py`` (Zipf slice sizes, geometric fiber lengths, rank-Zipf or Poisson
row degrees, distinct pseudo-uniform coordinates, COO in random order), drawn on the device because a case of tens
of millions of nonzeros takes numpy too long.
"""
import math

import numpy as np
import torch

import paper_2311_09549_b200 as sa

#: Ranks the library is compiled for, per expression and rank name.
RANKS = {
    "spttm_ttm3": {"L": (16, 32), "M": (16, 32)},
    "spttm_ttm4": {"L": (16,), "M": (16,), "N": (16,)},
    "sddmm_spmm": {"K": (32, 64, 128), "L": (32, 64, 128)},
    "spmm_gemm": {"L": (128, 256), "M": (32, 64)},
    "ttmc3": {"L": (16, 32), "M": (16, 32), "N": (16, 32)},
    "sddmm_spmm_gemm": {"K": (32, 64, 128), "L": (32, 64, 128), "M": (32, 64)},
    "spmmh_gemm": {"L": (128, 256), "M": (32, 64)},
    "mttkrp_gemm": {"R": (32,), "M": (32, 64)},
    "spttm_spttm": {"L": (32, 64), "M": (32, 64)},
}
ORDER = {"spttm_ttm3": 3, "spttm_ttm4": 4, "ttmc3": 3, "mttkrp_gemm": 3, "spttm_spttm": 3,
         "sddmm_spmm": 2, "spmm_gemm": 2, "sddmm_spmm_gemm": 2, "spmmh_gemm": 2}


def _csf(name, expr, dims, nnz, alpha, fiber, **ranks):
    """Order-3 or order-4 tensor: Zipf(alpha) slice sizes (0: uniform coordinates over i), mean fan-out `fiber`."""
    return dict({"name": name, "expr": expr, "nnz": nnz, "alpha": alpha, "fiber": fiber},
                **{"d%d" % i: d for i, d in enumerate(dims)}, **{"rank_" + k: v for k, v in ranks.items()})


def _csr(name, expr, dims, nnz, alpha, cap, **ranks):
    """Matrix: rank-Zipf(alpha) row degrees of at most `cap` (alpha 0: Poisson degrees), uniform distinct columns."""
    return dict({"name": name, "expr": expr, "nnz": nnz, "alpha": alpha, "cap": cap},
                **{"d%d" % i: d for i, d in enumerate(dims)}, **{"rank_" + k: v for k, v in ranks.items()})


def listed():
    return [
        # The smallest call: a 200^3 tensor (configuration 1), where launches and the host's part of the call count.
        _csf("ttm3-small", "spttm_ttm3", (200, 200, 200), 20_000, 0.0, 1.3, L=16, M=16),
        # A TTMc step of a Tucker decomposition on an ordinary tensor of odd sizes, unequal ranks, mild skew.
        _csf("ttm3-ordinary", "spttm_ttm3", (9_973, 12_007, 15_013), 2_300_003, 1.0, 5.0, L=32, M=16),
        # The headline workload (configuration 2): 50 M nonzeros, strong skew, 410 MB of output.
        _csf("ttm3-large", "spttm_ttm3", (100_000, 80_000, 80_000), 50_000_000, 1.2, 8.0, L=32, M=32),
        # The order-4 TTMc chain (configuration 5 at its quarter scale).
        _csf("ttm4", "spttm_ttm4", (12_500, 20_000, 20_000, 20_000), 25_000_000, 1.2, 6.0, L=16, M=16, N=16),
        # Attention-like SDDMM -> SpMM on a power-law graph (configuration 3).
        _csr("sddmm-spmm", "sddmm_spmm", (1_000_000, 1_000_000), 30_000_000, 1.5, 50_000, K=64, L=64),
        # One layer of a graph network on a small graph (workload 7 at its mini scale): several short launches.
        _csr("sddmm-spmm-gemm-small", "sddmm_spmm_gemm", (6_000, 6_000), 60_000, 1.5, 1_500, K=32, L=32, M=32),
        # Feature aggregation and projection over a whole graph (configuration 4 at its quarter scale).
        _csr("spmm-gemm", "spmm_gemm", (1_000_000, 1_000_000), 25_000_000, 0.0, 0, L=256, M=64),
        # The same for a batch of rows against a large feature table: few rows, the other association order.
        _csr("spmm-gemm-few-rows", "spmm_gemm", (20_011, 1_000_000), 500_009, 0.0, 0, L=128, M=32),
        # SpMM with a Hadamard product, then a projection (workload 8 at its quarter scale).
        _csr("spmmh-gemm", "spmmh_gemm", (1_000_000, 1_000_000), 25_000_000, 0.0, 0, L=256, M=64),
        # All-mode TTMC, the core update of a Tucker decomposition (workload 6, nell-2 shaped, a quarter of the nonzeros).
        _csf("ttmc3", "ttmc3", (12_000, 9_000, 288_000), 19_220_000, 1.2, 8.0, L=16, M=16, N=16),
        # MTTKRP of a CP decomposition followed by a small dense factor (workload 9, a quarter of it).
        _csf("mttkrp-gemm", "mttkrp_gemm", (25_000, 80_000, 80_000), 12_500_000, 1.2, 8.0, R=32, M=32),
        # Two sparse tensor-times-matrix products with a sparse output (workload 10, a quarter of it, odd sizes).
        _csf("spttm-spttm", "spttm_spttm", (24_989, 79_999, 80_021), 12_499_993, 1.2, 8.0, L=32, M=32),
    ]


def _log_int(rng, lo, hi):
    return int(round(math.exp(rng.uniform(math.log(lo), math.log(hi)))))


def draw(rng):
    expr = rng.choice(sorted(RANKS))
    ranks = {k: rng.choice(v) for k, v in sorted(RANKS[expr].items())}
    nnz = _log_int(rng, 10_000, 12_000_000 if ORDER[expr] == 4 else 16_000_000)
    if ORDER[expr] == 2:
        rows = min(1_000_000, max(64, int(nnz / math.exp(rng.uniform(math.log(4), math.log(60))))))
        cols = min(1_000_000, max(1_000, int(rows * math.exp(rng.uniform(math.log(0.5), math.log(4))))))
        alpha = rng.choice([0.0, 0.8, 1.2, 1.5]) if expr.startswith("sddmm") else 0.0
        cap = min(50_000, max(cols // 4, 2 * (nnz // rows + 1)))
        c = _csr("", expr, (rows, cols), nnz, alpha, cap if alpha else 0, **ranks)
    else:
        order = ORDER[expr]
        per_slice = math.exp(rng.uniform(math.log(50), math.log(4_000)))
        dims = [min(300_000, max(64, int(nnz / per_slice)))]
        dims += [_log_int(rng, 1_000, 100_000 if order == 3 else 30_000) for _ in range(order - 1)]
        # room for the head slice of the steepest law
        dims[-1] = max(dims[-1], 64 * nnz // math.prod(dims[1:-1]) + 1)
        c = _csf("", expr, dims, nnz, rng.choice([0.0, 0.8, 1.0, 1.2, 1.3]), round(math.exp(rng.uniform(math.log(1.5), math.log(20 if order == 3 else 8))), 2), **ranks)
    del c["name"]
    return c


# ---------------------------------------------------------------------------------------------- inputs

def _dims(case):
    return [case["d%d" % i] for i in range(ORDER[case["expr"]])]


def _zipf_sizes(case):
    """Slice sizes by rank (largest first), summing to the number of nonzeros; alpha > 0."""
    w = np.arange(1, case["d0"] + 1, dtype=np.float64) ** -case["alpha"]
    x = case["nnz"] * (w / w.sum())
    n = np.floor(x).astype(np.int64)
    n[np.argsort(n - x, kind="stable")[:case["nnz"] - int(n.sum())]] += 1
    return n


def _mix(x, key, salt):
    """31 pseudo-random bits per element, from integer arithmetic alone."""
    h = x * -7046029254386353131 + key * -4658895280553007687 + (salt + 1) * 1181783497276652981
    h = (h ^ (h >> 29)) * -4417276706812531889
    return ((h ^ (h >> 32)) * 2685821657736338717 >> 33) & 0x7fffffff


def _distinct(index, key, dim):
    """The index-th of dim distinct pseudo-uniform values in [0, dim): a permutation keyed by `key` (a Feistel network
    over two mixed-radix digits, walked on until the value lies in range)."""
    a = math.isqrt(dim - 1) + 1
    b = -(-dim // a)

    def once(v, key):
        hi, lo = torch.div(v, b, rounding_mode="floor"), v % b
        for r in range(3):
            hi = (hi + _mix(lo, key, 2 * r)) % a
            lo = (lo + _mix(hi, key, 2 * r + 1)) % b
        return hi * b + lo

    v = once(index, key)
    while True:
        out = (v >= dim).nonzero().flatten()
        if out.numel() == 0:
            return v
        v[out] = once(v[out], key[out])


def _starts_to_ids(start):
    return torch.cumsum(start.to(torch.int64), 0) - 1


def _index_since(start):
    """Position of every element since the last set flag."""
    at = torch.arange(start.numel(), device=start.device)
    return at - start.nonzero().flatten()[_starts_to_ids(start)]


def _open(parent_start, prob, gen, longest, most, total):
    """Flags where a child level opens: at every parent, elsewhere with probability `prob`, after `longest` nonzeros at the
    latest, at most `most` times per parent; some at random more or fewer, so that there are `total` of them."""
    n, dev = parent_start.numel(), parent_start.device
    must = parent_start | (_index_since(parent_start) % longest == 0)
    flag = must | (torch.rand(n, device=dev, generator=gen) < prob)
    excess = int(flag.sum()) - total
    free = (flag & ~must if excess > 0 else ~flag).nonzero().flatten()
    flag[free[torch.randperm(free.numel(), device=dev, generator=gen)[:abs(excess)]]] = excess < 0
    child = _starts_to_ids(flag)
    first = child[parent_start.nonzero().flatten()][_starts_to_ids(parent_start)]
    return flag & (child - first < most)


def _coords(case, gen):
    """int64 coordinates of B on the device, one tensor per mode, sorted."""
    dims, nnz, order = _dims(case), case["nnz"], ORDER[case["expr"]]
    dev = gen.device
    salt = int(torch.randint(1 << 40, (1,), device=dev, generator=gen))
    if case["alpha"] == 0:
        sizes = torch.bincount(torch.randint(dims[0], (nnz,), device=dev, generator=gen), minlength=dims[0])
        if order == 2:
            # a row holds at most `cols` distinct columns (far above the Poisson degrees of every case)
            assert int(sizes.max()) <= dims[1]
    else:
        by_rank = torch.from_numpy(_zipf_sizes(case) if order > 2 else _powerlaw_degrees(case)).to(dev)
        sizes = torch.empty_like(by_rank)
        sizes[torch.randperm(dims[0], device=dev, generator=gen)] = by_rank
    i = torch.repeat_interleave(torch.arange(dims[0], device=dev), sizes)
    start = torch.ones(nnz, dtype=torch.bool, device=dev)
    start[1:] = i[1:] != i[:-1]
    if order == 2:
        return [i, _distinct(_index_since(start), i + salt, dims[1])]
    starts = [start]
    per_slice = sizes[i].to(torch.float64)
    counts = _level_counts(case)
    above = torch.zeros(nnz, dtype=torch.float64, device=dev)      # chance that a nonzero opens the level above
    for level in range(1, order - 1):
        prob = torch.full((nnz,), case["fiber"] ** -(order - 1.0 - level), dtype=torch.float64, device=dev)
        if level == 1:      # a slice has room for dims[1] fibers: where that binds they are longer
            prob = torch.minimum(prob, 0.9 * dims[1] / per_slice)
        prob = torch.maximum(prob, above)
        below = math.prod(dims[level + 1:])
        starts.append(_open(starts[-1], (prob - above) / (1 - above), gen, max(1, below // 2), dims[level],
                            int(round(counts[level]))))
        above = prob
    cols = [i]
    for level in range(1, order):
        parent = starts[level - 1]
        if level == order - 1:
            index = _index_since(parent)
        else:
            child = _starts_to_ids(starts[level])
            index = child - child[parent.nonzero().flatten()][_starts_to_ids(parent)]
        cols.append(_distinct(index, _starts_to_ids(parent) + salt * (level + 1), dims[level]))
    return cols


def _powerlaw_degrees(case):
    """Row degrees by rank: min(cap, s rank^-alpha) with s such that they sum to the number of nonzeros."""
    law, cap, nnz = np.arange(1, case["d0"] + 1, dtype=np.float64) ** -case["alpha"], min(case["cap"], case["d1"]), case["nnz"]
    lo, hi = 0.0, float(cap) * case["d0"] ** case["alpha"] + 1.0
    for _ in range(60):
        mid = 0.5 * (lo + hi)
        lo, hi = (mid, hi) if np.minimum(cap, mid * law).sum() < nnz else (lo, mid)
    x = np.minimum(cap, hi * law)
    d = np.floor(x).astype(np.int64)
    missing = nnz - int(d.sum())
    if missing > 0:
        d[np.argsort(np.where(d < cap, d - x, 1.0), kind="stable")[:missing]] += 1
    elif missing < 0:
        d[np.nonzero(d > 0)[0][missing:]] -= 1
    return d


def _operand_shapes(case):
    d = _dims(case)
    r = {k[5:]: v for k, v in case.items() if k.startswith("rank_")}
    return {
        "spttm_ttm3": lambda: [(d[1], r["L"]), (d[2], r["M"])],
        "spttm_ttm4": lambda: [(d[1], r["L"]), (d[2], r["M"]), (d[3], r["N"])],
        "sddmm_spmm": lambda: [(d[0], r["K"]), (d[1], r["K"]), (d[1], r["L"])],
        "spmm_gemm": lambda: [(d[1], r["L"]), (r["L"], r["M"])],
        "ttmc3": lambda: [(d[0], r["L"]), (d[1], r["M"]), (d[2], r["N"])],
        "sddmm_spmm_gemm": lambda: [(d[0], r["K"]), (d[1], r["K"]), (d[1], r["L"]), (r["L"], r["M"])],
        "spmmh_gemm": lambda: [(d[1], r["L"]), (d[1], r["L"]), (r["L"], r["M"])],
        "mttkrp_gemm": lambda: [(d[1], r["R"]), (d[2], r["R"]), (r["R"], r["M"])],
        "spttm_spttm": lambda: [(d[2], r["L"]), (r["L"], r["M"])],
    }[case["expr"]]()


def inputs(case, seed):
    """(dims, COO coordinates, values, dense operands): coordinates and values in random order, all on the device."""
    dev = torch.device("cuda")
    gen = torch.Generator(device=dev)
    gen.manual_seed(seed)
    cols = _coords(case, gen)
    perm = torch.randperm(case["nnz"], device=dev, generator=gen)
    coords = torch.stack([c.to(torch.int32)[perm] for c in cols], dim=1)
    del cols, perm
    vals = torch.rand(case["nnz"], device=dev, generator=gen)
    if not case["expr"].startswith("sddmm"):
        vals = 2 * vals - 1
    draw_dense = torch.randn if ORDER[case["expr"]] == 2 else torch.rand
    ops = [draw_dense(s, device=dev, generator=gen) for s in _operand_shapes(case)]
    if ORDER[case["expr"]] > 2:
        ops = [2 * x - 1 for x in ops]
    return _dims(case), coords, vals, ops


def prepare(case, seed):
    dims, coords, vals, ops = inputs(case, seed)
    fmt = sa.SA_FMT_CSR if len(dims) == 2 else sa.SA_FMT_CSF
    B = sa.SparseTensor(dims, coords.cpu().numpy(), vals.cpu().numpy(), fmt, device=0)
    return {"B": B, "expr": case["expr"], "ops": ops}


def run(state):
    out, _ = state["B"].run(state["expr"], state["ops"])
    return out


# ------------------------------------------------------------------------------------- what a pass needs

def _level_counts(case):
    """Expected numbers of non-empty slices and of fibers per level below (order 3: [S, F2], order 4: [S, F2, F3])."""
    d, nnz = _dims(case), case["nnz"]
    n = np.full(d[0], nnz / d[0]) if case["alpha"] == 0 else _zipf_sizes(case).astype(np.float64)
    counts = [float(d[0] * -math.expm1(-nnz / d[0])) if case["alpha"] == 0 else float(np.count_nonzero(n))]
    n = n[n > 0]
    for level in range(1, len(d) - 1):
        prob = np.full(n.shape, case["fiber"] ** -(len(d) - 1.0 - level))
        cap = np.minimum(1.0, 0.9 * d[1] / n)
        head = np.minimum(np.full(n.shape, case["fiber"] ** -(len(d) - 2.0)), cap)
        prob = np.maximum(prob, head) if level > 1 else head
        counts.append(float((1 + (n - 1) * prob).sum()))
    return counts


def work(case):
    """Bytes and operations a pass cannot do without: B's compressed arrays, the rows of the dense operands that B refers
    to and the output once each; the multiply-adds of the cheaper association order."""
    d, nnz, expr = _dims(case), float(case["nnz"]), case["expr"]
    r = {k[5:]: float(v) for k, v in case.items() if k.startswith("rank_")}
    used = lambda dim: dim * -math.expm1(-nnz / dim)      # expected distinct coordinates of a mode  # noqa: E731
    shapes = _operand_shapes(case)
    if len(d) == 2:
        I, J = d
        rows = used(I) if case["alpha"] == 0 else float(np.count_nonzero(_powerlaw_degrees(case)))
        dense = sum(4.0 * s[1] * (rows if s[0] == I and n == 0 and expr.startswith("sddmm") else min(used(J), s[0])) for n, s in enumerate(shapes))
        flops = {
            "sddmm_spmm": lambda: nnz * 2 * (r["K"] + r["L"]),
            "sddmm_spmm_gemm": lambda: nnz * 2 * (r["K"] + r["L"]) + 2 * rows * r["L"] * r["M"],
            "spmm_gemm": lambda: min(2 * nnz * r["L"] + 2 * rows * r["L"] * r["M"], 2 * used(J) * r["L"] * r["M"] + 2 * nnz * r["M"]),
            "spmmh_gemm": lambda: min(3 * nnz * r["L"] + 2 * rows * r["L"] * r["M"], used(J) * (r["L"] + 2 * r["L"] * r["M"]) + 2 * nnz * r["M"]),
        }[expr]()
        out = 4.0 * I * (r["L"] if expr == "sddmm_spmm" else r["M"])
        return {"bytes": 8 * nnz + 4 * (I + 1) + dense + out, "flops": flops}
    counts = _level_counts(case)
    S, F2 = counts[0], counts[1]
    F3 = counts[2] if len(d) == 4 else nnz
    tensor = 8 * nnz + 8 * sum(counts)
    dense = sum(4.0 * s[1] * min(used(s[0]), s[0]) for s in shapes)
    flops, out = {
        "spttm_ttm3": lambda: (2 * nnz * r["M"] + 2 * F2 * r["L"] * r["M"], d[0] * r["L"] * r["M"]),
        "spttm_ttm4": lambda: (2 * (nnz * r["N"] + F3 * r["M"] * r["N"] + F2 * r["L"] * r["M"] * r["N"]), d[0] * r["L"] * r["M"] * r["N"]),
        "ttmc3": lambda: (2 * (nnz * r["N"] + F2 * r["M"] * r["N"] + S * r["L"] * r["M"] * r["N"]), r["L"] * r["M"] * r["N"]),
        "mttkrp_gemm": lambda: (2 * (nnz * r["R"] + F2 * r["R"] + S * r["R"] * r["M"]), d[0] * r["M"]),
        "spttm_spttm": lambda: (min(2 * nnz * r["L"] + 2 * F2 * r["L"] * r["M"], 2 * used(d[2]) * r["L"] * r["M"] + 2 * nnz * r["M"]), F2 * r["M"]),
    }[expr]()
    return {"bytes": tensor + dense + 4.0 * out, "flops": flops}


def tolerance(case):
    """fp32 inputs, sums and results: four times the distance from an fp64 evaluation on the device, the largest over the
    listed and ten drawn cases.  Chains whose sums all run in fp32 arithmetic were off by 3.0e-7 (largest element: 3.0e-5).
    Where a stage runs on tensor cores with every operand in two parts (TF32 parts in the per-slice contractions, BF16
    parts in the dense stage) it was 4.5e-6 (largest element: 3.0e-4, in sums that cancel)."""
    if case["expr"] in ("sddmm_spmm", "spmmh_gemm"):
        return {"rel": 1.2e-6, "max": 1.2e-4}
    return {"rel": 1.8e-5, "max": 1.2e-3}
