"""The work that users of this library have it do, as cases that can be timed: what a case's inputs are, one pass
through the public entry points, the bytes and operations that pass cannot do without, and how far two correct
implementations may differ.

Sizes are those of the benchmark's five workloads (`synth/configs.py`), of the second workload shape (the
hypersparse matrix), and generic smaller ones in between; index laws follow the workloads too. Widths of the dense
operands are the ones in use: powers of two, and ranks and feature counts that are none (10, 25, 50, ...).
"""
import math

import numpy as np
import torch

import paper_2102_05187_b200 as comet
from paper_2102_05187_b200 import CN, CU, D, S

ZIPF_S, ZIPF_CAP = 1.8, 10_000                 # row lengths of the matrices with a power law
FORMATS = {"csr": (D, CU), "dcsr": (CU, CU), "coo": (CN, S), "csf": (CU, CU, CU), "coo3": (CN, S, S)}


def listed():
    return [
        # the smallest product a solver calls in a loop: launches and latency are what it costs
        {"name": "spmv-small", "op": "spmv", "format": "csr", "dtype": "f64", "dims": "4096x4096", "law": "uniform", "nnz": 65_536},
        # a power-law graph's matrix times a vector that fits no shared memory (PageRank-like iteration)
        {"name": "spmv-graph", "op": "spmv", "format": "csr", "dtype": "f64", "dims": "1048576x1048576", "law": "zipf", "nnz": 0},
        # feature aggregation over a mid-sized graph: fp32, a width that is no power of two
        {"name": "spmm-features", "op": "spmm", "format": "csr", "dtype": "f32", "dims": "170003x170003", "law": "zipf", "nnz": 0, "R": 50},
        # the benchmark's SpMM: power-law rows, B four times as large as the L2 cache
        {"name": "spmm-graph", "op": "spmm", "format": "csr", "dtype": "f64", "dims": "1048576x1048576", "law": "zipf", "nnz": 0, "R": 64},
        # hypersparse matrix in DCSR (94 % of the rows are empty), a few right-hand sides
        {"name": "spmm-hypersparse", "op": "spmm", "format": "dcsr", "dtype": "f64", "dims": "67108864x1048576", "law": "uniform", "nnz": 4_194_304, "R": 8},
        # tensor times vector, power-law slices, sparse CSR result
        {"name": "ttv-slices", "op": "ttv", "format": "csf", "dtype": "f64", "dims": "20000x20000x20000", "law": "slices", "nnz": 50_000_000},
        # tensor times matrix, short fibers (mean 8), as in Tucker / HOOI sweeps
        {"name": "ttm-fibers", "op": "ttm", "format": "csf", "dtype": "f64", "dims": "100000x50000x20000", "law": "fibers", "nnz": 30_000_000, "R": 16},
        # mode-1 MTTKRP of a large power-law tensor kept as sorted coordinates
        {"name": "mttkrp-coo", "op": "mttkrp", "format": "coo3", "dtype": "f64", "dims": "1000000x500000x200000", "law": "power", "nnz": 100_000_000, "R": 32, "mode": 0},
        # the three MTTKRPs of one CP-ALS iteration on one packed tensor: the largest piece of work
        {"name": "cp-sweep", "op": "sweep", "format": "csf", "dtype": "f64", "dims": "1000000x500000x200000", "law": "power", "nnz": 100_000_000, "R": 32},
        # the same on an ordinary tensor in fp32, with a rank that is no power of two
        {"name": "cp-sweep-mid", "op": "sweep", "format": "csf", "dtype": "f32", "dims": "40009x30011x20021", "law": "power", "nnz": 3_000_000, "R": 25},
        # conversion of the benchmark's matrix from shuffled coordinates to CSR
        {"name": "pack-csr", "op": "pack", "format": "csr", "dtype": "f64", "dims": "1048576x1048576", "law": "zipf", "nnz": 0},
        # a small tensor that has just arrived: pack it, contract it once
        {"name": "fresh-small", "op": "fresh", "format": "csf", "dtype": "f32", "dims": "1203x997x801", "law": "fibers", "nnz": 60_000, "R": 16},
    ]


def _log_uniform(rng, lo, hi):
    return int(round(math.exp(rng.uniform(math.log(lo), math.log(hi)))))


def draw(rng):
    op = rng.choice(["spmv", "spmm", "spmm", "ttv", "ttm", "mttkrp", "sweep", "pack", "fresh"])
    case = {"op": op, "dtype": rng.choice(["f64", "f64", "f32"])}
    matrix = op in ("spmv", "spmm") or (op == "pack" and rng.random() < 0.5)
    nnz = _log_uniform(rng, 20_000, 200_000 if op == "fresh" else 30_000_000)
    if matrix:
        case["format"] = rng.choice(["csr", "csr", "csr", "dcsr", "coo"])
        case["law"] = rng.choice(["zipf", "uniform"])
        if case["law"] == "zipf":
            rows = max(1000, nnz // 20)
            case["nnz"] = 0
        else:
            rows = max(500, int(nnz / rng.choice([3, 8, 16, 40, 100])))
            case["nnz"] = nnz
        cols = max(500, int(rows * rng.uniform(0.3, 2.0)))
        case["dims"] = "%dx%d" % (rows, cols)
    else:
        case["format"] = "csf" if op == "fresh" else rng.choice(["csf", "csf", "coo3"])
        case["law"] = rng.choice(["fibers", "power"] if op == "fresh" else ["slices", "fibers", "power"])
        case["nnz"] = nnz
        side = max(200.0, (nnz * 1e3) ** (1 / 3) * rng.uniform(1.0, 8.0))
        if case["law"] == "slices":                # the largest slice holds more than half of the entries
            side = max(side, (16.0 * nnz) ** 0.5)
        case["dims"] = "x".join(str(int(side * rng.uniform(0.6, 1.6))) for _ in range(3))
    if op in ("spmm", "ttm", "mttkrp", "sweep", "fresh"):
        case["R"] = rng.choice([rng.choice([4, 8, 16, 32, 64]), rng.choice([10, 20, 50, 100]), rng.randint(1, 100)])
    if op == "mttkrp":
        case["mode"] = rng.randint(0, 2)
    return case


# ------------------------------------------------------------------------------------------------- inputs

def _dims(case):
    return tuple(int(d) for d in case["dims"].split("x"))


def _uniform(n, bound, gen):
    return torch.randint(0, bound, (n,), generator=gen, device="cuda", dtype=torch.int64)


def _distinct(keys, n, gen):
    """Up to n of the distinct keys (all of them for n = 0), shuffled."""
    keys = torch.unique(keys)
    order = torch.randperm(keys.numel(), generator=gen, device="cuda")
    return keys[order[:n]] if n else keys[order]


def _zipf_lengths(rows, cap, gen):
    k = np.arange(1, cap, dtype=np.float64)
    zeta = float(np.sum(np.arange(1, 200_000, dtype=np.float64) ** -ZIPF_S)) + 200_000.0 ** (1 - ZIPF_S) / (ZIPF_S - 1)
    cdf = torch.from_numpy(np.cumsum(k ** -ZIPF_S) / zeta).cuda()
    u = torch.rand(rows, generator=gen, device="cuda", dtype=torch.float64)
    return torch.searchsorted(cdf, u, right=True) + 1          # the tail beyond the cap is lumped on it


def _zipf_cap(rows, cols):
    return max(1, min(ZIPF_CAP, cols // 4))


def _nnz(case):
    """Entries of a case (of the power-law matrices: the expected number; draws that repeat a cell are dropped)."""
    if case["law"] != "zipf":
        return case["nnz"]
    rows, cols = _dims(case)
    cap = _zipf_cap(rows, cols)
    k = np.arange(1, cap, dtype=np.float64)
    zeta = float(np.sum(np.arange(1, 200_000, dtype=np.float64) ** -ZIPF_S)) + 200_000.0 ** (1 - ZIPF_S) / (ZIPF_S - 1)
    p = k ** -ZIPF_S / zeta
    return int(rows * (float(np.sum(k * p)) + cap * (1.0 - float(np.sum(p)))))


def _cells(case, gen):
    """Distinct cells of the tensor as row-major linear numbers, shuffled."""
    dims, law, n = _dims(case), case["law"], case["nnz"]
    total = math.prod(dims)
    if law == "zipf":                              # row lengths min(Zipf(1.8), cap), uniform columns
        rows, cols = dims
        row = torch.repeat_interleave(torch.arange(rows, device="cuda"), _zipf_lengths(rows, _zipf_cap(rows, cols), gen))
        return _distinct(row * cols + _uniform(row.numel(), cols, gen), 0, gen)
    if law == "uniform":
        return _distinct(_uniform(int(n * 1.02) + 64, total, gen), n, gen)
    if law == "slices":                            # slice sizes ~ rank^-2, uniform inside a slice
        w = np.arange(1, dims[0] + 1, dtype=np.float64) ** -2.0
        cdf = torch.from_numpy(np.cumsum(w) / np.sum(w)).cuda()
        u = torch.rand(int(n * 1.06) + 64, generator=gen, device="cuda", dtype=torch.float64)
        rank = torch.searchsorted(cdf, u, right=True).clamp_(max=dims[0] - 1)
        i = torch.randperm(dims[0], generator=gen, device="cuda")[rank]
        return _distinct(i * (dims[1] * dims[2]) + _uniform(i.numel(), dims[1] * dims[2], gen), n, gen)
    if law == "fibers":                            # distinct uniform (i, j), fiber lengths geometric with mean 8
        fibers = max(1, n // 8)
        ij = _distinct(_uniform(int(fibers * 1.02) + 64, dims[0] * dims[1], gen), fibers, gen)
        u = torch.rand(ij.numel(), generator=gen, device="cuda", dtype=torch.float64)
        length = (torch.log1p(-u) / math.log1p(-1 / 8)).long().clamp_(max=dims[2] // 4) + 1
        ij = torch.repeat_interleave(ij, length)
        return _distinct(ij * dims[2] + _uniform(ij.numel(), dims[2], gen), 0, gen)
    assert law == "power"                          # per-mode index frequencies ~ (k + 100)^-1.5, relabelled
    m = int(n * 1.08) + 4096
    key = torch.zeros(m, dtype=torch.int64, device="cuda")
    for d in dims:
        u = torch.rand(m, generator=gen, device="cuda", dtype=torch.float64)
        lo, hi = 100.0 ** -0.5, (d + 100.0) ** -0.5
        k = ((lo - u * (lo - hi)) ** -2 - 100.0).long().clamp_(0, d - 1)
        key = key * d + torch.randperm(d, generator=gen, device="cuda")[k]
    return _distinct(key, n, gen)


def _coordinates(case, gen):
    """Shuffled coordinates. The pattern is the case's own; the seed renumbers the indices of every mode and shuffles
    the entries, so that other seeds have other entries and yet as many entries, rows and fibers (the sizes of sparse
    results)."""
    pattern = torch.Generator(device="cuda")
    pattern.manual_seed(20210205)
    cells = _cells(case, pattern)
    cells = cells[torch.randperm(cells.numel(), generator=gen, device="cuda")]
    coords = []
    for d in reversed(_dims(case)):
        number = torch.randperm(d, generator=gen, device="cuda", dtype=torch.int32)
        coords.append(number[cells % d])
        cells = cells // d
    coords.reverse()
    return coords


def _dense(shape, gen, dtype):
    return torch.rand(shape, generator=gen, device="cuda", dtype=dtype) * 2 - 1


def prepare(case, seed):
    gen = torch.Generator(device="cuda")
    gen.manual_seed(int(seed))
    dims, op = _dims(case), case["op"]
    dtype = torch.float32 if case["dtype"] == "f32" else torch.float64
    coords = _coordinates(case, gen)
    val = _dense((coords[0].numel(),), gen, dtype)
    state = {"op": op, "dims": dims, "attr": FORMATS[case["format"]], "order": tuple(range(len(dims)))}
    R = case.get("R", 1)
    if op in ("pack", "fresh"):                    # the coordinates are what the program holds
        state["coords"], state["val"] = coords, val
    else:                                          # the packed tensor is
        state["A"] = comet.pack(coords, val, dims, state["order"], state["attr"])
    if op == "spmv":
        state["x"] = _dense((dims[1],), gen, dtype)
    elif op == "spmm":
        state["B"] = _dense((dims[1], R), gen, dtype)
    elif op == "ttv":
        state["v"] = _dense((dims[2],), gen, dtype)
        state["Y"] = comet.ttv_symbolic(state["A"], 2)
    elif op in ("ttm", "fresh"):
        state["U"] = _dense((dims[2], R), gen, dtype)
        if op == "ttm":
            state["Y"] = comet.ttm_symbolic(state["A"], 2, R)
    elif op in ("mttkrp", "sweep"):
        state["F"] = [_dense((d, R), gen, dtype) for d in dims]
        state["modes"] = [case["mode"]] if op == "mttkrp" else [0, 1, 2]
    return state


def run(state):
    op = state["op"]
    if op == "spmv":
        return comet.spmv(state["A"], state["x"])
    if op == "spmm":
        return comet.spmm(state["A"], state["B"])
    if op == "ttv":
        return comet.ttv(state["A"], 2, state["v"], state["Y"]).val
    if op == "ttm":
        return comet.ttm(state["A"], 2, state["U"], state["Y"]).val
    if op in ("mttkrp", "sweep"):
        return [comet.mttkrp(state["A"], m, state["F"]) for m in state["modes"]]
    A = comet.pack(state["coords"], state["val"], state["dims"], state["order"], state["attr"])
    if op == "fresh":
        Y = comet.ttm(A, 2, state["U"])
        return [Y.crd(0), Y.pos(1), Y.crd(1), Y.val]
    out = [A.val]
    for level in range(len(state["attr"])):
        out += [A.pos(level), A.crd(level)]
    return out


# ------------------------------------------------------------------------------------------------- bounds

def work(case):
    """Index 4 bytes, value 4 or 8; every input once, every output once; a multiply and an add per term."""
    dims, op, n = _dims(case), case["op"], _nnz(case)
    v, R = 4 if case["dtype"] == "f32" else 8, case.get("R", 1)
    modes = len(dims)
    if case["law"] == "fibers":
        fibers = max(1, n // 8)
    else:                                          # distinct (i, j): at most one per entry
        fibers = min(n, dims[0] * dims[1]) if modes == 3 else 0
        if case["law"] == "slices":
            fibers = min(fibers, n // 36 + 1)
        elif case["law"] == "power":
            fibers = min(fibers, n * 3 // 10 + 1)
    stored = {"csr": 4 * (n + dims[0]), "dcsr": 4 * (n + 2 * min(n, dims[0])), "coo": 8 * n, "coo3": 12 * n,
              "csf": 4 * n + 8 * fibers}[case["format"]] + v * n
    if op == "pack":
        return {"bytes": (4 * modes + v) * n + stored, "flops": 0}
    if op == "fresh":
        return {"bytes": (12 + v) * n + v * R * (dims[2] + fibers), "flops": 2 * n * R}
    if op == "spmv":
        return {"bytes": stored + v * (min(n, dims[1]) + dims[0]), "flops": 2 * n}
    if op == "spmm":
        return {"bytes": stored + v * R * (min(n, dims[1]) + dims[0]), "flops": 2 * n * R}
    if op == "ttv":
        return {"bytes": stored + v * (dims[2] + fibers), "flops": 2 * n}
    if op == "ttm":
        return {"bytes": stored + v * R * (dims[2] + fibers), "flops": 2 * n * R}
    one = stored + v * R * sum(min(n, d) for d in dims)
    return {"bytes": one * (3 if op == "sweep" else 1), "flops": 3 * n * R * (3 if op == "sweep" else 1)}


def tolerance(case):
    """Packing copies values: exact. Sums are formed in double whatever the type and rounded when they are stored (a
    row that spans several tiles once more). Measured against the same sums in double in another order, over all cases
    and some drawn ones: fp64 up to rel 5.5e-15, max 7.8e-13 (rows of half a million terms), fp32 up to rel 2.8e-8,
    max 5.5e-7. Four times that is stated."""
    if case["op"] == "pack":
        return "exact"
    if case["dtype"] == "f32":
        return {"rel": 1.2e-7, "max": 2.2e-6}
    return {"rel": 2.2e-14, "max": 3.2e-12}
