"""The calls that programs built on this package spend their time in, with inputs of their usual shapes.

A case names a call (``op``), the pattern of its sparse operand, its encoding, its sizes and the width of
positions and coordinates.  Patterns are those of ``paper_2202_04305_b200.inputs`` (uniform cells, entries
confined to a tenth of the rows, power-law row lengths, a band of full rows, Zipf-skewed tensors), drawn
here on the device because a case's inputs are made many times over.
"""
import math

import torch

from paper_2202_04305_b200 import binding as sp

# level types (0 dense, 1 compressed) and level -> dimension order
ENCODINGS = {
    "csr": ((0, 1), (0, 1)), "dcsr": ((1, 1), (0, 1)), "csc": ((0, 1), (1, 0)), "dcsc": ((1, 1), (1, 0)),
    "cdr": ((1, 0), (0, 1)),
    "csf": ((1, 1, 1), (0, 1, 2)), "dss": ((0, 1, 1), (0, 1, 2)), "csf_021": ((1, 1, 1), (0, 2, 1)),
}
ZIPF_ROWS, ZIPF_MODES = 1.5, 1.2
POWERLAW_MEAN = 16


def listed():
    return [
        # The smallest calls: the 1,024 x 1,024 matrix of density 0.01.  An iterative method multiplies with it
        # thousands of times, and an application that assembles small operators packs one per step.
        {"name": "spmv_csr_1k", "op": "spmv", "pattern": "uniform", "enc": "csr", "m": 1024, "n": 1024, "nnz": 10486, "bits": 32},
        {"name": "pack_csr_1k", "op": "pack", "pattern": "uniform", "enc": "csr", "m": 1024, "n": 1024, "nnz": 10486, "bits": 32},
        # Building storage from unsorted coordinates: a large, mostly empty matrix by columns, and a
        # skewed third-order tensor as compressed fibres.
        {"name": "pack_csc_5m", "op": "pack", "pattern": "confined", "enc": "csc", "m": 1 << 20, "n": 1 << 20, "nnz": 5000000, "bits": 32},
        {"name": "pack_csf_20m", "op": "pack", "pattern": "zipf3", "enc": "csf", "m": 16384, "nnz": 20000000, "bits": 32},
        # Storage to storage: a ragged matrix re-encoded from rows to columns with 64-bit positions and coordinates.
        {"name": "convert_csr_csc_odd", "op": "convert", "pattern": "uniform", "enc": "csr", "to": "csc", "m": 70001, "n": 50021,
         "nnz": 1500007, "bits": 64},
        # The row-band matrix whose first 1,000 rows are full: a product that streams 65.5 million entries.
        {"name": "spmv_csr_band", "op": "spmv", "pattern": "band", "enc": "csr", "m": 65536, "n": 65536, "nnz": 65536000, "bits": 32},
        # Blocks of vectors times a graph-like matrix of power-law rows.
        {"name": "spmm_csr_powerlaw", "op": "spmm", "pattern": "powerlaw", "enc": "csr", "m": 65536, "n": 65536,
         "nnz": POWERLAW_MEAN * 65536, "cols": 64, "bits": 32},
        # The large, mostly empty matrix by stored rows (forward) and by columns (the transposed direction).
        {"name": "spmm_dcsr_5m", "op": "spmm", "pattern": "confined", "enc": "dcsr", "m": 1 << 20, "n": 1 << 20, "nnz": 5000000,
         "cols": 32, "bits": 32},
        {"name": "spmm_csc_5m", "op": "spmm", "pattern": "confined", "enc": "csc", "m": 1 << 20, "n": 1 << 20, "nnz": 5000000,
         "cols": 32, "bits": 32},
        # Sampled products (gradients of factorisations): two million samples, 128 features.
        {"name": "sddmm_csr_2m", "op": "sddmm", "pattern": "uniform", "enc": "csr", "m": 131072, "n": 131072, "nnz": 2000000,
         "cols": 128, "bits": 32},
        # The step of a rank-32 CP decomposition over the skewed tensor.
        {"name": "mttkrp_csf_20m", "op": "mttkrp", "pattern": "zipf3", "enc": "csf", "m": 16384, "nnz": 20000000, "cols": 32, "bits": 32},
        # Sparse times sparse at density 0.01, the largest size of the paper's table.
        {"name": "spmspm_csr_8k", "op": "spmspm", "pattern": "uniform", "enc": "csr", "m": 8192, "n": 8192, "nnz": 671089, "bits": 32},
    ]


def _log(rng, lo, hi):
    """An integer spread over the logarithm of [lo, hi]."""
    return int(round(math.exp(rng.uniform(math.log(lo), math.log(hi)))))


def _draw_matrix(rng, biggest):
    """Pattern, sizes and entries of a matrix with at most about ``biggest`` entries."""
    pattern = rng.choice(["uniform", "confined", "powerlaw"])
    if pattern == "powerlaw":
        m = _log(rng, 1000, max(1000, biggest // POWERLAW_MEAN))
        return {"pattern": pattern, "m": m, "n": max(1000, int(m * rng.uniform(0.5, 2.0))), "nnz": POWERLAW_MEAN * m}
    nnz = _log(rng, 10000, biggest)
    # between about 5 and 100 entries a row on average, confined rows ten times that where they hold any
    m = max(1000, min(1 << 20, int(nnz / _log(rng, 5, 100))))
    n = max(1000, min(1 << 20, int(m * rng.uniform(0.5, 2.0))))
    return {"pattern": pattern, "m": m, "n": n, "nnz": min(nnz, m * n // 50)}


def draw(rng):
    op = rng.choice(["spmv", "spmv", "spmm", "spmm", "pack", "pack", "sddmm", "mttkrp", "spmspm", "convert"])
    bits = rng.choice([32, 32, 32, 64])
    if op == "mttkrp" or (op == "pack" and rng.random() < 0.4):
        c = {"op": op, "pattern": "zipf3", "enc": rng.choice(["csf", "dss", "csf_021"]), "m": _log(rng, 300, 16384), "bits": bits}
        c["nnz"] = min(_log(rng, 30000, 20000000), c["m"] ** 3 // 100)
        if op == "mttkrp":
            c["cols"] = rng.choice([8, 16, 17, 24, 32, 32, 48, 50, 64])
            c["nnz"] = min(c["nnz"], 20000000 * 32 // max(32, c["cols"]))
        return c
    if op == "spmspm":
        n, density = _log(rng, 1000, 8192), rng.uniform(0.002, 0.01)
        return {"op": op, "pattern": "uniform", "enc": "csr", "m": n, "n": n, "nnz": int(n * n * density), "bits": bits}
    if op == "spmv" and rng.random() < 0.25:
        m, n = _log(rng, 2000, 65536), _log(rng, 2000, 65536)
        rows = rng.randint(200, 1000)
        return {"op": op, "pattern": "band", "enc": rng.choice(["csr", "cdr"]), "m": m, "n": n, "nnz": rows * n, "bits": bits}
    c = dict(_draw_matrix(rng, {"sddmm": 2000000, "convert": 3000000}.get(op, 5000000)), op=op, bits=bits)
    if op == "convert":
        c["enc"], c["to"] = rng.choice([("csr", "csc"), ("csc", "csr"), ("csr", "dcsr"), ("dcsr", "dcsc")])
    else:
        c["enc"] = rng.choice(["csr", "csr", "dcsr", "csc"])
    if op == "spmm":
        c["cols"] = rng.choice([8, 16, 20, 32, 32, 33, 50, 64, 64, 100, 128])
        c["nnz"] = min(c["nnz"], 5000000 * 32 // max(32, c["cols"]))
        if c["pattern"] == "powerlaw":
            c["m"] = min(c["m"], c["nnz"] // POWERLAW_MEAN)
            c["nnz"] = POWERLAW_MEAN * c["m"]
    elif op == "sddmm":
        c["cols"] = rng.choice([16, 32, 50, 64, 96, 100, 128, 128])
    return c


# ----------------------------------------------------------------------------------------------- inputs

def _rand(g, n):
    return torch.rand(n, dtype=torch.float64, device="cuda", generator=g)


def _values(g, *shape):
    """Uniform in [-1, 1)."""
    return _rand(g, shape).mul_(2.0).sub_(1.0)


def _distinct(g, count, total_draw):
    """``count`` distinct keys out of what ``total_draw(k)`` draws."""
    k = int(count * 1.1) + 64
    keys = torch.unique(total_draw(k))
    while keys.numel() < count:
        keys = torch.unique(torch.cat([keys, total_draw(k)]))
    return keys[torch.randperm(keys.numel(), device="cuda", generator=g)[:count]]


def _row_lengths(g, m):
    """Row lengths with P(len = k) ~ k^-1.5 up to the smallest cut whose mean is at least 16."""
    k = torch.arange(1, 4097, dtype=torch.float64)      # on the host: sums in one order, the same every time
    w = k ** -ZIPF_ROWS
    mean = torch.cumsum(k * w, 0) / torch.cumsum(w, 0)
    kmax = int((mean < POWERLAW_MEAN).sum()) + 1
    cdf = torch.cumsum(w[:kmax], 0).cuda()
    return torch.searchsorted(cdf, _rand(g, m) * cdf[-1]).clamp_(max=kmax - 1) + 1


def _zipf(g, cdf, n):
    return torch.searchsorted(cdf, _rand(g, n) * cdf[-1]).clamp_(max=cdf.numel() - 1)


def _pattern(case, g):
    """One int64 coordinate array per dimension, entries distinct and in no particular order."""
    m, nnz = case["m"], case["nnz"]
    if case["pattern"] == "zipf3":
        cdf = torch.cumsum(torch.arange(1, m + 1, dtype=torch.float64) ** -ZIPF_MODES, 0).cuda()
        keys = _distinct(g, nnz, lambda k: (_zipf(g, cdf, k) * m + _zipf(g, cdf, k)) * m + _zipf(g, cdf, k))
        return [keys // (m * m), keys // m % m, keys % m]
    n = case["n"]
    if case["pattern"] == "band":
        keys = torch.randperm(nnz, device="cuda", generator=g)
    elif case["pattern"] == "confined":
        rows = torch.randperm(m, device="cuda", generator=g)[: max(1, -(-m // 10))]
        keys = _distinct(g, nnz, lambda k: rows[torch.randint(rows.numel(), (k,), device="cuda", generator=g)] * n
                         + torch.randint(n, (k,), device="cuda", generator=g))
    elif case["pattern"] == "powerlaw":
        lens = _row_lengths(g, m).clamp_(max=n)
        rows = torch.repeat_interleave(torch.arange(m, device="cuda"), lens)
        keys = torch.unique(rows * n + torch.randint(n, rows.shape, device="cuda", generator=g))
    else:
        keys = _distinct(g, nnz, lambda k: torch.randint(m * n, (k,), device="cuda", generator=g))
    return [keys // n, keys % n]


def _dims(case):
    return (case["m"],) * 3 if case["pattern"] == "zipf3" else (case["m"], case["n"])


def _coo(case, g, relabel, which=0):
    """Coordinates of the case's width and f64 values, in random order: what an application hands to sp_pack.

    The pattern is drawn once for the case and its dimensions are relabelled at random for every seed, so
    that inputs of different seeds differ in all entries and agree in how many rows, fibres and results
    they have.  A band's rows stay the first ones."""
    fixed = torch.Generator(device="cuda")
    fixed.manual_seed(1234 + which)
    coords = _pattern(case, fixed)
    if case["pattern"] != "band":
        coords = [p[c] for p, c in zip(relabel, coords)]
    order = torch.randperm(coords[0].numel(), device="cuda", generator=g)
    kind = torch.int32 if case["bits"] == 32 else torch.int64
    return [c[order].to(kind) for c in coords], _values(g, order.numel())


def prepare(case, seed):
    g = torch.Generator(device="cuda")
    g.manual_seed(seed)
    dims, bits, op = _dims(case), case["bits"], case["op"]
    lt, od = ENCODINGS[case["enc"]]
    relabel = [torch.randperm(d, device="cuda", generator=g) for d in dims]
    coords, vals = _coo(case, g, relabel)
    s = {"op": op, "dims": dims, "bits": bits, "lt": lt, "od": od}
    if op == "pack":
        s.update(coords=coords, vals=vals)
        return s
    s["A"] = sp.sp_pack(dims, coords, vals, lt, od, bits, bits)      # the matrix a program keeps
    cols = case.get("cols")
    # dense operands and, as an iterative program does, an output buffer kept from call to call
    if op == "spmv":
        s.update(x=_values(g, dims[1]), y=torch.empty(dims[0], dtype=torch.float64, device="cuda"))
    elif op == "spmm":
        s.update(B=_values(g, dims[1], cols), C=torch.empty((dims[0], cols), dtype=torch.float64, device="cuda"))
    elif op == "sddmm":
        s.update(L=_values(g, dims[0], cols), R=_values(g, cols, dims[1]), xv=torch.empty(s["A"].nval, dtype=torch.float64, device="cuda"))
    elif op == "mttkrp":
        s.update(B=_values(g, dims[1], cols), C=_values(g, dims[2], cols), M=torch.empty((dims[0], cols), dtype=torch.float64, device="cuda"))
    elif op == "spmspm":
        coords, vals = _coo(case, g, [relabel[1], relabel[0]], 1)
        s["B"] = sp.sp_pack(dims, coords, vals, lt, od, bits, bits)
    elif op == "convert":
        s["to"] = ENCODINGS[case["to"]]
    return s


def _arrays(t):
    """Everything a handle stores."""
    out = {"values": t.values()}
    for level, kind in enumerate(t.lt):
        if kind:
            out[f"pos{level}"], out[f"crd{level}"] = t.positions(level), t.coordinates(level)
    return out


def run(s):
    op, bits = s["op"], s["bits"]
    if op == "spmv":
        return sp.sp_spmv(s["A"], s["x"], s["y"])
    if op == "spmm":
        return sp.sp_spmm(s["A"], s["B"], s["C"])
    if op == "sddmm":
        return sp.sp_sddmm(s["A"], s["L"], s["R"], s["xv"])
    if op == "mttkrp":
        return sp.sp_mttkrp(s["A"], s["B"], s["C"], s["M"])
    if op == "pack":
        return _arrays(sp.sp_pack(s["dims"], s["coords"], s["vals"], s["lt"], s["od"], bits, bits))
    if op == "convert":
        return _arrays(sp.sp_convert(s["A"], s["to"][0], s["to"][1], bits, bits))
    return _arrays(sp.sp_spmspm(s["A"], s["B"], bits, bits))


# --------------------------------------------------------------------------------------- work, tolerance

def _stored_bytes(case, enc):
    """Bytes of the case's matrix or tensor in an encoding; levels whose size depends on the data (stored
    rows, fibres) are counted where the pattern fixes them."""
    nnz, w = case["nnz"], case["bits"] // 8
    if case["pattern"] == "zipf3":
        return nnz * (8 + w)                      # slices and fibres not counted
    lt, od = ENCODINGS[enc]
    outer = (case["m"], case["n"])[od[0]]
    if enc == "cdr":
        return nnz * 8
    if lt[0] == 1:
        rows = min(outer, nnz)
        if case["pattern"] == "confined" and od[0] == 0:
            rows = min(rows, -(-case["m"] // 10))
        if case["pattern"] == "band" and od[0] == 0:
            rows = nnz // case["n"]
        return nnz * (8 + w) + rows * 2 * w
    return nnz * (8 + w) + (outer + 1) * w


def work(case):
    op, nnz, m = case["op"], case["nnz"], case["m"]
    cols = case.get("cols", 1)
    rank = 3 if case["pattern"] == "zipf3" else 2
    stored = _stored_bytes(case, case["enc"])
    if op == "pack":
        return {"bytes": nnz * (8 + rank * case["bits"] // 8) + stored, "flops": 0}
    if op == "convert":
        return {"bytes": stored + _stored_bytes(case, case["to"]), "flops": 0}
    if op == "mttkrp":
        return {"bytes": stored + 3 * m * cols * 8, "flops": 2 * nnz * cols}
    n = case["n"]
    if op == "spmspm":
        products = nnz * nnz / m
        filled = m * n * -math.expm1(-products / (m * n))          # uniform operands
        return {"bytes": 2 * stored + filled * (8 + case["bits"] // 8) + (m + 1) * case["bits"] // 8, "flops": 2 * products}
    if op == "sddmm":
        return {"bytes": stored + (m + n) * cols * 8 + nnz * 8, "flops": 2 * nnz * cols + nnz}
    return {"bytes": stored + (m + n) * cols * 8, "flops": 2 * nnz * cols}     # spmv, spmm


def tolerance(case):
    # Packing moves numbers: structure and values come out bit for bit.
    if case["op"] in ("pack", "convert"):
        return "exact"
    # f64 sums in another order, about four times what the products' sums in random order differ by: 1e-15
    # and 1.5e-14 at most for matrices; 8.4e-15 and 1.3e-13 where rows have 65,536 terms; 1.6e-14 and 4.3e-13
    # for tensors, whose longest sums have millions.
    if case["op"] == "mttkrp":
        return {"rel": 6e-14, "max": 2e-12}
    if case["pattern"] == "band":
        return {"rel": 3.4e-14, "max": 5e-13}
    return {"rel": 4e-15, "max": 6e-14}
