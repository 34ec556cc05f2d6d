"""The work that users of this library have it do, as cases that can be timed.

A case names one call sequence through the public entry points (`op`), the code (`m_lo`, `m_hi`), the sizes and the options:

  gemv / gemv_sorted        one fused dequantization + matrix-vector product, stored stream / load-time sorted layout
  gemv_multi                several products in one launch (sorted layout): the linear layers of a decode step
  gemv_sg / gemv_sorted_sg  the shape-gain form (gain codebook + row scales)
  gemm / gemm_sorted        the small-batch product, stored stream / sorted layout
  dequant                   index stream -> bf16 matrix
  encode                    real vectors -> points, indices and the stored stream

Inputs follow the repository's recipe for synthetic layers: indices uniform over the code, gains fp16(|z| * 0.02),
activations N(0, 1) in bf16, Gaussian vectors for the encoder (at lattice scale 2.5 where the ball is the code).
"""
from __future__ import annotations

import functools

import torch

import paper_2603_11021_b200 as P

LATTICE_SCALE = 2.5                                   # Gaussian source -> integer coordinates: about 89 % of it lies inside the ball of shells 2..13
CHI24_LEVELS = {0: [4.8484], 1: [4.3157, 5.4413], 2: [3.8436, 4.6049, 5.2679, 6.0774]}   # gain codebooks matched to |N(0, I_24)|
MAX_WEIGHTS = 28672 * 8192                            # no drawn product is larger than the largest listed one
MAX_ENCODE = {"euclidean": 4096 * 4096 // 24, "angular": 1024 * 4096 // 24}


def listed():
    return [
        # The smallest call: one projection of a small model at batch 1, where the launch and its fixed costs are what is paid.
        dict(name="gemv_sorted_512x1024", op="gemv_sorted", m_lo=2, m_hi=13, rows=512, cols=1024, y="bf16"),
        # One token through one matrix straight from the stored stream (no load-time rearrangement), binary32 result.
        dict(name="gemv_11008x4096", op="gemv", m_lo=2, m_hi=13, rows=11008, cols=4096, y="f32"),
        # The headline workload: the three layer shapes of a 7B decoder step in one launch, sorted layout.
        dict(name="gemv_multi_7b", op="gemv_multi", m_lo=2, m_hi=13, shapes="4096x4096 11008x4096 4096x11008", y="bf16"),
        # Shape-gain form at the same rate (47 + 1 bits), long rows that end inside a block (11008 = 458 * 24 + 16).
        dict(name="gemv_sorted_sg_4096x11008", op="gemv_sorted_sg", m_lo=2, m_hi=12, gain_bits=1, rows=4096, cols=11008, y="f32"),
        # The 3-bit code (72-bit indices), one token from the stored stream.
        dict(name="gemv_72_4096x4096", op="gemv", m_lo=2, m_hi=53, rows=4096, cols=4096, y="bf16"),
        # A batch of 16 requests, stored stream, the square layer of a 70B-class decoder.
        dict(name="gemm_8192x8192_b16", op="gemm", m_lo=2, m_hi=13, rows=8192, cols=8192, batch=16),
        # The largest product: its widest layer at the largest batch, sorted layout.
        dict(name="gemm_sorted_28672x8192_b64", op="gemm_sorted", m_lo=2, m_hi=13, rows=28672, cols=8192, batch=64),
        # The 3-bit code at a batch that is no multiple of the tile, sorted layout.
        dict(name="gemm_sorted_72_8192x8192_b21", op="gemm_sorted", m_lo=2, m_hi=53, rows=8192, cols=8192, batch=21),
        # Bulk dequantization of a square layer (blocks over the flattened matrix), e.g. ahead of a prefill in bf16.
        dict(name="dequant_4096x4096", op="dequant", m_lo=2, m_hi=13, rows=4096, cols=4096, layout="flat"),
        # The same for the 3-bit code, row by row, with a width that is no multiple of the block.
        dict(name="dequant_72_1376x11004", op="dequant", m_lo=2, m_hi=53, rows=1376, cols=11004, layout="rowwise"),
        # Quantizing one 4096 x 4096 matrix with spherical shaping: nearest points, their indices, the stored stream.
        dict(name="encode_euclidean_4096x4096", op="encode", m_lo=2, m_hi=13, blocks=4096 * 4096 // 24, metric="euclidean", gain_bits=0),
        # Quantizing a 1024 x 4096 matrix in the shape-gain form: best direction on the code, one gain bit beside it.
        dict(name="encode_angular_1024x4096", op="encode", m_lo=2, m_hi=12, blocks=1024 * 4096 // 24, metric="angular", gain_bits=1),
    ]


def _log_int(rng, lo, hi):
    return int(round(lo * (hi / lo) ** rng.random()))


def _sizes(rng, op):
    """Rows and columns of a layer: spread over the logarithm, half of them ragged."""
    while True:
        rows, cols = _log_int(rng, 256, 28672), _log_int(rng, 480, 14336)
        if rng.random() < 0.5:
            rows, cols = max(rows // 128, 2) * 128, max(cols // 128, 4) * 128
        if op.startswith("gemm"):
            cols = cols // 8 * 8                      # the batched products take 16-byte rows of X
        if rows * cols <= MAX_WEIGHTS:
            return rows, cols


def draw(rng):
    op = rng.choice(["gemv", "gemv_sorted", "gemv_multi", "gemv_sg", "gemv_sorted_sg", "gemm", "gemm_sorted", "dequant", "encode"])
    if op == "encode":
        metric = rng.choice(["euclidean", "angular"])
        m_hi, bits = (13, 0) if metric == "euclidean" else rng.choice([(12, 1), (11, 2), (13, 0)])
        return dict(op=op, m_lo=2, m_hi=m_hi, blocks=_log_int(rng, 2000, MAX_ENCODE[metric]), metric=metric, gain_bits=bits)
    if op == "gemv_multi":
        # matrices that read the same input (q, k, v; gate, up), or the unrelated layers of a step
        cols = _log_int(rng, 1024, 8192)
        shapes = []
        for _ in range(rng.randint(2, 4)):
            shapes.append("%dx%d" % (_log_int(rng, 1024, 14336), cols if rng.random() < 0.7 else _log_int(rng, 1024, 11008)))
        return dict(op=op, m_lo=2, m_hi=13, shapes=" ".join(shapes), y=rng.choice(["f32", "bf16"]))
    rows, cols = _sizes(rng, op)
    if op in ("gemv_sg", "gemv_sorted_sg"):
        m_hi, bits = rng.choice([(12, 1), (11, 2), (13, 0)])
        return dict(op=op, m_lo=2, m_hi=m_hi, gain_bits=bits, rows=rows, cols=cols, y=rng.choice(["f32", "bf16"]))
    # the 2-bit code mostly, the 3-bit code, and the single shell of 24-bit indices
    m_lo, m_hi = rng.choice([(2, 13), (2, 13), (2, 13), (2, 53), (2, 53), (3, 3)])
    case = dict(op=op, m_lo=m_lo, m_hi=m_hi, rows=rows, cols=cols)
    if op == "dequant":
        return dict(case, layout=rng.choice(["flat", "rowwise"]))
    if op.startswith("gemm"):
        return dict(case, batch=rng.choice([rng.randint(1, 64), 16, 32, 64]))
    if op == "gemv_sorted" and m_hi == 53:
        case["cols"] = cols // 8 * 8                  # this code's sorted product takes 16-byte aligned rows of x
    return dict(case, y=rng.choice(["f32", "bf16"]))


@functools.lru_cache(maxsize=None)
def _context(m_lo, m_hi):
    """A program builds the tables of its code once."""
    return P.Context(m_lo, m_hi, device=0)


def _blocks_per_row(cols):
    return (cols + 23) // 24


def _stream(ctx, nblocks, g, gain_bits=0):
    """A stored stream of uniform indices (and uniform gain indices)."""
    if ctx.index_bits <= 64:
        index = torch.randint(0, ctx.num_points, (nblocks,), generator=g, dtype=torch.int64, device="cuda")
        k = torch.randint(0, 1 << gain_bits, (nblocks,), generator=g, dtype=torch.uint8, device="cuda") if gain_bits else None
        return P.llvq_pack_fields(ctx, index, k, gain_bits)
    assert ctx.index_bits == 72
    low = torch.randint(0, 256, (nblocks, 8), generator=g, dtype=torch.uint8, device="cuda")
    high = torch.randint(0, ctx.num_points >> 64, (nblocks, 1), generator=g, dtype=torch.uint8, device="cuda")
    out = torch.zeros(ctx.index_bytes(nblocks), dtype=torch.uint8, device="cuda")
    out[:nblocks * 9] = torch.cat([low, high], dim=1).reshape(-1)
    return out


def _gains(nblocks, g):
    return (torch.randn(nblocks, generator=g, device="cuda").abs() * 0.02).half()


def _y_dtype(case):
    return torch.float32 if case["y"] == "f32" else torch.bfloat16


def _shapes(case):
    return [tuple(int(v) for v in s.split("x")) for s in case["shapes"].split()]


def prepare(case, seed):
    g = torch.Generator(device="cuda")
    g.manual_seed(seed)
    ctx, op = _context(case["m_lo"], case["m_hi"]), case["op"]
    s = {"case": case, "ctx": ctx}
    if op == "encode":
        v = torch.randn((case["blocks"], 24), generator=g, device="cuda")
        if case["metric"] == "euclidean":
            v *= LATTICE_SCALE
        s["v"], s["k"] = v, None
        if case["gain_bits"]:
            levels = torch.tensor(CHI24_LEVELS[case["gain_bits"]], device="cuda")
            s["k"] = (v.norm(dim=1)[:, None] - levels[None, :]).abs().argmin(dim=1).to(torch.uint8)
        return s
    if op == "gemv_multi":
        xs, s["mats"] = {}, []
        for rows, cols in _shapes(case):
            nblocks = rows * _blocks_per_row(cols)
            weights = P.llvq_sort_blocks(ctx, _stream(ctx, nblocks, g), rows, cols)
            if cols not in xs:
                xs[cols] = torch.randn(cols, generator=g, device="cuda").bfloat16()
            y = torch.empty(rows, dtype=_y_dtype(case), device="cuda")
            s["mats"].append((weights, _gains(nblocks, g), rows, cols, xs[cols], y))
        return s
    rows, cols = case["rows"], case["cols"]
    flat = case.get("layout") == "flat"
    nblocks = (rows * cols + 23) // 24 if flat else rows * _blocks_per_row(cols)
    if op in ("gemv_sg", "gemv_sorted_sg"):
        bits = case["gain_bits"]
        s["weights"] = _stream(ctx, nblocks, g, bits)
        s["codebook"] = torch.tensor(CHI24_LEVELS[bits], device="cuda")
        s["scale"] = 0.02 * (1 + 0.1 * torch.randn(rows, generator=g, device="cuda").clamp(-3, 3))
        if op == "gemv_sorted_sg":
            s["weights"] = P.llvq_sort_blocks_sg(ctx, s["weights"], bits, rows, cols)
    else:
        s["weights"], s["gain"] = _stream(ctx, nblocks, g), _gains(nblocks, g)
        if op == "gemv_sorted":
            s["weights"] = P.llvq_sort_blocks(ctx, s["weights"], rows, cols)
        elif op == "gemm_sorted":
            s["weights"] = P.llvq_sort_blocks_gemm(ctx, s["weights"], rows, cols)
    if op != "dequant":
        shape = (case["batch"], cols) if op.startswith("gemm") else (cols,)
        s["x"] = torch.randn(shape, generator=g, device="cuda").bfloat16()
    return s


def run(s):
    case, ctx = s["case"], s["ctx"]
    op = case["op"]
    if op == "encode":
        metric = P.LLVQ_EUCLIDEAN if case["metric"] == "euclidean" else P.LLVQ_ANGULAR
        points, index = P.llvq_encode_blocks(ctx, s["v"], metric)
        fields = P.llvq_pack_fields(ctx, index, s["k"], case["gain_bits"])
        return {"points": points, "index": index, "fields": fields}
    if op == "gemv_multi":
        P.llvq_gemv_sorted_multi(ctx, s["mats"], y_dtype=_y_dtype(case))
        return [m[5] for m in s["mats"]]
    rows, cols = case["rows"], case["cols"]
    if op == "dequant":
        layout = P.LLVQ_LAYOUT_FLAT if case["layout"] == "flat" else P.LLVQ_LAYOUT_ROWWISE
        return P.llvq_dequant_matrix(ctx, s["weights"], s["gain"], rows, cols, layout)
    if op == "gemv":
        return P.llvq_gemv(ctx, s["weights"], s["gain"], rows, cols, s["x"], y_dtype=_y_dtype(case))
    if op == "gemv_sorted":
        return P.llvq_gemv_sorted(ctx, s["weights"], s["gain"], rows, cols, s["x"], y_dtype=_y_dtype(case))
    if op == "gemv_sg":
        return P.llvq_gemv_sg(ctx, s["weights"], case["gain_bits"], s["codebook"], s["scale"], rows, cols, s["x"], y_dtype=_y_dtype(case))
    if op == "gemv_sorted_sg":
        return P.llvq_gemv_sorted_sg(ctx, s["weights"], case["gain_bits"], s["codebook"], s["scale"], rows, cols, s["x"], y_dtype=_y_dtype(case))
    if op == "gemm":
        return P.llvq_gemm_small_batch(ctx, s["weights"], s["gain"], rows, cols, s["x"])
    return P.llvq_gemm_small_batch_sorted(ctx, s["weights"], s["gain"], rows, cols, s["x"])


def work(case):
    """Bytes: stored fields, gains and inputs read once, results written once.  Operations: those of the product (of the gain
    step for `dequant`, of scoring one point for `encode`); the index -> point map has no fixed count."""
    bits = _context(case["m_lo"], case["m_hi"]).index_bits
    op = case["op"]
    if op == "encode":
        n = case["blocks"]
        return {"bytes": n * (24 * 4 + 24 + 8 + (bits + case["gain_bits"]) / 8 + (1 if case["gain_bits"] else 0)), "flops": n * 24 * 3}
    if op == "gemv_multi":
        nbytes = flops = 0
        for rows, cols in _shapes(case):
            nbytes += rows * _blocks_per_row(cols) * (bits / 8 + 2) + cols * 2 + rows * (4 if case["y"] == "f32" else 2)
            flops += 2 * rows * cols
        return {"bytes": nbytes, "flops": flops}
    rows, cols = case["rows"], case["cols"]
    if op == "dequant":
        nblocks = (rows * cols + 23) // 24 if case["layout"] == "flat" else rows * _blocks_per_row(cols)
        return {"bytes": nblocks * (bits / 8 + 2) + rows * cols * 2, "flops": rows * cols}
    nblocks, batch = rows * _blocks_per_row(cols), case.get("batch", 1)
    weights = nblocks * (bits + case["gain_bits"]) / 8 + rows * 4 if "gain_bits" in case else nblocks * (bits / 8 + 2)
    return {"bytes": weights + batch * (cols * 2 + rows * (4 if case.get("y") == "f32" else 2)), "flops": 2 * rows * cols * batch}


def tolerance(case):
    if case["op"] in ("encode", "dequant"):
        return "exact"                                # whole numbers; weights rounded once
    if case.get("y") == "f32":
        return {"rel": 1e-5}                          # binary32 sums in another order
    return {"rel": 1e-2}                              # bf16 results
