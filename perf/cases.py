"""The work this library does for its users, as cases that can be timed.

Five kinds of pass:

* ``layers``: the linear layers of one transformer block for one decode step: q/k/v and gate/up as grouped
  calls (their members read the same activations), o and down as single calls.  The step of every token of a
  generation.  With ``graph`` the four calls are captured once and replayed, as a serving loop does with its
  decode step; without, the program makes the four calls itself for every pass.
* ``linear``: one projection alone (``vq_gemv`` at batch 1), with or without block-wise normalisation: the
  smallest call there is, where launch and latency count.
* ``host``: the same block for a program that keeps activations in pinned host memory: every call takes its
  inputs from the host and puts its outputs there, and the program waits for the step before it reads them.
* ``decode``: a layer's weights materialised as binary16, with or without block-wise normalisation: what comes
  before the dense product of a prompt (prefill), and the transfer + decode comparison.
* ``assign``: the quantizer's nearest-centroid step over a dense layer, which writes the index stream (encode).

Formats are those of ``vq_synth.CONFIGS``; shapes are the projections listed there, and generic ones between.
Weights are drawn as there: uniform random indices (every pattern is valid), binary16 entries ~ N(0, sigma),
8-bit entries and 4-bit entries uniform, scales uniform in a narrow range, activations ~ N(0, 1).
"""
import torch

import paper_2402_15319_b200 as vq

FP16, INT8, INT4 = vq.VQ_CB_FP16, vq.VQ_CB_INT8_SCALED, vq.VQ_CB_INT4_G128

# vq_dim, index_bits, block_rows, block_cols, codebook type
FORMATS = {
    "2d4b_row1024_fp16": (2, 4, 1, 1024, FP16),
    "1d4b_row2048_int8": (1, 4, 1, 2048, INT8),
    "2d4b_row2048_int8": (2, 4, 1, 2048, INT8),
    "2d6b_128x128_fp16": (2, 6, 128, 128, FP16),
    "4d8b_256x512_fp16": (4, 8, 256, 512, FP16),
    "2d6b_32x256_int8": (2, 6, 32, 256, INT8),
    "2d6b_32x128_int4": (2, 6, 32, 128, INT4),
    "2d5b_4x256_int8": (2, 5, 4, 256, INT8),
}


def _layers(name, fmt, hidden, kv, ffn, batch, graph):
    return {"name": name, "kind": "layers", "format": fmt, "hidden": hidden, "kv": kv, "ffn": ffn, "batch": batch, "graph": graph}


def listed():
    return [
        # one attention projection of a 7B-class model, one token: launch and latency, 5 MB of weights
        {"name": "linear_4096_2d4b", "kind": "linear", "format": "2d4b_row1024_fp16", "n": 4096, "k": 4096, "batch": 1, "norm": 0},
        # a block of a 7B-class model, one token, 3.125 bits per value, the decode step captured
        _layers("block_7b_2d6b_b1", "2d6b_128x128_fp16", 4096, 4096, 11008, 1, True),
        # a block of a 13B-class model, eight sequences at once, 4-D entries
        _layers("block_13b_4d8b_b8", "4d8b_256x512_fp16", 5120, 5120, 13824, 8, False),
        # a block of a 70B-class model, one token, 2.13 bits per value, captured: the benchmark's default workload
        _layers("block_70b_2d4b_b1", "2d4b_row2048_int8", 8192, 1024, 28672, 1, True),
        # the same block for sixteen sequences: the largest batch, the largest pass
        _layers("block_70b_2d4b_b16", "2d4b_row2048_int8", 8192, 1024, 28672, 16, False),
        # a block of an 8B-class model in the format the paper deploys, one token, captured
        _layers("block_8b_2d6b_int8_b1", "2d6b_32x256_int8", 4096, 1024, 14336, 1, True),
        # 4-bit codebooks, a model of ragged width, an odd number of sequences
        _layers("block_ragged_int4cb_b5", "2d6b_32x128_int4", 3328, 416, 9088, 5, False),
        # small codebook blocks at 2.75 bits per value, three sequences
        _layers("block_8b_2d5b_b3", "2d5b_4x256_int8", 4096, 1024, 14336, 3, False),
        # activations that live on the host: the deployed format's block, one token
        {"name": "host_8b_2d6b_int8_b1", "kind": "host", "format": "2d6b_32x256_int8", "hidden": 4096, "kv": 1024, "ffn": 14336, "batch": 1},
        # gate projection with block-wise normalisation (sub-rows of 32 columns), one token
        {"name": "linear_14336_norm32", "kind": "linear", "format": "2d6b_32x256_int8", "n": 14336, "k": 4096, "batch": 1, "norm": 32},
        # a 7B-class gate projection materialised for a prompt
        {"name": "decode_11008_2d6b", "kind": "decode", "format": "2d6b_128x128_fp16", "n": 11008, "k": 4096, "norm": 0},
        # the same layer's quantization step
        {"name": "assign_11008_2d6b", "kind": "assign", "format": "2d6b_128x128_fp16", "n": 11008, "k": 4096, "hessian": True},
    ]


def _log(rng, lo, hi):
    return lo * (hi / lo) ** rng.random()


def _near(x, step):
    return max(step, int(round(x / step)) * step)


def draw(rng):
    kind = rng.choices(("layers", "linear", "host", "decode", "assign"), (6, 2, 1, 2, 1))[0]
    fmt = rng.choice(sorted(FORMATS))
    if kind == "assign":   # (the quantizer's step takes binary16 and 8-bit codebooks)
        fmt = rng.choice([f for f in sorted(FORMATS) if FORMATS[f][4] != INT4])
    d, b, br, bc, cb = FORMATS[fmt]
    batch = rng.choice((1, 1, 1, 2, 3, 4, 5, 6, 7, 8, 11, 13, 16))
    if kind in ("layers", "host"):
        wide = fmt in ("2d4b_row2048_int8", "2d4b_row1024_fp16")   # the 2-bit formats are used up to the 70B class
        rows = max(br, 8)
        step = max(rows, bc)   # hidden and ffn are rows of one layer and columns of another
        hidden = _near(_log(rng, 1024, 8192 if wide else 5120), step)
        kv = hidden if rng.random() < 0.4 else min(hidden, _near(hidden / rng.choice((2, 4, 8)), rows))
        ffn = _near(hidden * rng.uniform(2.5, 3.5), step)
        case = {"kind": kind, "format": fmt, "hidden": hidden, "kv": kv, "ffn": ffn, "batch": batch}
        if kind == "layers":
            case["graph"] = rng.random() < 0.5
        return case
    rows = br if br > 1 else rng.choice((1, 8, 64))
    n = _near(_log(rng, 512, 14336), rows)
    k = _near(_log(rng, 1024, 14336), bc)
    if kind == "assign":
        k = _near(_log(rng, 1024, 4096), bc)
        n = min(n, 11008 // rows * rows)
        if b == 8:
            n = _near(min(n, 4096), rows)
        return {"kind": kind, "format": fmt, "n": n, "k": k, "hessian": rng.random() < 0.5}
    norm = rng.choice((16, 32, 64)) if rng.random() < 0.3 and bc % 64 == 0 else 0
    if kind == "linear":
        return {"kind": kind, "format": fmt, "n": n, "k": k, "batch": batch, "norm": norm}
    return {"kind": kind, "format": fmt, "n": n, "k": k, "norm": norm}


# ---------------------------------------------------------------------------------------------------------------


def _fmt(case, n, k):
    return vq.VQFormat(n, k, *FORMATS[case["format"]])


def _calls(case):
    """[(K, [rows of the members])] of a block's four calls."""
    h, kv, f = case["hidden"], case["kv"], case["ffn"]
    return [(h, [h, kv, kv]), (h, [h]), (h, [f, f]), (f, [h])]


class _Draw:
    def __init__(self, seed):
        self.g = torch.Generator(device="cuda")
        self.g.manual_seed(int(seed))

    def bytes(self, *shape):
        return torch.randint(0, 256, shape, dtype=torch.uint8, device="cuda", generator=self.g)

    def normal(self, *shape, sigma=1.0):
        return (torch.randn(shape, device="cuda", generator=self.g) * sigma).half()

    def uniform(self, lo, hi, *shape):
        return (torch.rand(shape, device="cuda", generator=self.g) * (hi - lo) + lo).half()

    def weights(self, fmt):
        """(indices, codebooks, scales or None)"""
        info = vq.vq_pack_info(fmt)
        idx = self.bytes(fmt.n_rows, info.row_stride_bytes)
        cb, scale = self.codebooks(fmt, info)
        return idx, cb, scale

    def codebooks(self, fmt, info):
        if fmt.cb_type == INT4:
            return (self.bytes(info.n_blocks, info.entries * fmt.vq_dim // 2), self.uniform(0.001, 0.004, fmt.n_rows, fmt.k_cols // 128))
        if fmt.cb_type == INT8:
            cb = torch.randint(-127, 128, (info.n_blocks, info.entries, fmt.vq_dim), dtype=torch.int8, device="cuda", generator=self.g)
            return cb, self.uniform(0.0005, 0.002, info.n_blocks)
        return self.normal(info.n_blocks, info.entries, fmt.vq_dim, sigma=0.02), None


def _zeros(n):
    return torch.zeros(n, dtype=torch.uint8, device="cuda")


def _prepare_block(case, rnd, host):
    calls, outs = [], []
    batch = case["batch"]
    for k, rows in _calls(case):
        total = _fmt(case, sum(rows), k)
        x = rnd.normal(batch, k)
        ys = [torch.empty((batch, n), dtype=torch.float16, device="cuda") for n in rows]
        if host:
            x, ys = x.cpu().pin_memory(), [torch.empty((batch, n), dtype=torch.float16).pin_memory() for n in rows]
        members = [(*rnd.weights(_fmt(case, n, k)), y, n) for n, y in zip(rows, ys)]
        if not host:
            ws = vq.vq_workspace_bytes(total, batch)
        elif len(rows) > 1:
            ws = vq.vq_workspace_bytes_grouped_host(total, len(rows), batch)
        else:
            ws = vq.vq_workspace_bytes_host(total, batch)
        calls.append((total, members, x, _zeros(ws)))
        outs += ys
    return {"calls": calls, "batch": batch, "out": outs}


def _block(calls, batch):
    for fmt, members, x, ws in calls:
        if len(members) > 1:
            vq.vq_gemm_small_batch_grouped(fmt, members, x, batch, ws)
        else:
            idx, cb, scale, y, _ = members[0]
            vq.vq_gemm_small_batch(fmt, idx, cb, scale, x, y, batch, ws)


def _block_host(calls, batch):
    for fmt, members, x, ws in calls:
        if len(members) > 1:
            vq.vq_gemm_small_batch_grouped_host(fmt, members, x, batch, ws)
        else:
            idx, cb, scale, y, _ = members[0]
            vq.vq_gemm_small_batch_host(fmt, idx, cb, scale, x, y, batch, ws)
    torch.cuda.current_stream().synchronize()   # the program reads the outputs next


def _norm(rnd, fmt, cols):
    _, codes, lut = vq.vq_norm_info(fmt, cols)
    return rnd.bytes(codes), rnd.uniform(0.25, 4.0, lut // 2)


def prepare(case, seed):
    rnd = _Draw(seed)
    kind = case["kind"]
    if kind in ("layers", "host"):
        state = _prepare_block(case, rnd, kind == "host")
        torch.cuda.synchronize()   # weights are complete before the first call that reads them
        if case.get("graph"):
            _block(state["calls"], state["batch"])
            torch.cuda.synchronize()
            graph = torch.cuda.CUDAGraph()
            with torch.cuda.graph(graph):
                _block(state["calls"], state["batch"])
            state["graph"] = graph
    else:
        fmt = _fmt(case, case["n"], case["k"])
        state = {"fmt": fmt, "norm": case.get("norm", 0)}
        if kind == "assign":
            state["w"] = rnd.normal(fmt.n_rows, fmt.k_cols, sigma=0.02)
            info = vq.vq_pack_info(fmt)
            state["cb"], state["scale"] = rnd.codebooks(fmt, info)
            state["hdiag"] = torch.rand(fmt.k_cols, device="cuda", generator=rnd.g) * 4 + 0.25 if case["hessian"] else None
            state["out"] = torch.empty((fmt.n_rows, info.row_stride_bytes), dtype=torch.uint8, device="cuda")
        else:
            state["idx"], state["cb"], state["scale"] = rnd.weights(fmt)
            if state["norm"]:
                state["codes"], state["lut"] = _norm(rnd, fmt, state["norm"])
            if kind == "linear":
                state["batch"] = case["batch"]
                state["x"] = rnd.normal(case["batch"], fmt.k_cols)
                state["out"] = torch.empty((case["batch"], fmt.n_rows), dtype=torch.float16, device="cuda")
                state["ws"] = _zeros(vq.vq_workspace_bytes(fmt, case["batch"]))
            else:
                state["out"] = torch.empty((fmt.n_rows, fmt.k_cols), dtype=torch.float16, device="cuda")
        torch.cuda.synchronize()
    state["kind"] = kind
    return state


def run(state):
    s, kind = state, state["kind"]
    if kind == "layers":
        if "graph" in s:
            s["graph"].replay()
        else:
            _block(s["calls"], s["batch"])
    elif kind == "host":
        _block_host(s["calls"], s["batch"])
    elif kind == "linear":
        if s["norm"]:
            vq.vq_gemm_small_batch_normalized(s["fmt"], s["idx"], s["cb"], s["scale"], s["codes"], s["lut"], s["norm"], s["x"], s["out"], s["batch"])
        elif s["batch"] == 1:
            vq.vq_gemv(s["fmt"], s["idx"], s["cb"], s["scale"], s["x"], s["out"], s["ws"])
        else:
            vq.vq_gemm_small_batch(s["fmt"], s["idx"], s["cb"], s["scale"], s["x"], s["out"], s["batch"], s["ws"])
    elif kind == "decode":
        if s["norm"]:
            vq.vq_decode_weights_normalized(s["fmt"], s["idx"], s["cb"], s["scale"], s["codes"], s["lut"], s["norm"], s["out"])
        else:
            vq.vq_decode_weights(s["fmt"], s["idx"], s["cb"], s["scale"], s["out"])
    else:
        vq.vq_assign_indices(s["fmt"], s["w"], s["cb"], s["scale"], s["hdiag"], s["out"])
    return s["out"]


def work(case):
    """Stored weights, activations and outputs once each; a multiply and an add per weight and sequence."""
    kind = case["kind"]
    if kind in ("layers", "host"):
        byt = flops = 0
        for k, rows in _calls(case):
            byt += 2 * case["batch"] * k
            for n in rows:
                byt += vq.vq_pack_info(_fmt(case, n, k)).total_bytes + 2 * case["batch"] * n
                flops += 2 * n * k * case["batch"]
        return {"bytes": byt, "flops": flops}
    fmt = _fmt(case, case["n"], case["k"])
    n, k, info = case["n"], case["k"], vq.vq_pack_info(fmt)
    if kind == "assign":   # per vector and centroid: d differences, 2 d products, d - 1 sums, a comparison
        d = fmt.vq_dim
        return {"bytes": 2 * n * k + info.total_bytes, "flops": n * (k // d) * info.entries * 4 * d}
    byt = info.total_bytes
    if case["norm"]:
        _, codes, lut = vq.vq_norm_info(fmt, case["norm"])
        byt += codes + lut
    if kind == "decode":
        return {"bytes": byt + 2 * n * k, "flops": n * k if fmt.cb_type != FP16 or case["norm"] else 0}
    return {"bytes": byt + 2 * case["batch"] * (n + k), "flops": 2 * n * k * case["batch"]}


def tolerance(case):
    """Weights and indices are defined bit by bit.  Outputs are binary16, accumulated in binary32: one rounding of
    the result, and one of each weight where a scale enters it (the kernels choose whether the scale multiplies
    entries or sums).  Against products of the exact weights in binary64 the rounding of the result alone gives
    2.1e-4 (largest 4.9e-4), with the weights' rounding up to 3.5e-4 (largest 1.3e-3); stated here: four times that."""
    if case["kind"] in ("decode", "assign"):
        return "exact"
    return {"rel": 1.3e-3, "max": 5e-3}


def _weights64(fmt, idx, cb, scale, r0, r1, norm=None):
    """Rows r0..r1-1 of the weight matrix in binary64, unrounded: entry, times the block's or row group's scale,
    times the sub-row's scale under normalisation."""
    n, k, d, b, br, bc = fmt.n_rows, fmt.k_cols, fmt.vq_dim, fmt.index_bits, fmt.block_rows, fmt.block_cols
    dev = idx.device
    bit = torch.arange(k // d, device=dev) * b   # index j: bits j*b .. j*b + b - 1, least significant first
    rows = torch.nn.functional.pad(idx[r0:r1], (0, 1)).short()
    e = ((rows[:, bit // 8] | (rows[:, bit // 8 + 1] << 8)).int() & 0xFFFF) >> (bit % 8).int() & ((1 << b) - 1)
    blk = torch.arange(r0, r1, device=dev)[:, None] // br * (k // bc) + (torch.arange(k // d, device=dev) * d // bc)[None, :]
    if fmt.cb_type == INT4:
        raw = cb.reshape(-1)
        nib = torch.stack((raw & 15, raw >> 4), 1).reshape(-1).double()
        entries = torch.where(nib >= 8, nib - 16, nib)
    else:
        entries = cb.reshape(-1).double()
    w = entries.reshape(-1, d)[blk * (1 << b) + e]   # [rows, K/d, d]
    if fmt.cb_type == INT8:
        w = w * scale.double()[blk][..., None]
    w = w.reshape(r1 - r0, k)
    if fmt.cb_type == INT4:
        w = w * scale[r0:r1].double().repeat_interleave(128, 1)
    if norm:
        codes, lut, cols = norm
        codes = codes.reshape(n, -1)[r0:r1]
        code = torch.stack((codes & 15, codes >> 4), 2).reshape(r1 - r0, -1)[:, : k // cols].long()
        block = torch.arange(r0, r1, device=dev)[:, None] // br * (k // bc) + (torch.arange(k // cols, device=dev) * cols // bc)[None, :]
        w = w * lut.double()[block * 16 + code].repeat_interleave(cols, 1)
    return w


def _product64(fmt, idx, cb, scale, x, norm=None):
    x = x.cuda().double()
    step = max(1, (1 << 24) // fmt.k_cols)
    return torch.cat([x @ _weights64(fmt, idx, cb, scale, r, min(r + step, fmt.n_rows), norm).T for r in range(0, fmt.n_rows, step)], 1)


def exact(case, seed):
    """What run() returns for these inputs, in binary64 from the stored bytes (index streams have no such value)."""
    kind = case["kind"]
    if kind == "assign":
        return None
    s = prepare({**case, "graph": False}, seed)
    if kind in ("layers", "host"):
        return [_product64(_fmt(case, n, k), idx, cb, scale, x)
                for (k, _), (_, members, x, _) in zip(_calls(case), s["calls"]) for idx, cb, scale, _, n in members]
    norm = (s["codes"], s["lut"], s["norm"]) if s["norm"] else None
    if kind == "linear":
        return _product64(s["fmt"], s["idx"], s["cb"], s["scale"], s["x"], norm)
    step = max(1, (1 << 24) // s["fmt"].k_cols)
    return torch.cat([_weights64(s["fmt"], s["idx"], s["cb"], s["scale"], r, min(r + step, s["fmt"].n_rows), norm)
                      for r in range(0, s["fmt"].n_rows, step)], 0)
