"""The work a user of this framework has it do, as cases that can be timed and compared.

A case is one pass through the public entry points:

    decode    one token step (or up to 16 rows of x) through a projection, or through the six projections of a decoder
              layer (q, k, v, o, up, down), y = (D + S) x on packed weights
    experts   one token through the routed feed-forward block of a layer: its active experts in two grouped launches
              with the gated activation and the routing-weighted sum fused into the stores
    prefill   a prompt of m rows of x through one projection
    encode    float weights -> outlier extraction, codebooks, auto-selected bit width, packed blob, and the matrix the
              blob stands for (the check of a quantise-on-load run)
    load      quantised tensors of a checkpoint -> packed blob -> fp16 matrix

mode 0 is V2 (a codebook per output channel), mode 1 is V2a (a library of 32 codebooks, a group of 128 weights names
one).  Sizes and bit widths are those of this repository's workloads and tests, and ragged ones beside them.
"""
import math

import torch

import paper_2605_14844_b200 as xfp
from paper_2605_14844_b200 import quant_binding as qb
from paper_2605_14844_b200 import synth

LIB = 32        # codebooks of a V2a library
GROUP = 128     # weights of a V2a group
MAX_WEIGHTS = 28672 * 8192
MAX_PRODUCTS = 1024 * MAX_WEIGHTS
DTYPES = {"fp16": torch.float16, "bf16": torch.bfloat16}


def listed():
    return [
        # One call on one projection (configuration 1 of the benchmark): launch and latency are what a user waits for.
        {"name": "decode_projection", "op": "decode", "mode": 0, "rows": 4096, "cols": 4096, "inter": 0, "bits": 4,
         "rate": 0.003, "batch": 1, "dtype": "fp16"},
        # A token through one decoder layer of the benchmark's stack, bf16 activations as the paper's kernel takes them.
        {"name": "decode_layer_v2", "op": "decode", "mode": 0, "rows": 4096, "cols": 4096, "inter": 12288, "bits": 4,
         "rate": 0.01, "batch": 1, "dtype": "bf16"},
        # The same layer in the library form.
        {"name": "decode_layer_v2a", "op": "decode", "mode": 1, "rows": 4096, "cols": 4096, "inter": 12288, "bits": 4,
         "rate": 0.005, "batch": 1, "dtype": "fp16"},
        # The largest projection of the repository's sweep at one row of x: weight traffic is everything.
        {"name": "decode_large", "op": "decode", "mode": 0, "rows": 28672, "cols": 8192, "inter": 0, "bits": 5,
         "rate": 0.01, "batch": 1, "dtype": "bf16"},
        # Several requests decoded together: one pass over the weights for eight rows of x.
        {"name": "decode_batch", "op": "decode", "mode": 0, "rows": 4096, "cols": 4096, "inter": 12288, "bits": 4,
         "rate": 0.003, "batch": 8, "dtype": "bf16"},
        # A token through the routed block of a mixture-of-experts layer (configuration 3): eight active experts.
        {"name": "experts", "op": "experts", "hidden": 4096, "inter": 1536, "active": 8, "bits": 3, "rate": 0.001,
         "dtype": "bf16"},
        # A short prompt on an attention projection.
        {"name": "prefill_short", "op": "prefill", "mode": 0, "rows": 4096, "cols": 4096, "bits": 4, "rate": 0.009,
         "m": 100, "dtype": "bf16"},
        # A prompt of odd length on a matrix whose sizes are multiples of nothing but the group, in the library form.
        {"name": "prefill_ragged_v2a", "op": "prefill", "mode": 1, "rows": 10007, "cols": 4992, "bits": 4, "rate": 0.003,
         "m": 301, "dtype": "bf16"},
        # A long prompt on the largest projection: the dense contraction at full size.
        {"name": "prefill_long", "op": "prefill", "mode": 0, "rows": 28672, "cols": 8192, "bits": 4, "rate": 0.003,
         "m": 1024, "dtype": "fp16"},
        # Quantise-on-load of an up projection: per-channel codebooks, candidates and threshold of attention layers.
        {"name": "encode_v2", "op": "encode", "mode": 0, "rows": 12288, "cols": 4096, "cands": "4,5", "tau": 0.96},
        # Quantise-on-load of an expert's gate_up projection in the library form, candidates and threshold of experts.
        {"name": "encode_v2a", "op": "encode", "mode": 1, "rows": 3072, "cols": 4096, "cands": "2,4", "tau": 0.93},
        # A checkpoint that is quantised already: pack for this device, reconstruct the fp16 matrix.
        {"name": "load_v2a", "op": "load", "mode": 1, "rows": 12289, "cols": 4096, "bits": 4, "rate": 0.01},
    ]


def _log(rng, lo, hi, multiple=1):
    v = int(round(math.exp(rng.uniform(math.log(lo), math.log(hi))) / multiple)) * multiple
    return min(max(v, -(-lo // multiple) * multiple), hi // multiple * multiple)


def _matrix(rng, lo, hi, most):
    """rows (any number, also odd ones) and cols (a multiple of the group) with at most `most` weights."""
    cols = _log(rng, lo, min(hi, 16384), GROUP)
    rows = _log(rng, lo, max(lo, min(hi, most // cols)))
    return (rows if rng.random() < 0.5 else max(64, rows // 64 * 64)), cols


def draw(rng):
    op = rng.choice(["decode"] * 5 + ["experts"] + ["prefill"] * 3 + ["encode"] * 2 + ["load"])
    mode, dtype = rng.randrange(2), rng.choice(["fp16", "bf16"])
    rate = rng.choice([0.0, round(rng.uniform(0.0005, 0.02), 4), 0.003])
    if op == "decode":
        batch = rng.choice([1, 1, 1, 2, 4, rng.randrange(2, 17)])
        inter = 0
        if rng.random() < 0.4:
            rows = cols = _log(rng, 1024, 8192, GROUP)
            inter = _log(rng, cols, min(4 * cols, 28672), GROUP)
        else:
            rows, cols = _matrix(rng, 512, 28672, MAX_WEIGHTS)
        return {"op": op, "mode": mode, "rows": rows, "cols": cols, "inter": inter, "bits": rng.randrange(2, 7),
                "rate": rate, "batch": batch, "dtype": dtype}
    if op == "experts":
        return {"op": op, "hidden": _log(rng, 1024, 7168, GROUP), "inter": _log(rng, 512, 3072, GROUP),
                "active": rng.randrange(2, 11), "bits": rng.randrange(2, 5), "rate": min(rate, 0.005), "dtype": dtype}
    if op == "prefill":
        rows, cols = _matrix(rng, 1024, 28672, MAX_WEIGHTS)
        # V2a libraries of 32 codebooks reach the tensor-core kernel up to 5 bits
        return {"op": op, "mode": mode, "rows": rows, "cols": cols, "bits": rng.randrange(2, 6 if mode else 7), "rate": rate,
                "m": _log(rng, 17, min(2048, max(64, MAX_PRODUCTS // (rows * cols)))), "dtype": dtype}
    if op == "encode":
        rows, cols = _matrix(rng, 512, 12288, 3072 * 4096 if mode else 6144 * 4096)
        cands, tau = rng.choice([("4,5", 0.96), ("2,4", 0.93), ("3,4", 0.985)])
        return {"op": op, "mode": mode, "rows": rows, "cols": min(cols, 8192), "cands": cands, "tau": tau}
    rows, cols = _matrix(rng, 512, 28672, 12288 * 8192)
    return {"op": op, "mode": mode, "rows": rows, "cols": cols, "bits": rng.randrange(2, 7), "rate": rate}


def _shapes(case):
    """The projections of a decode pass: one, or q, k, v, o, up and down of a layer."""
    rows, cols, inter = case["rows"], case["cols"], case["inter"]
    return [(rows, cols)] * 4 + [(inter, cols), (rows, inter)] if inter else [(rows, cols)]


def _quantized(mode, rows, cols, bits, rate, seed, library=None):
    return synth.random_quantized_torch(mode, rows, cols, bits, rate, seed, lib_size=LIB, group_size=GROUP,
                                        library=library)


def _normal(shape, seed, dtype):
    g = torch.Generator(device="cuda")
    g.manual_seed(seed)
    return torch.randn(shape, generator=g, device="cuda").to(dtype)


def _pointers(tensors):
    return torch.tensor([t.data_ptr() for t in tensors], dtype=torch.int64, device="cuda")


def _float_weights(rows, cols, seed):
    """Gaussian bulk with heavy outlier columns: half of the weights of 2 % of the input columns lie at 10 .. 49 sigma."""
    g = torch.Generator(device="cuda")
    g.manual_seed(seed)
    W = torch.randn((rows, cols), generator=g, device="cuda") * synth.SIGMA0
    hot = torch.randperm(cols, generator=g, device="cuda")[:max(1, cols // 50)]
    mag = (torch.rand((rows, hot.numel()), generator=g, device="cuda") * 39.0 + 10.0) * synth.SIGMA0
    coin = torch.rand((rows, hot.numel()), generator=g, device="cuda")
    W[:, hot] = torch.where(coin < 0.25, mag, torch.where(coin < 0.5, -mag, W[:, hot]))
    return W


def prepare(case, seed):
    op = case["op"]
    if op == "decode":
        dt = DTYPES[case["dtype"]]
        layers, xs = [], {}
        for j, (rows, cols) in enumerate(_shapes(case)):
            pm = xfp.pack_tensors(_quantized(case["mode"], rows, cols, case["bits"], case["rate"], seed * 64 + j))
            if cols not in xs:
                xs[cols] = _normal((case["batch"], cols), seed * 64 + 32 + len(xs), dt)
            layers.append((pm, xs[cols], torch.empty((case["batch"], rows), dtype=dt, device="cuda")))
        return {"op": op, "typed": dt == torch.bfloat16, "batch": case["batch"], "layers": layers}
    if op == "experts":
        dt, n, hidden, inter = DTYPES[case["dtype"]], case["active"], case["hidden"], case["inter"]
        sides = []
        for s, (rows, cols) in enumerate(((2 * inter, hidden), (hidden, inter))):
            library, pms = None, []
            for j in range(n):
                q = _quantized(1, rows, cols, case["bits"], case["rate"], seed * 64 + 16 * s + j, library)
                library = q.codebook          # the experts of a layer share one library per projection
                pms.append(xfp.pack_tensors(q))
            d = pms[0].desc
            desc = xfp.XfpDesc(d.mode, d.rows, d.cols, d.bits, d.group_size, d.lib_size, d.col_bits,
                               max(p.desc.nnz for p in pms))
            ws = torch.zeros(n * xfp.xfp_packed_size(desc)[1], dtype=torch.uint8, device="cuda")
            sides.append((desc, pms, _pointers([p.packed for p in pms]), ws))
        x = _normal((1, hidden), seed * 64 + 40, dt)
        h = torch.empty((n, inter), dtype=dt, device="cuda")
        y = torch.empty((1, hidden), dtype=dt, device="cuda")
        weights = torch.softmax(_normal((n,), seed * 64 + 41, torch.float32), 0)
        return {"op": op, "n": n, "dtype": dt, "up": sides[0], "down": sides[1], "x": x, "h": h, "y": y, "weights": weights,
                "x_ptr": _pointers([x] * n), "h_ptr": _pointers([h[j] for j in range(n)]), "y_ptr": _pointers([y] * n)}
    if op == "prefill":
        dt = DTYPES[case["dtype"]]
        pm = xfp.pack_tensors(_quantized(case["mode"], case["rows"], case["cols"], case["bits"], case["rate"], seed * 64))
        ws = torch.zeros(xfp.xfp_gemm_typed_workspace_size(pm.desc, case["m"], dt), dtype=torch.uint8, device="cuda")
        return {"op": op, "pm": pm, "x": _normal((case["m"], case["cols"]), seed * 64 + 1, dt), "ws": ws,
                "y": torch.empty((case["m"], case["rows"]), dtype=dt, device="cuda")}
    if op == "encode":
        return {"op": op, "mode": case["mode"], "W": _float_weights(case["rows"], case["cols"], seed),
                "cands": tuple(int(c) for c in case["cands"].split(",")), "tau": case["tau"]}
    return {"op": op, "q": _quantized(case["mode"], case["rows"], case["cols"], case["bits"], case["rate"], seed * 64)}


def run(state):
    op = state["op"]
    if op == "decode":
        for pm, x, y in state["layers"]:
            if state["typed"]:
                xfp.xfp_gemv_typed(pm.desc, pm.packed, x, state["batch"], y, pm.workspace)
            else:
                pm.gemv(x, y=y, y_fp16=True)
        return [y for _, _, y in state["layers"]]
    if op == "experts":
        n, dt = state["n"], state["dtype"]
        desc, _, blobs, ws = state["up"]
        xfp.xfp_gemv_grouped_typed(desc, n, blobs, state["x_ptr"], dt, state["h_ptr"], dt, xfp.XFP_EPI_SWIGLU, None, ws)
        desc, _, blobs, ws = state["down"]
        xfp.xfp_gemv_grouped_typed(desc, n, blobs, state["h_ptr"], dt, state["y_ptr"], dt, xfp.XFP_EPI_COMBINE,
                                   state["weights"], ws)
        return [state["h"], state["y"]]
    if op == "prefill":
        pm = state["pm"]
        xfp.xfp_gemm_typed(pm.desc, pm.packed, state["x"], state["y"], state["ws"])
        return state["y"]
    if op == "encode":
        pm, res = qb.quantize_and_pack(state["W"], state["mode"], state["cands"], state["tau"], lib_size=LIB)
        return {"bits": res.bits, "nnz": res.nnz, "mu": res.mu, "sigma": res.sigma, "median_cos": res.median_cos,
                "W": pm.dequant()}
    return xfp.pack_tensors(state["q"]).dequant()


def _blob_bytes(mode, rows, cols, bits, rate):
    """Indices, codebooks or library and group metadata, outliers (column and value) with their row pointers."""
    b = rows * cols * bits / 8 + (rows if mode == 0 else LIB) * (1 << bits) * 2 + 4 * rate * rows * cols + 4 * (rows + 1)
    return b + (rows * (cols // GROUP) * 5 if mode else 0)


def work(case):
    op = case["op"]
    if op == "decode":
        shapes, m = _shapes(case), case["batch"]
        x = 2 * m * sum({cols: cols for _, cols in shapes}.values())
        return {"bytes": x + sum(_blob_bytes(case["mode"], r, c, case["bits"], case["rate"]) + 2 * m * r for r, c in shapes),
                "flops": sum(2 * m * r * c for r, c in shapes)}
    if op == "experts":
        n, hidden, inter = case["active"], case["hidden"], case["inter"]
        return {"bytes": n * sum(_blob_bytes(1, r, c, case["bits"], case["rate"]) for r, c in ((2 * inter, hidden), (hidden, inter)))
                + 2 * (hidden + n * inter * 2 + hidden), "flops": 6 * n * hidden * inter}
    rows, cols = case["rows"], case["cols"]
    if op == "prefill":
        m = case["m"]
        return {"bytes": _blob_bytes(case["mode"], rows, cols, case["bits"], case["rate"]) + 2 * m * (rows + cols),
                "flops": 2 * m * rows * cols}
    if op == "encode":
        # W in, the packed blob and its fp16 matrix out; every candidate tried looks every weight up once
        least = int(case["cands"].split(",")[0])
        return {"bytes": 4 * rows * cols + _blob_bytes(case["mode"], rows, cols, least, 0.01) + 2 * rows * cols,
                "flops": 2 * rows * cols}
    blob = _blob_bytes(case["mode"], rows, cols, case["bits"], case["rate"])
    return {"bytes": rows * cols + blob + 2 * rows * cols, "flops": 2 * rows * cols}


def tolerance(case):
    if case["op"] == "load":
        return "exact"                       # the format defines every fp16 value of the matrix
    if case["op"] == "encode":
        # the encoder's decisions are taken in fp64 in an order the method states: the matrix, the width and the count are
        # one answer; mu, sigma and the cosine are sums whose order is free
        return {"rel": 1e-7, "max": 1e-6, "differ": 0.0}
    # one rounding of the sum to the output type; the decoded weight may be rounded to fp16 (prefill) or not (decode),
    # and in the routed block the stored activation is rounded between the two projections
    return {"rel": 8e-3} if case["dtype"] == "bf16" else {"rel": 2e-3}
