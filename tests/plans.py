"""What the library decides on the host: the kernel that takes a GEMV call, the plan of a prefill call of more than 64 rows."""
import ctypes as C

import paper_2605_14844_b200 as xfp

FIELDS = ("T", "Tp", "parts", "tok_tiles", "row_pairs", "slots", "whole", "stream", "dealt", "ks", "sc_slice", "smem", "smem_max",
          "min_slots", "max_pairs", "pairs", "ctrl_bytes", "workspace", "SC")
KERNELS = ("none", "frag", "lane", "lane_batch", "gemm", "pair", "batch", "v2a", "generic")


def gemv_kernel(desc, batch, n=1, x_type=xfp.XFP_T_F16, y_type=xfp.XFP_T_F32, epilogue=0):
    """Which kernel file takes the call: xfp_gemv_<name>.cu (gemm: xfp_gemm_tc.cu; none: refused)."""
    k = C.c_int32()
    assert xfp.load_library().xfp_debug_gemv_kernel(C.byref(desc), batch, n, x_type, y_type, epilogue, C.byref(k)) == 0
    return KERNELS[k.value]


def dequant_plan(desc):
    """(super-chunks of a block, blocks of a row-block, outliers added to the staged rows)"""
    out = (C.c_int32 * 3)()
    assert xfp.load_library().xfp_debug_dequant_plan(C.byref(desc), out) == 0
    return out[0], out[1], bool(out[2])


def plan(desc, m):
    """A dict of FIELDS; None where the pair kernel does not take the call."""
    out = (C.c_int64 * len(FIELDS))()
    if xfp.load_library().xfp_debug_prefill_plan(C.byref(desc), m, out):
        return None
    return dict(zip(FIELDS, out))


def pieces(desc, m):
    """[pair] -> its pieces of work, (tile, first super-chunk, end)."""
    fn, out, got = xfp.load_library().xfp_debug_prefill_piece, (C.c_int32 * 3)(), []
    for g in range(plan(desc, m)["pairs"]):
        mine, i = [], 0
        while fn(C.byref(desc), m, g, i, out):
            mine.append(tuple(out))
            i += 1
        got.append(mine)
    return got


def features(desc, m):
    """What of the kernel a call reaches: two products per stage, the shortest ring, K cut over a cluster, tiles cut through the
    workspace, a pair that ends one tile and begins the next, whole tiles."""
    p = plan(desc, m)
    f = set()
    if p["parts"] == 2:
        f.add("two products")
    if p["slots"] == p["min_slots"]:
        f.add("shortest ring")
    if p["ks"] > 1:
        f.add("cluster")
        return f
    if p["whole"] or (p["dealt"] and p["dealt"] * p["SC"] == p["stream"]):
        f.add("whole tiles")
    if p["dealt"] and p["dealt"] * p["SC"] != p["stream"]:
        f.add("cut")
        if any(len(q) - p["whole"] > 1 for q in pieces(desc, m)):
            f.add("two pieces")
    return f
