"""The plan of the prefill kernel on pairs of SMs and the kernel that takes a GEMV call: host code of the library, no GPU."""
import ctypes as C
import random

import pytest

from plans import gemv_kernel, pieces, plan
import paper_2605_14844_b200 as xfp
from paper_2605_14844_b200 import build as xbuild


@pytest.fixture(scope="module", autouse=True)
def _built():
    xbuild.build()


def _desc(mode, rows, cols, bits, lib_size=32, group=128, nnz=0):
    return xfp.XfpDesc(mode, rows, cols, bits, group, lib_size if mode else 0, 32, nnz)


def _shape(rng):
    mode, bits = rng.randrange(2), rng.randrange(2, 7)
    lib = rng.choice([n for n in (1, 7, 16, 32, 64, 256) if n << bits <= 1024]) if mode else 0
    cols = 128 * max(1, int(2 ** rng.uniform(0, 9)))
    rows = max(1, int(2 ** rng.uniform(0, min(15, 28 - cols.bit_length()))))
    return _desc(mode, rows, cols, bits, lib, rng.choice([64, 128]) if mode else 128), max(65, int(2 ** rng.uniform(6, 13)))


@pytest.mark.parametrize("seed", range(8))
def test_every_plan_covers_its_tiles_and_fits(seed):
    rng = random.Random(100 + seed)
    for _ in range(60):
        d, m = _shape(rng)
        p = plan(d, m)
        assert p is not None, (d.mode, d.rows, d.cols, d.bits, m)
        assert p["min_slots"] <= p["slots"] <= 12 and p["smem"] <= p["smem_max"]
        assert 64 <= p["T"] <= 512 and p["T"] % 32 == 0 and (p["tok_tiles"] - 1) * p["T"] < m <= p["tok_tiles"] * p["T"]
        assert p["parts"] == (2 if p["T"] > 256 else 1) and p["Tp"] % 32 == 0 and p["Tp"] <= 256
        assert (p["parts"] - 1) * p["Tp"] < p["T"] <= p["parts"] * p["Tp"]
        # every super-chunk of every tile once, in ascending runs
        tiles = p["row_pairs"] * p["tok_tiles"]
        work = pieces(d, m)
        got = {}
        for g, mine in enumerate(work):
            assert mine, g
            if p["ks"] > 1:
                assert len(mine) == 1 and mine[0][0] == g // p["ks"]          # the pairs of a cluster have one tile
            else:
                assert len(mine) <= p["whole"] + 2
                assert all(q[1:] == (0, p["SC"]) for q in mine[:p["whole"]])
                if len(mine) == p["whole"] + 2:                                # the second begins the next tile
                    assert mine[-1][0] == mine[-2][0] + 1 and mine[-1][1] == 0 and mine[-2][2] == p["SC"]
            for tile, a, b in mine:
                assert 0 <= a < b <= p["SC"]
                got.setdefault(tile, []).append((a, b))
        assert sorted(got) == list(range(tiles))
        for runs in got.values():
            runs.sort()
            assert runs[0][0] == 0 and runs[-1][1] == p["SC"] and all(x[1] == y[0] for x, y in zip(runs, runs[1:]))
        # counters: two for each dealt tile behind the error word; parts: two of either half for every dealt pair
        if p["ks"] == 1:
            assert tiles - p["whole"] * p["max_pairs"] < p["max_pairs"] or not p["dealt"]
            assert 4 * (1 + 2 * (tiles - p["whole"] * p["max_pairs"])) <= p["ctrl_bytes"]
        cut = p["ks"] == 1 and any(len(r) > 1 for r in got.values())
        assert p["workspace"] >= p["ctrl_bytes"] + (p["dealt"] * 4 * p["T"] * 128 * 4 if cut else 0)


def test_counters_do_not_depend_on_the_rows_of_x():
    rng = random.Random(7)
    for _ in range(40):
        d, _ = _shape(rng)
        assert len({plan(d, m)["ctrl_bytes"] for m in (65, 100, 300, 1024, 1792, 5000)}) == 1


@pytest.mark.parametrize("kernel,mode,rows,cols,bits,kw,batches", [
    ("frag", 0, 4096, 4096, 4, {}, (3, 4, 5, 8, 9, 16)), ("frag", 1, 4096, 4096, 4, {}, (3, 5, 16)),
    ("frag", 0, 256, 1024, 4, {}, (1,)), ("frag", 0, 28672, 8192, 4, {}, (5, 8)), ("frag", 1, 28672, 8192, 4, {}, (5, 8)),
    ("frag", 0, 33, 65536, 5, {}, (5, 8, 9, 16)), ("frag", 1, 24, 48128, 5, {}, (10,)),
    ("lane", 0, 4096, 4096, 4, {}, (1,)), ("lane", 1, 28672, 8192, 4, {}, (1,)),
    ("lane_batch", 0, 9600, 2048, 6, {}, (2, 4)), ("lane_batch", 1, 2500, 768, 4, {"group": 64}, (2, 4, 8, 16)),
    ("gemm", 0, 28672, 8192, 4, {}, (9, 16)), ("gemm", 1, 28672, 8192, 4, {}, (9, 16)),
    ("pair", 0, 4096, 4096, 4, {}, (2,)), ("batch", 0, 28672, 4096, 3, {}, (3, 4)), ("v2a", 1, 19000, 512, 3, {}, (2,)),
    ("generic", 1, 64, 256, 6, {"lib_size": 256}, (1, 2, 8, 16)), ("generic", 1, 200, 1024, 4, {"group": 64}, (2, 4, 8))])
def test_which_kernel_takes_a_gemv_call(kernel, mode, rows, cols, bits, kw, batches):
    """The dispatch at the sizes its rules name, fp16 x and 0.3 % outliers."""
    d = _desc(mode, rows, cols, bits, nnz=int(0.003 * rows * cols), **kw)
    assert {gemv_kernel(d, b) for b in batches} == {kernel}
