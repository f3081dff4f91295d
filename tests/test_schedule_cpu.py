"""The work schedule of a batch, built on the host by the code the setup kernel runs: every query gets
each record of its domain exactly once, whichever kernel takes a tile, for whole databases, row shards
and the chunks of a streamed database, and no launch reads past its records."""
import ctypes
import os
import random
import subprocess

import pytest

ROOT = os.path.dirname(os.path.dirname(os.path.abspath(__file__)))
SHARD_ALIGN = 32768


class Result(ctypes.Structure):
    _fields_ = [("tc_units", ctypes.c_uint64), ("n_units", ctypes.c_uint64), ("lane_bits", ctypes.c_uint32),
                ("shape_lane_bits", ctypes.c_uint32), ("qpw", ctypes.c_uint32), ("tc_min_active", ctypes.c_uint32),
                ("tc_shape", ctypes.c_uint32), ("pad", ctypes.c_uint32)]


@pytest.fixture(scope="module")
def sched(tmp_path_factory):
    so = str(tmp_path_factory.mktemp("schedule") / "schedule.so")
    subprocess.run(["g++", "-std=c++17", "-O2", "-shared", "-fPIC", "-I", "/usr/local/cuda/include",
                    os.path.join(ROOT, "tests", "schedule_host.cpp"), "-o", so], check=True)
    L = ctypes.CDLL(so)
    L.schedule_what.restype = ctypes.c_char_p
    L.schedule_check.argtypes = [ctypes.c_uint64, ctypes.c_uint64, ctypes.c_uint32, ctypes.c_void_p, ctypes.c_int,
                                 ctypes.c_uint64, ctypes.c_uint64, ctypes.c_int, ctypes.c_void_p]
    L.schedule_tile_bits.argtypes = [ctypes.c_uint64, ctypes.c_uint32, ctypes.c_uint32, ctypes.c_int]

    def check(N, B, counts, sms=152, lo=0, hi=0, n_launch=None, add=0):
        hist = (ctypes.c_uint32 * 41)()
        for m, k in counts.items():
            hist[m] += k
        r = Result()
        st = L.schedule_check(N, n_launch or N, (B + 15) // 16, hist, sms, lo, hi, add, ctypes.byref(r))
        assert st == 0, (L.schedule_what().decode(), N, B, dict(counts), sms, lo, hi)
        return r

    check.lib = L
    check.tile_bits = lambda N, B, n, sms=152: L.schedule_tile_bits(N, (B + 15) // 16, n, sms)
    return check


# many queries of domains below one tensor-core tile, a few above: a warp kernel's tile can be smaller
# than a tensor-core tile, and the line between the two kernels may not fall inside the latter
@pytest.mark.parametrize("N,B,counts", [
    (544, 272, {9: 29970, 10: 30}),
    (600, 512, {9: 30000, 10: 30}),
    (1000, 512, {9: 30000, 10: 30}),
    (1100, 512, {8: 30000, 11: 40}),
    (1500, 512, {9: 30000, 11: 40}),
    (5000, 4096, {7: 30000, 13: 30}),
    (1 << 20, 4096, {9: 30000, 20: 95}),
    (700, 16, {9: 80000, 10: 63}),
])
def test_the_line_between_the_kernels(sched, N, B, counts):
    sched(N, B, counts)


def batch(r, N, top):
    """Domain sizes of a batch: one to four sizes, one of them often far more frequent."""
    cover = max(1, (N - 1).bit_length())
    ms = [min(40, max(1, r.choice([cover, cover - r.randint(0, 12), r.randint(1, cover), r.randint(1, 14), 40])))
          for _ in range(r.randint(1, 4))]
    return {m: max(1, int(2 ** r.uniform(0, top))) for m in ms}


def size(r):
    B = r.choice([1, 16, 40, 64, 256, 272, 512, 528, 1024, 2048, 4096, 20000])
    return int(2 ** r.uniform(0, 15)) if r.random() < 0.6 else int(2 ** r.uniform(10, 25)), B


@pytest.mark.parametrize("seed", range(4))
def test_random_databases(sched, seed):
    r = random.Random(seed)
    took = 0
    for _ in range(2000):
        N, B = size(r)
        counts = batch(r, N, 17)
        took += sched(N, B, counts, sms=r.choice([148, 152])).tc_units > 0
        sched(N, B, counts, add=1)
    assert took > 50        # the tensor-core kernel is among what was checked


@pytest.mark.parametrize("seed", range(2))
def test_random_shards_and_chunks(sched, seed):
    r = random.Random(1000 + seed)
    took = 0
    for _ in range(700):
        N, B = size(r)
        counts = batch(r, N, 12)
        n = sum(counts.values())
        cuts = sorted({0, N, *(r.randrange(0, N, SHARD_ALIGN) for _ in range(r.randint(0, 3)))})
        for lo, hi in zip(cuts, cuts[1:]):
            took += sched(N, B, counts, lo=lo, hi=hi, n_launch=hi - lo).tc_units > 0
        # chunks of a streamed database: whole tiles of both kernels
        T = 32 << sched.tile_bits(N, B, n)
        chunk = T * r.randint(1, 1 + N // T)
        for lo in range(0, N, max(chunk, (N // 8 + T - 1) // T * T)):
            hi = min(N, lo + max(chunk, (N // 8 + T - 1) // T * T))
            took += sched(N, B, counts, lo=lo, hi=hi).tc_units > 0
    assert took > 50


def fewest(B):
    return 64 if (B + 15) // 16 <= 32 else 96


# (queries of a small domain, the large domain, its queries): a domain that ends inside a warp tile is no
# place to draw the line, but does not hand the tiles behind it to the tensor-core kernel either
@pytest.mark.parametrize("N,B,counts", [
    (1 << 24, 512, {10: 64, 24: 8}),
    (1 << 25, 256, {12: 200, 25: 1}),
    (1 << 20, 4096, {9: 30000, 20: 95}),
    (1 << 22, 64, {3: 100, 14: 20, 22: 40}),
])
def test_tiles_that_few_queries_reach_stay_with_the_warp_kernels(sched, N, B, counts):
    assert sched(N, B, counts).tc_units == 0


@pytest.mark.parametrize("seed", range(4))
def test_every_tensor_core_tile_has_enough_queries(sched, seed):
    r = random.Random(2000 + seed)
    took = 0
    for _ in range(2000):
        N, B = size(r)
        got = sched(N, B, batch(r, N, 13))
        if got.tc_units:
            took += 1
            assert got.tc_min_active >= fewest(B), (N, B)
    assert took > 50


def test_narrow_groups_of_the_widest_records_need_more_units(sched):
    """96 queries on 2^19 records of 4 KiB (512 units) are faster in the warp kernels, 104 are not, and
    1024 units gain with either."""
    assert sched(1 << 19, 4096, {19: 96}).tc_units == 0
    assert sched(1 << 19, 4096, {19: 104}).tc_units == 512
    assert sched(1 << 20, 4096, {20: 96}).tc_units == 1024
    assert sched(1 << 18, 4096, {18: 128}).tc_units == 256


@pytest.mark.parametrize("B", [16, 512, 528, 4096])
def test_shapes_that_are_launched_with_fewer_warps(sched, B):
    """Of all shapes that impir_set_config takes, the two that include/impir.h names."""
    import paper_2509_06514_gb300 as impir
    from paper_2509_06514_gb300 import build
    build.build()
    h = impir.impir_db_attach(1 << 20, 1 << 20, B, B)      # an address that is never read
    fewer, taken = set(), 0
    for lane_bits in range(11):
        for qpw in (1, 2, 4, 8, 16):
            for warps in range(4, 21):
                try:
                    impir.impir_set_config(h, lane_bits, qpw, warps)
                except impir.ImpirError:
                    continue
                taken += 1
                got = sched.lib.launched_warps(lane_bits, qpw, warps)
                if got != warps:
                    fewer.add((qpw << lane_bits, warps, got))
    impir.impir_db_free(h)
    assert taken > 400 and fewer == {(2048, 12, 11), (4096, 6, 5)}
