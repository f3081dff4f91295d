"""Batches that the tensor-core kernel is known to take (the workspace header counts its units): domains
below a tile and above the database, records of odd widths, row shards that start past record 0, and
chunks of a streamed database on both of its streams. Answers equal the warp kernels' (an explicit shape
keeps a batch on them) and, for a sample, the oracle's. The files on that kernel also run on the debug
library, which checks every index."""
import os
import subprocess
import sys

import numpy as np
import pytest

import paper_2509_06514_gb300 as impir
from paper_2509_06514_gb300 import workloads
from test_gpu_schedule import random_key
from test_schedule_cpu import sched  # noqa: F401  (fixture)

pytestmark = pytest.mark.gpu

ROOT = os.path.dirname(os.path.dirname(os.path.abspath(__file__)))


def batch(seed, ms):
    rng = np.random.default_rng(seed)
    return [random_key(rng, m, int(rng.integers(0, 2)), i % 2) for i, m in enumerate(ms)]


def answers(h, keys, B):
    """Answers of a handle and the tensor-core kernel's units (header bytes 48 to 55)."""
    import torch
    stride = (B + 15) // 16 * 16
    blob, offs = impir.pack_keys(keys)
    d_keys = torch.from_numpy(np.frombuffer(blob, np.uint8).copy()).cuda()
    d_off = torch.from_numpy(offs.view(np.int32).copy()).cuda()
    out = torch.zeros((len(keys), B), dtype=torch.uint8, device="cuda")
    wsb = impir.impir_workspace_bytes(len(keys), stride)
    ws = torch.empty(wsb, dtype=torch.uint8, device="cuda")
    impir.impir_answer_async(h, d_keys, d_off, len(keys), out, ws, wsb, torch.cuda.current_stream())
    torch.cuda.synchronize()
    assert impir.impir_workspace_status(ws) == (0, 0xFFFFFFFF)
    return out.cpu().numpy(), int(ws[48:56].cpu().numpy().view("<u8")[0])


def warp_answers(db, N, B, keys):
    h = impir.impir_db_load(db, N, B)
    try:
        impir.impir_set_config(h, lane_bits=4, queries_per_warp=4)
        got, units = answers(h, keys, B)
    finally:
        impir.impir_db_free(h)
    assert units == 0
    return got


CASES = [
    (320_000, 100, [19, 16, 13, 11, 10, 9, 6, 1, 40] * 115),    # domains below a tile, groups that shrink
    (120_000, 1040, [17, 16] * 256),                            # 65 words: a last pass of one word
    (640_001, 1, [20] * 64),                                    # one byte a record, one record in the last tile
    (160_000, 272, [18] * 200 + [10] * 40 + [5] * 30),          # exactly a tile, and a warp's width
]


@pytest.mark.parametrize("N,B,ms", CASES)
def test_resident(orc, N, B, ms):
    keys = batch(N + B, ms)
    db = workloads.make_db(N, B, seed=N)
    h = impir.impir_db_load(db, N, B)
    try:
        got, units = answers(h, keys, B)
    finally:
        impir.impir_db_free(h)
    assert units > 0
    assert np.array_equal(got, warp_answers(db, N, B, keys))
    for i in {ms.index(m) for m in ms if m <= 20}:
        assert got[i].tobytes() == orc.answer(keys[i], db, N, B, threads=8), ms[i]


def test_shards_past_record_zero():
    N, B, cut = 262_144 + 77, 512, 131_072
    keys = batch(6, [19, 18] * 170 + [9] * 40)
    db = workloads.make_db(N, B, seed=6)
    parts = []
    for lo, rows in ((0, cut), (cut, N - cut)):
        h = impir.impir_db_load_rows(db[lo:lo + rows], rows, B, lo, N)
        try:
            part, units = answers(h, keys, B)
        finally:
            impir.impir_db_free(h)
        assert units > 0, lo
        parts.append(part)
    assert np.array_equal(parts[0] ^ parts[1], warp_answers(db, N, B, keys))


def test_streamed_on_both_streams(sched):  # noqa: F811
    N, B, chunk = 600_000, 272, 245_760
    ms = [20] * 500 + [17] * 6 + [9] * 6
    counts = {m: ms.count(m) for m in set(ms)}
    sms = impir.impir_device_sm_count()
    bounds = [0, chunk // 4, chunk // 4 + chunk, N]    # a quarter first, then whole chunks
    for lo, hi in zip(bounds, bounds[1:]):
        assert sched(N, B, counts, sms=sms, lo=lo, hi=hi).tc_units > 0
    keys = batch(7, ms)
    db = workloads.make_db(N, B, seed=7)
    got, _ = impir.impir_answer_streamed(db, N, B, b"".join(keys), len(keys), chunk * B)
    assert np.array_equal(got, warp_answers(db, N, B, keys))


def test_index_checks_of_the_tensor_core_kernel():
    if impir.BOUNDS:
        pytest.skip("this is the run on the debug library")
    from paper_2509_06514_gb300 import build
    build.build(bounds=True)
    r = subprocess.run([sys.executable, "-m", "pytest", "-x", "-q", "-m", "gpu", "-p", "no:cacheprovider",
                        "tests/test_gpu_tensor_scan.py", "tests/test_gpu_tensor_kernel.py", "tests/test_gpu_schedule.py"],
                       cwd=ROOT, env=dict(os.environ, IMPIR_BOUNDS="1"), capture_output=True, text=True, timeout=900)
    assert r.returncode == 0 and " passed" in r.stdout, r.stdout[-4000:] + r.stderr[-4000:]
