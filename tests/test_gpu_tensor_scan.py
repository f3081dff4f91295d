"""The tensor-core form of the XOR answer: every answer equals the warp kernels' (an explicit launch
shape keeps a batch on them; they are compared with the oracle elsewhere) and, for a sample, the
oracle's, bit for bit. Sizes sit on the edges of its tiles (1024 records, 64-record operand tiles,
32-byte column passes, 128 rows): ragged record counts, odd numbers of 16-byte words, domains below a
tile and above the database, groups that shrink from tile to tile."""
import numpy as np
import pytest

import paper_2509_06514_gb300 as impir
from paper_2509_06514_gb300 import workloads

pytestmark = pytest.mark.gpu


def random_key(rng, m, prf, party=0):
    kb = 8 + 64 * (m + 1)
    k = np.zeros(kb, np.uint8)
    k[0], k[1], k[2], k[3] = 1, prf, m, party
    k[8:] = rng.integers(0, 256, kb - 8, dtype=np.uint8)
    for t, x in ((0, 1), (1, 0), (1, 1)):
        o = 8 + t * 32 * (m + 1) + (x * (m + 1)) * 16
        k[o:o + 16] = 0
    return k.tobytes()


def batch(seed, ms):
    rng = np.random.default_rng(seed)
    return [random_key(rng, m, int(rng.integers(0, 2)), i % 2) for i, m in enumerate(ms)]


def check(orc, N, B, keys, sample):
    db = workloads.make_db(N, B, seed=N + B)
    blob, _ = impir.pack_keys(keys)
    h = impir.impir_db_load(db, N, B)
    try:
        got = impir.impir_answer(h, blob, len(keys), B)
        impir.impir_set_config(h, lane_bits=4, queries_per_warp=4)
        assert np.array_equal(got, impir.impir_answer(h, blob, len(keys), B))
        for i in sample:
            assert got[i].tobytes() == orc.answer_points(keys[i], db, N, B) if keys[i][2] > 20 else \
                got[i].tobytes() == orc.answer(keys[i], db, N, B, threads=8), i
    finally:
        impir.impir_db_free(h)
    return db, blob, got


@pytest.mark.parametrize("N,B,ms", [
    (623_617, 16, [20] * 64),                                # 609 tiles, one record in the last; one column pass
    (640_000, 40, [20] * 65),                                # three words: a one-word last pass
    (78_000, 256, [17] * 1024),                              # eight full groups of 128 rows
    (80_001, 100, [17, 16, 13, 11, 10, 9, 6, 1, 40] * 115),  # domains below a tile, groups that shrink
    (700_000, 64, [20] * 5 + [19] * 130),                    # 5 queries past 2^19: the warp kernel's share
    (700_000, 64, [20] * 5 + [12] * 300 + [3] * 9),          # too few units: all the warp kernel's
    (120_065, 528, [17, 30] * 100),                          # 33 words, more than 512 bytes
    (235_000, 512, [18] * 64),
    (60_000, 1040, [16, 15] * 256),
])
def test_tensor_scan_matches_the_warp_kernels(orc, N, B, ms):
    keys = batch(N * 3 + B, ms)
    check(orc, N, B, keys, [0, len(keys) - 1])


def test_shards_streaming_and_scratch_take_it_too(orc):
    """Row shards, a streamed database and the no-alloc call on a batch large enough for it."""
    import torch
    N, B = 163_840 + 77, 512
    keys = batch(5, [18, 17] * 190)
    db, blob, want = check(orc, N, B, keys, [1])
    cut = 98_304
    parts = []
    for lo, rows in ((0, cut), (cut, N - cut)):
        h = impir.impir_db_load_rows(db[lo:lo + rows], rows, B, lo, N)
        parts.append(impir.impir_answer(h, blob, len(keys), B))
        impir.impir_db_free(h)
    assert np.array_equal(parts[0] ^ parts[1], want)
    streamed, _ = impir.impir_answer_streamed(db, N, B, blob, len(keys), 24 << 20)
    assert np.array_equal(streamed, want)
    d_db = torch.from_numpy(db).cuda()
    _, offs = impir.pack_keys(keys)
    d_keys = torch.from_numpy(np.frombuffer(blob, np.uint8).copy()).cuda()
    d_off = torch.from_numpy(offs.view(np.int32).copy()).cuda()
    out = torch.zeros((len(keys), B), dtype=torch.uint8, device="cuda")
    impir.impir_answer_noalloc(d_db, N, B, B, d_keys, d_off, len(keys), out)
    torch.cuda.synchronize()
    assert np.array_equal(out.cpu().numpy(), want)
