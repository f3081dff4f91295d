"""Batches whose domains end inside one tile of the tensor-core kernel, against the oracle: databases
below one tile, and many queries of small domains beside a few of larger ones."""
import numpy as np
import pytest

import paper_2509_06514_gb300 as impir
from paper_2509_06514_gb300 import workloads

pytestmark = pytest.mark.gpu


def random_key(rng, m, prf, party=0):
    k = np.zeros(8 + 64 * (m + 1), np.uint8)
    k[0], k[1], k[2], k[3] = 1, prf, m, party
    k[8:] = rng.integers(0, 256, k.size - 8, dtype=np.uint8)
    for t, x in ((0, 1), (1, 0), (1, 1)):
        o = 8 + t * 32 * (m + 1) + (x * (m + 1)) * 16
        k[o:o + 16] = 0
    return k.tobytes()


@pytest.mark.parametrize("N,B,counts", [
    (600, 512, [(9, 30000), (10, 30)]),
    (544, 272, [(9, 29970), (10, 30)]),
    (1100, 512, [(8, 30000), (11, 40)]),
    (1500, 512, [(9, 30000), (11, 200)]),
    (900, 64, [(6, 40000), (10, 40000)]),
])
def test_many_queries_of_domains_below_a_tile(orc, N, B, counts):
    rng = np.random.default_rng(N + B)
    db = workloads.make_db(N, B, seed=N)
    keys, groups = [], []
    for m, n in counts:     # four distinct keys of each domain, spread over the batch
        ks = [random_key(rng, m, i % 2, i // 2) for i in range(4)]
        groups += [(k, range(len(keys) + i, len(keys) + n, 4)) for i, k in enumerate(ks)]
        keys += [ks[i % 4] for i in range(n)]
    blob, _ = impir.pack_keys(keys)
    h = impir.impir_db_load(db, N, B)
    try:
        got = impir.impir_answer(h, blob, len(keys), B)
    finally:
        impir.impir_db_free(h)
    for key, rows in groups:
        want = np.frombuffer(orc.answer(key, db, N, B, threads=8), np.uint8)
        assert (got[rows.start:rows.stop:4] == want).all(), key[2]
