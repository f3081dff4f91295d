"""What is measured of this framework: answers of PIR batches through its public entry points.

A case is one batch of queries against one database that is already resident on the device:

  entry   "answer": host keys in, host answers out, the call waits (a request handled by itself);
          "async": device keys and answers on the caller's stream (a server's batches);
          "add32": the additive answer over Z_2^32, on the caller's stream
  n, b    records and bytes of a record
  q       queries of the batch
  m, dm   domain bits: query i has m - (one of 0..dm), drawn from the seed, so that batches mix
          queries against prefixes of the database; m covers the database
  prf     0: AES keyed by the node's seed, 1: the fixed-key form, 2: a batch that mixes both

Targets are uniform, database bytes uniform random, keys come from the library's own generator
and alternate between the two parties. Answers are whole bytes and are exact.
"""
import random

import numpy as np
import torch

import paper_2509_06514_gb300 as impir

DEV = "cuda"

LISTED = [
    # one query against a 2 MiB database, handled by itself: launches and latency
    dict(name="single_2m", entry="answer", n=1 << 16, b=32, q=1, m=16, dm=0, prf=0),
    # a small batch on the smallest database a server keeps resident
    dict(name="batch_16m_64b", entry="async", n=1 << 18, b=64, q=16, m=18, dm=0, prf=0),
    # one query against a 1 GiB database, handled by itself: a request under low load
    dict(name="single_1g", entry="answer", n=1 << 22, b=256, q=1, m=22, dm=0, prf=0),
    # odd sizes everywhere: records that need padding, a record count that ends inside a tile,
    # mixed domains and both PRFs in one batch
    dict(name="ragged_100b", entry="async", n=1_000_003, b=100, q=37, m=20, dm=6, prf=2),
    # the batched workload: 256 MiB, 64 queries in one launch
    dict(name="batch_256m", entry="async", n=1 << 20, b=256, q=64, m=20, dm=0, prf=0),
    # the same batch, additive answers
    dict(name="add32_256m", entry="add32", n=1 << 20, b=256, q=64, m=20, dm=0, prf=0),
    # a few queries against an 8 GiB database of 512-byte records: a server under low load
    dict(name="few_8g_512b", entry="async", n=1 << 24, b=512, q=8, m=24, dm=0, prf=0),
    # the widest records, 1 GiB
    dict(name="wide_1g_4k", entry="async", n=1 << 18, b=4096, q=128, m=18, dm=0, prf=0),
    # a server's mean batch, clients that use the fixed-key PRF
    dict(name="mmo_1g", entry="async", n=1 << 22, b=256, q=125, m=22, dm=0, prf=1),
    # the GB-scale workload: 4 GiB of 1 KiB records, 256 queries
    dict(name="batch_4g_1k", entry="async", n=1 << 22, b=1024, q=256, m=22, dm=0, prf=0),
    # the uneven workload's largest batch: 8 GiB, domains of 2^23 to 2^25
    dict(name="uneven_8g", entry="async", n=1 << 25, b=256, q=416, m=25, dm=2, prf=0),
]


def listed():
    return [dict(c) for c in LISTED]


def _cost(n, b, q):
    """Operations of a batch in units of one table lookup: the tree and the scan."""
    return q * n * (2 * 158.0 + b / 8.0)


def draw(rng):
    """Batches over the same ranges: 2^10 to 2^25 records of 1 to 4096 bytes (at most 8 GiB),
    1 to 416 queries, all entry points, both PRFs, mixed domains, odd sizes."""
    top = _cost(1 << 25, 256, 416) / 3
    while True:
        entry = rng.choice(["answer", "async", "async", "add32"])
        n = int(2 ** rng.uniform(10, 25))
        if rng.random() < 0.4:
            n = 1 << n.bit_length() - 1
        b = int(2 ** rng.uniform(0, 12.01))
        if rng.random() < 0.5:
            b = 1 << b.bit_length() - 1
        b = min(4096, b)
        if entry == "add32":
            b = max(4, b // 4 * 4)
        q = int(2 ** rng.uniform(0, 8.71))
        if n * b > 8 << 30 or _cost(n, b, q) > top:
            continue
        return dict(entry=entry, n=n, b=b, q=q, m=max(1, (n - 1).bit_length()), dm=rng.choice([0, 0, 2, 6]),
                    prf=rng.choice([0, 0, 0, 1, 2]))


def _domains(case, seed):
    r = random.Random(seed * 7919 + 1)
    return [max(1, case["m"] - r.randint(0, case["dm"])) for _ in range(case["q"])]


def _keys(case, seed):
    """The batch's wire keys, as the clients sent them."""
    r = random.Random(seed * 7919 + 2)
    keys = []
    for i, m in enumerate(_domains(case, seed)):
        alpha = r.randrange(min(case["n"], 1 << m))
        prf = i % 2 if case["prf"] == 2 else case["prf"]
        keys.append(impir.dpf_gen(alpha, m, prf, r.randbytes(32))[(i // 2) % 2])
    return keys


def _records(case, seed):
    """(N, stride) uint8 on the device: uniform random records, zero padding to 16 bytes."""
    n, b = case["n"], case["b"]
    stride = (b + 15) // 16 * 16
    g = torch.Generator(device=DEV).manual_seed(seed * 7919 + 3)
    if stride == b:
        return torch.randint(-(1 << 63), (1 << 63) - 1, (n * b // 8,), dtype=torch.int64, device=DEV,
                             generator=g).view(torch.uint8).view(n, b)
    d = torch.zeros((n, stride), dtype=torch.uint8, device=DEV)
    d[:, :b] = torch.randint(0, 256, (n, b), dtype=torch.uint8, device=DEV, generator=g)
    return d


class State:
    """What a server holds for a database and a batch: the handle, the keys where the entry
    point wants them, the answer buffer and the workspace."""

    def __init__(self, case, seed):
        self.case = case
        self.db = _records(case, seed)
        n, b, q = case["n"], case["b"], case["q"]
        stride = self.db.shape[1]
        self.handle = impir.impir_db_attach(self.db, n, b, stride)
        self.keys, offs = impir.pack_keys(_keys(case, seed))
        if case["entry"] != "answer":
            self.d_keys = torch.from_numpy(np.frombuffer(self.keys, np.uint8).copy()).to(DEV)
            self.d_off = torch.from_numpy(offs.view(np.int32).copy()).to(DEV)
            self.out = torch.zeros((q, b), dtype=torch.uint8, device=DEV)
            self.ws_bytes = impir.impir_workspace_bytes(q, stride)
            self.ws = torch.empty(self.ws_bytes, dtype=torch.uint8, device=DEV)

    def __del__(self):
        if getattr(self, "handle", None):
            impir.impir_db_free(self.handle)
            self.handle = None


def prepare(case, seed):
    return State(case, seed)


def run(state):
    c = state.case
    if c["entry"] == "answer":
        return impir.impir_answer(state.handle, state.keys, c["q"], c["b"])
    call = impir.impir_answer_async if c["entry"] == "async" else impir.impir_answer_add32_async
    call(state.handle, state.d_keys, state.d_off, c["q"], state.out, state.ws, state.ws_bytes,
         torch.cuda.current_stream())
    return state.out


def work(case):
    """Bytes: the records and keys once, the answers once. Operations: two PRF calls per inner
    node of every tree (160 byte substitutions and as many XORs each), and one operation per
    32-bit word of a record and query (half the records are selected: that many XORs; the
    additive answer multiplies and adds)."""
    n, b, q, m = case["n"], case["b"], case["q"], case["m"]
    cover = sum(min(n, 1 << max(1, m - d)) for d in range(case["dm"] + 1)) / (case["dm"] + 1)  # mean over the queries
    blocks = 2 * cover
    per_word = 2.0 if case["entry"] == "add32" else 0.5
    return {"bytes": float(n * b + q * (b + impir.impir_key_bytes(m))),
            "flops": q * (blocks * 320 + cover * b / 4 * per_word)}


# ---- the answers in plain torch ----

def _sbox():
    p, q, box = 1, 1, [0] * 256
    while True:
        p = (p ^ (p << 1) ^ (0x1B if p & 0x80 else 0)) & 0xFF
        q ^= q << 1
        q ^= q << 2
        q ^= q << 4
        q &= 0xFF
        if q & 0x80:
            q ^= 0x09
        rot = lambda v, k: ((v << k) | (v >> (8 - k))) & 0xFF
        box[p] = q ^ rot(q, 1) ^ rot(q, 2) ^ rot(q, 3) ^ rot(q, 4) ^ 0x63
        if p == 1:
            break
    box[0] = 0x63
    return box


def _aes(key, block):
    """AES-128 (FIPS-197) of (n, 16) blocks under (n, 16) or (1, 16) keys, uint8 on the device."""
    box = torch.tensor(_sbox(), dtype=torch.uint8, device=DEV)
    sub = lambda t: box.index_select(0, t.reshape(-1).int()).view(t.shape)
    dbl = lambda t: (t << 1) ^ ((t >> 7) * 0x1B)
    shift = torch.tensor([0, 5, 10, 15, 4, 9, 14, 3, 8, 13, 2, 7, 12, 1, 6, 11], device=DEV)
    k, s, rc = key.clone(), block ^ key, 1
    for r in range(1, 11):
        t = sub(k[:, [13, 14, 15, 12]])
        t[:, 0] ^= rc
        rc = (rc << 1) ^ (0x11B if rc & 0x80 else 0)
        w = k.view(-1, 4, 4).clone()
        w[:, 0] ^= t
        for i in range(1, 4):
            w[:, i] ^= w[:, i - 1]
        k = w.view(-1, 16)
        s = sub(s)[:, shift]
        if r < 10:
            a = s.view(-1, 4, 4)
            x = a[:, :, 0] ^ a[:, :, 1] ^ a[:, :, 2] ^ a[:, :, 3]
            s = (a ^ dbl(a ^ a[:, :, [1, 2, 3, 0]]) ^ x[:, :, None]).view(-1, 16)
        s = s ^ k
    return s


_FIXED = [b"IM-PIR MMO key 0", b"IM-PIR MMO key 1"]


def _leaves(key, cover):
    """The first `cover` leaves R(m, j) of a wire key, (cover, 16) uint8."""
    prf, m = key[1], key[2]
    cw = torch.from_numpy(np.frombuffer(key, np.uint8)[8:].copy()).to(DEV).view(2, 2, m + 1, 16)
    nodes = cw[0, 0, 0].view(1, 16)
    for d in range(1, m + 1):
        nodes = nodes[: (cover + (1 << (m - d + 1)) - 1) >> (m - d + 1)]  # parents of leaves below cover
        t = (nodes[:, 0] & 1).long()
        kids = []
        for x in (0, 1):
            if prf == 0:
                blk = torch.zeros_like(nodes)
                blk[:, 0] = x
                f = _aes(nodes, blk)
            else:
                fixed = torch.from_numpy(np.frombuffer(_FIXED[x], np.uint8).copy()).to(DEV).view(1, 16)
                f = _aes(fixed, nodes) ^ nodes
            kids.append(f ^ cw[t, x, d])
        nodes = torch.stack(kids, 1).view(-1, 16)
    return nodes[:cover]


def exact(case, seed):
    n, b, q = case["n"], case["b"], case["q"]
    if q * n > 1 << 24 or n * b > 1 << 30:
        return None
    db = _records(case, seed)[:, :b].contiguous()
    out = torch.zeros((q, b), dtype=torch.uint8, device=DEV)
    place = torch.arange(8, dtype=torch.uint8, device=DEV)
    for i, key in enumerate(_keys(case, seed)):
        leaves = _leaves(key, min(n, 1 << key[2]))
        if case["entry"] == "add32":
            share = leaves[:, :4].contiguous().view(torch.int32).long()
            share = -share if key[3] else share
            total = torch.zeros(b // 4, dtype=torch.int64, device=DEV)
            for lo in range(0, len(share), 1 << 16):
                words = db[lo: lo + (1 << 16)][: len(share) - lo].view(torch.int32).long()
                total += (words * share[lo: lo + (1 << 16), None]).sum(0)
            out[i] = (total & 0xFFFFFFFF).view(torch.uint8).view(-1, 8)[:, :4].reshape(-1)
        else:
            picked = db[: len(leaves)][(leaves[:, 0] & 1).bool()]
            odd = torch.zeros((b, 8), dtype=torch.int64, device=DEV)
            for lo in range(0, len(picked), 1 << 14):
                odd += ((picked[lo: lo + (1 << 14), :, None] >> place) & 1).sum(0, dtype=torch.int64)
            out[i] = ((odd & 1).to(torch.uint8) << place).sum(1, dtype=torch.uint8)
    return out.cpu().numpy() if case["entry"] == "answer" else out
