"""Where an asynchronous answer may be accumulated in the caller's buffer, and where it may not: padded
records, unaligned or host memory, and answers laid over the call's own inputs, which must have been read
first. The answers are the same everywhere; the number of kernels launched tells the two ways apart."""
import numpy as np
import pytest

import paper_2509_06514_gb300 as impir

pytestmark = pytest.mark.gpu

N, Q = 5000, 20


class Case:
    """Inputs in one device buffer each, so that answers can be laid over them."""

    def __init__(self, B, add, cfg=None):
        import torch
        self.torch, self.B, self.add = torch, B, add
        self.stride = (B + 15) // 16 * 16
        g = torch.Generator(device="cuda").manual_seed(B)
        self.db = torch.zeros((N, self.stride), dtype=torch.uint8, device="cuda")
        self.db[:, :B] = torch.randint(0, 256, (N, B), dtype=torch.uint8, device="cuda", generator=g)
        self.h = impir.impir_db_attach(self.db, N, B, self.stride)
        if cfg:
            impir.impir_set_config(self.h, **cfg)
        keys = [impir.dpf_gen(i * 211 % N, 13, i % 2, bytes([i] * 32))[i % 2] for i in range(Q)]
        blob, offs = impir.pack_keys(keys)
        self.keys = np.frombuffer(blob, np.uint8).copy()
        self.offs = offs.view(np.uint8).copy()
        self.wsb = impir.impir_workspace_bytes(Q, self.stride)
        self.ws = torch.empty(self.wsb, dtype=torch.uint8, device="cuda")

    def room(self, data):
        """A device copy of data, with room for the batch's answers behind its first bytes."""
        t = self.torch.zeros(max(data.size, Q * self.B) + 64, dtype=self.torch.uint8, device="cuda")
        t[:data.size] = self.torch.from_numpy(data)
        return t

    def answer(self, out, d_keys=None, d_off=None):
        """Launches of the answer (as the library counts them) into device pointer `out`."""
        d_keys = self.room(self.keys) if d_keys is None else d_keys
        d_off = self.room(self.offs) if d_off is None else d_off
        impir.impir_timing_enable(True)
        call = impir.impir_answer_add32_async if self.add else impir.impir_answer_async
        call(self.h, d_keys.data_ptr(), d_off.data_ptr(), Q, out, self.ws, self.wsb, None)
        self.torch.cuda.synchronize()
        n = impir.impir_timing_read()[2]
        impir.impir_timing_enable(False)
        return n

    def apart(self):
        """(launches, answers, the 64 bytes behind them): answers, keys and offsets in a row in one buffer."""
        k_at = Q * self.B + 64
        o_at = k_at + (self.keys.size + 15) // 16 * 16
        buf = self.torch.full((o_at + self.offs.size,), 0xA5, dtype=self.torch.uint8, device="cuda")
        buf[k_at:k_at + self.keys.size] = self.torch.from_numpy(self.keys)
        buf[o_at:] = self.torch.from_numpy(self.offs)
        n = self.answer(buf.data_ptr(), d_keys=buf[k_at:], d_off=buf[o_at:])
        return n, self.get(buf), buf[Q * self.B:k_at].cpu().numpy()

    def new_out(self):
        return self.torch.full((Q * self.B + 64,), 0xA5, dtype=self.torch.uint8, device="cuda")

    def get(self, t, at=0):
        return t[at:at + Q * self.B].cpu().numpy()


@pytest.mark.parametrize("add", [False, True])
@pytest.mark.parametrize("B", [64, 4096])
def test_in_place_and_not(B, add):
    c = Case(B, add)
    try:
        n, want, edge = c.apart()
        assert n == 2 and (edge == 0xA5).all()
        for at in (4, 8):                                              # unaligned
            out = c.new_out()
            assert c.answer(out.data_ptr() + at) == 3
            assert np.array_equal(c.get(out, at), want)
            edge = out[Q * B + at:].cpu().numpy()
            assert (out[:at].cpu().numpy() == 0xA5).all() and (edge == 0xA5).all()
        pinned = c.torch.zeros(Q * B, dtype=c.torch.uint8, pin_memory=True)
        assert c.answer(pinned.data_ptr()) == 3                        # host memory that the device can write
        assert np.array_equal(pinned.numpy(), want)
        k = c.room(c.keys)
        assert c.answer(k.data_ptr(), d_keys=k) == 3                   # over the keys
        assert np.array_equal(c.get(k), want)
        k = c.room(c.keys)
        assert c.answer(k.data_ptr() + 32, d_keys=k) == 3              # inside them
        assert np.array_equal(c.get(k, 32), want)
        o = c.room(c.offs)
        assert c.answer(o.data_ptr(), d_off=o) == 3                    # over the offsets
        assert np.array_equal(c.get(o), want)
        assert c.answer(c.db.data_ptr() + 48 * B) == 3                 # over records (which it then replaces)
        assert np.array_equal(c.db.view(-1)[48 * B:(48 + Q) * B].cpu().numpy(), want)
    finally:
        impir.impir_db_free(c.h)


def test_an_input_behind_the_keys_bounds_them():
    """Keys, offsets and answers one after the other in one buffer: nothing overlaps."""
    c = Case(64, False)
    try:
        kb, ob = c.keys.size, c.offs.size
        o_at = (kb + 15) // 16 * 16
        out_at = (o_at + ob + 15) // 16 * 16
        buf = c.torch.zeros(out_at + Q * 64, dtype=c.torch.uint8, device="cuda")
        buf[:kb] = c.torch.from_numpy(c.keys)
        buf[o_at:o_at + ob] = c.torch.from_numpy(c.offs)
        assert c.answer(buf.data_ptr() + out_at, d_keys=buf, d_off=buf[o_at:]) == 2
        assert np.array_equal(c.get(buf, out_at), c.apart()[1])
    finally:
        impir.impir_db_free(c.h)


def test_padded_records_and_one_query_launches():
    c = Case(40, False)
    try:
        n, want, edge = c.apart()
        assert n == 3 and (edge == 0xA5).all()
        k = c.room(c.keys)
        assert c.answer(k.data_ptr(), d_keys=k) == 3
        assert np.array_equal(c.get(k), want)
    finally:
        impir.impir_db_free(c.h)
    # one launch per query, answers over the keys: a key lies at or behind its own answer's place
    c = Case(64, False, dict(lane_bits=3, queries_per_warp=1, queries_per_launch=1))
    try:
        n, want, _ = c.apart()
        assert n == 2 * Q
        k = c.room(c.keys)
        assert c.answer(k.data_ptr(), d_keys=k) == 3 * Q
        assert np.array_equal(c.get(k), want)
    finally:
        impir.impir_db_free(c.h)
