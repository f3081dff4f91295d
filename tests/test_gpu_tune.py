"""A tuned shape is launched as the tuner timed it, tensor-core kernel or not, from a fresh tuning and
from a saved cache."""
import numpy as np
import pytest

import paper_2509_06514_gb300 as impir

N, B, Q = 1 << 18, 512, 128


def line(cols, path):
    path.write_text(" ".join(str(c) for c in cols) + "\n")
    return str(path)


def saved(path):
    impir.impir_tune_cache_save(str(path))
    return [ln.split() for ln in path.read_text().splitlines() if not ln.startswith("#")]


def test_cache_keeps_the_choice_of_kernels(tmp_path):
    from paper_2509_06514_gb300 import build
    build.build()
    assert impir.impir_tune_cache_load(line([7, 1 << 20, 256, 64, 5, 8, 16, 0, 1], tmp_path / "a")) == 1
    assert impir.impir_tune_cache_load(line([7, 1 << 20, 256, 96, 5, 8, 16, 0], tmp_path / "b")) == 1
    rows = saved(tmp_path / "c")
    assert "7 1048576 256 64 5 8 16 0 1".split() in rows and "7 1048576 256 96 5 8 16 0".split() in rows


class Batch:
    def __init__(self):
        import torch
        self.db = torch.randint(0, 256, (N, B), dtype=torch.uint8, device="cuda")
        self.h = impir.impir_db_attach(self.db, N, B, B)
        keys = [impir.dpf_gen(i * 977 % N, 18, 0, bytes([i] * 32))[0] for i in range(Q)]
        blob, offs = impir.pack_keys(keys)
        self.keys = torch.from_numpy(np.frombuffer(blob, np.uint8).copy()).cuda()
        self.off = torch.from_numpy(offs.view(np.int32).copy()).cuda()
        self.out = torch.zeros((Q, B), dtype=torch.uint8, device="cuda")
        self.wsb = impir.impir_workspace_bytes(Q, B)
        self.ws = torch.empty(self.wsb, dtype=torch.uint8, device="cuda")
        self.args = (self.h, self.keys, self.off, Q, self.out, self.ws, self.wsb, torch.cuda.current_stream())

    def tuned(self):
        return impir.impir_autotune(*self.args)

    def answer(self, n=None):
        """The answers, and the units of the tensor-core kernel (header bytes 48 to 55)."""
        args = self.args if n is None else self.args[:3] + (n,) + self.args[4:]
        impir.impir_answer_async(*args)
        return self.out.cpu().numpy().copy(), int(self.ws[48:56].cpu().numpy().view("<u8")[0])


@pytest.mark.gpu
def test_tuned_batches_run_what_was_timed(tmp_path):
    b = Batch()
    sms = impir.impir_device_sm_count()
    try:
        want, units = b.answer()
        assert units == N // 1024
        key = [sms, N, B, Q]
        for extra, expect in (([1], 0), ([], N // 1024)):
            assert impir.impir_tune_cache_load(line(key + [4, 4, 16, 0] + extra, tmp_path / "t")) == 1
            assert b.tuned().as_dict() == dict(lane_bits=4, queries_per_warp=4, warps_per_cta=16, queries_per_launch=0)
            got, units = b.answer()
            assert units == expect and np.array_equal(got, want)
            assert b.answer(Q - 1)[1] == N // 1024      # a batch size that was not timed: the default rule
        impir.impir_set_config(b.h, lane_bits=4, queries_per_warp=4)     # set, not tuned: as it is
        got, units = b.answer()
        assert units == 0 and np.array_equal(got, want)
    finally:
        impir.impir_db_free(b.h)


@pytest.mark.gpu
def test_a_fresh_tuning_says_what_it_chose(tmp_path):
    global Q
    Q = 130    # a batch size that no other test tunes
    b = Batch()
    try:
        want, _ = b.answer()
        c = b.tuned().as_dict()
        row = [r for r in saved(tmp_path / "s") if r[1:4] == [str(N), str(B), str(Q)]][0]
        assert [int(x) for x in row[4:8]] == list(c.values())
        got, units = b.answer()
        assert np.array_equal(got, want) and (units > 0) == (len(row) == 8)
    finally:
        impir.impir_db_free(b.h)
        Q = 128
