"""A wait that runs out inside the tensor-core kernel reaches the caller as an error, on every path
that can launch it. The debug library shortens the limit to a microsecond, so that a CTA's first wait
gives up while the nodes it waits for are computed; the kernel then returns by itself and the next call
with the usual limit answers rightly."""
import os
import subprocess
import sys

import pytest

pytestmark = pytest.mark.gpu

ROOT = os.path.dirname(os.path.dirname(os.path.abspath(__file__)))

COMMON = r'''
import os
import numpy as np
import torch
import paper_2509_06514_gb300 as impir
from paper_2509_06514_gb300 import workloads

assert impir.BOUNDS
N, B = 1 << 20, 64
db = workloads.make_db(N, B, seed=3)
key = impir.dpf_gen(7, 18, 0, bytes(range(32)))[0]
wide = impir.dpf_gen(N - 1, 20, 0, bytes(range(32)))[0]
keys = [key] * 512 + [wide] * 4
blob, offs = impir.pack_keys(keys)
n = len(keys)


def short():
    os.environ["IMPIR_BOUNDS_TEST_WAIT_NS"] = "1000"


def usual():
    del os.environ["IMPIR_BOUNDS_TEST_WAIT_NS"]


def refused(f):
    short()
    try:
        f()
    except impir.ImpirError as e:
        assert e.status == impir.IMPIR_ECUDA and "a wait" in str(e), e
    else:
        raise SystemExit("the wait that ran out was not reported")
    usual()
'''

STREAMED = r'''
# 2^16, then 2^18 records a chunk: the second chunk alone has the 608 units the tensor-core kernel takes,
# and its schedule's header is used again two chunks later
call = lambda: impir.impir_answer_streamed(db, N, B, blob, n, 16 << 20)[0]
want = call()
refused(call)
assert np.array_equal(call(), want)
h = impir.impir_db_load(db, N, B)
assert np.array_equal(impir.impir_answer(h, blob, n, B), want)
impir.impir_db_free(h)
'''


@pytest.fixture(scope="module")
def bounds_lib():
    from paper_2509_06514_gb300 import build
    return build.build(bounds=True)


def run(code):
    r = subprocess.run([sys.executable, "-c", COMMON + code + "\nprint('REPORTED')"], cwd=ROOT, capture_output=True,
                       text=True, timeout=300, env=dict(os.environ, IMPIR_BOUNDS="1"))
    assert r.returncode == 0 and "REPORTED" in r.stdout, r.stdout[-3000:] + r.stderr[-3000:]


SMALL = r"""
def no_tables(f):
    os.environ["IMPIR_BOUNDS_TEST_NO_TABLES"] = "1"
    try:
        f()
    except impir.ImpirError as e:
        assert e.status == impir.IMPIR_ECUDA and "not valid" in str(e), e
    else:
        raise SystemExit("the kernel that did not run was not reported")
    del os.environ["IMPIR_BOUNDS_TEST_NO_TABLES"]


# one query, three, and enough that the header comes back in a copy of its own; padded records too
for B in (64, 40):
    d = np.ascontiguousarray(db[: 1 << 18, :B])
    h = impir.impir_db_load(d, 1 << 18, B)
    for n in (1, 3, 63, 4000):
        blob, _ = impir.pack_keys([key] * n)
        for call in (impir.impir_answer, impir.impir_answer_add32):
            no_tables(lambda: call(h, blob, n, B))
            got = call(h, blob, n, B)
            assert (got == got[0]).all() and got.any()
    blob, _ = impir.pack_keys([key] * 3)
    impir.impir_set_config(h, lane_bits=4, queries_per_warp=1, queries_per_launch=1)
    no_tables(lambda: impir.impir_answer(h, blob, 3, B))
    impir.impir_db_free(h)
"""


ASYNC = r"""
d_db = torch.from_numpy(db).cuda()
d_keys = torch.from_numpy(np.frombuffer(blob, np.uint8).copy()).cuda()
d_off = torch.from_numpy(offs.view(np.int32).copy()).cuda()
out = torch.zeros((n, B), dtype=torch.uint8, device="cuda")


def noalloc():
    impir.impir_answer_noalloc(d_db, N, B, B, d_keys, d_off, n, out, None)
    assert impir.impir_noalloc_status() == (0, 0xFFFFFFFF)


try:
    impir.impir_noalloc_status()
    raise SystemExit("a status without a call")
except impir.ImpirError as e:
    assert e.status == impir.IMPIR_EINVAL
noalloc()
want = out.clone()
refused(noalloc)
noalloc()
assert torch.equal(out, want)

h = impir.impir_db_attach(d_db, N, B, B)
wsb = impir.impir_workspace_bytes(n, B)
ws = torch.empty(wsb, dtype=torch.uint8, device="cuda")


def resident():
    impir.impir_answer_async(h, d_keys, d_off, n, out, ws, wsb, None)
    impir.impir_workspace_status(ws)


refused(resident)
resident()
assert torch.equal(out, want)
refused(lambda: impir.impir_answer(h, blob, n, B))
assert np.array_equal(impir.impir_answer(h, blob, n, B), want.cpu().numpy())
impir.impir_db_free(h)
"""


def test_noalloc_and_workspace_status_report_it(bounds_lib):
    run(ASYNC)


def test_every_synchronous_call_reports_a_kernel_that_did_not_run(bounds_lib):
    run(SMALL)


def test_streamed_answers_report_a_wait_of_any_chunk(bounds_lib):
    run(STREAMED)
