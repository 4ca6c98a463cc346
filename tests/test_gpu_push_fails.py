"""A push that fails half way on the host: the context says so until the layer is begun again, and the next pass over it is as if
nothing had happened.  The failures are return codes of a stand-in for cudaStreamWaitEvent, in a process of its own."""
import os
import subprocess
import sys

import pytest

pytestmark = pytest.mark.gpu

SHIM = r"""
#define _GNU_SOURCE
#include <dlfcn.h>
static long calls = 0, fail_at = -1;
void arm(long n) { calls = 0; fail_at = n; }      /* call n (0 = the next one) is refused, once */
long seen(void) { return calls; }
int cudaStreamWaitEvent(void* stream, void* event, unsigned flags) {
  static int (*real)(void*, void*, unsigned) = 0;
  if (!real) real = (int (*)(void*, void*, unsigned))dlsym(dlopen("libcudart.so.12", RTLD_LAZY | RTLD_NOLOAD), "cudaStreamWaitEvent");
  return calls++ == fail_at ? 1 : real(stream, event, flags);   /* cudaErrorInvalidValue */
}
"""

CHILD = r"""
import ctypes, sys
from dataclasses import replace
import numpy as np
import paper_2607_17374_b200 as tb
import taurus_gen as tg

shim = ctypes.CDLL(sys.argv[1])
pool, mode, dims = int(sys.argv[2]), int(sys.argv[3]), tuple(int(d) for d in sys.argv[4].split("-"))
V = 1_500
w = replace(tg.scaled(tg.WORKLOADS["mid"], V, chunk=64), dims=dims, fanout=(0,), pool_slots=pool, hub_count=0, mode=mode)
g, model = tg.make_graph(w), tg.make_model(w, bias_scale=0.3)
x = tg.features(w.seed, 0, 0, V, dims[0])
ctx = tb.Context(V, g.E, g.row_ptr, g.col_idx, g.in_degree, w.mode, dims, model.W_neigh, model.W_self, model.bias, model.act, w.chunk, pool, 0,
                 w.fanout, w.seed, 0 if pool >= V else V, V)
chunks = [(s, min(s + w.chunk, V)) for s in range(0, V, w.chunk)]

def one_pass(begun=False):
    if not begun:
        ctx.layer_begin(0)
    for s, e in chunks:
        ctx.push_chunk(s, e, np.ascontiguousarray(x[s:e]))
    ids, rows = np.empty(V, np.int64), np.empty((V, dims[1]), np.float32)
    assert ctx.drain_completed(ids, rows, V) == V
    return rows[np.argsort(ids)], ctx.layer_end()

def check(got):
    assert np.linalg.norm(got[0] - want[0]) <= 1e-5 * np.linalg.norm(want[0])
    assert got[1] == want[1]

shim.arm(ctypes.c_long(-1))
want = one_pass()
waits = shim.seen()
assert waits > len(chunks)
refused = retried = 0
for n in list(range(0, 12)) + list(range(12, waits, max(1, waits // 25))):
    ctx.layer_begin(0)
    shim.arm(ctypes.c_long(n))
    failed = None
    try:
        for i, (s, e) in enumerate(chunks):
            ctx.push_chunk(s, e, np.ascontiguousarray(x[s:e]))
        i = None
        ids, rows = np.empty(V, np.int64), np.empty((V, dims[1]), np.float32)
        ctx.drain_completed(ids, rows, V)
    except tb.TaurusError as err:
        failed = err.code
    shim.arm(ctypes.c_long(-1))
    assert failed == tb.ERROR_CODES["CUDA"], (n, failed)
    # either nothing of the chunk was enqueued and the same push goes through, or every later call says that the layer is lost
    try:
        if i is not None:
            for s, e in chunks[i:]:
                ctx.push_chunk(s, e, np.ascontiguousarray(x[s:e]))
        ids, rows = np.empty(V, np.int64), np.empty((V, dims[1]), np.float32)
        count = ctx.drain_completed(ids, rows, V)
        assert count == V
        check((rows[np.argsort(ids)], ctx.layer_end()))
        retried += 1
    except tb.TaurusError as err:
        assert err.code == tb.ERROR_CODES["CUDA"], (n, err)
        for call in (ctx.get_stats, ctx.layer_end, lambda: ctx.push_chunk(*chunks[i or 0], np.ascontiguousarray(x[:64]))):
            try:
                call()
            except tb.TaurusError as again:
                assert again.code in (tb.ERROR_CODES["CUDA"], tb.ERROR_CODES["ORDER"]), (n, again)
            else:
                raise AssertionError("a call went through after push %s" % i)
        refused += 1
    check(one_pass())
assert refused > 0
print("refused", refused, "retried", retried)
"""


@pytest.mark.parametrize("pool,mode,dims", [(1_500, 0, "24-40"), (1_500, 0, "40-24"), (1_500, 1, "40-24"), (1_450, 0, "40-24"), (1_450, 0, "24-40")])
def test_a_failed_push_is_not_forgotten(tmp_path, pool, mode, dims):
    (tmp_path / "shim.c").write_text(SHIM)
    shim = str(tmp_path / "shim.so")
    subprocess.check_call(["gcc", "-O1", "-shared", "-fPIC", "-o", shim, str(tmp_path / "shim.c"), "-ldl"])
    root = os.path.dirname(os.path.dirname(os.path.abspath(__file__)))
    r = subprocess.run([sys.executable, "-c", CHILD, shim, str(pool), str(mode), dims], cwd=root, capture_output=True, text=True, timeout=600,
                       env=dict(os.environ, LD_PRELOAD=shim))
    assert r.returncode == 0 and "refused" in r.stdout, r.stdout[-2000:] + r.stderr[-3000:]
