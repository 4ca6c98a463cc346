"""Pools that hold every vertex: the push form (TAURUS_FLAG_PUSH_FORM, or too little memory for the pull form) and the way back to it
when an allocation of the pull form fails."""
import os
import subprocess
import sys
from dataclasses import replace

import numpy as np
import pytest

import taurus_gen as tg
from gpu_harness import run_library
from test_gpu_parity import _full_check

pytestmark = pytest.mark.gpu
PUSH = 16


@pytest.mark.parametrize("mode,heads,dims", [(tg.SAGE_MEAN, 1, (24, 40, 7)), (tg.SAGE_MEAN, 1, (100, 48)), (tg.GCN_SYM, 1, (33, 130, 16)),
                                             (tg.GIN_SUM, 1, (16, 64, 47)), (tg.GAT, 1, (20, 64)), (tg.GAT, 4, (36, 128))])
@pytest.mark.parametrize("fanout", [0, 10])
@pytest.mark.parametrize("hubs", [0, 25])
@pytest.mark.parametrize("dense", [False, True])
def test_push_form(mode, heads, dims, fanout, hubs, dense):
    V = 4_001
    w = replace(tg.scaled(tg.WORKLOADS["mid"], V, chunk=600), dims=dims, fanout=(fanout,) + (0,) * (len(dims) - 2), pool_slots=V, hub_count=hubs,
                mode=mode, gat_heads=heads)
    lib, _ = _full_check(w, flags=PUSH, dense_output=dense)
    # both forms: the same integers, and a push of this form takes more launches
    g, model = tg.make_graph(w), tg.make_model(w, bias_scale=0.3)
    pull = run_library(w, g, model, tg.features(w.seed, 0, 0, V, dims[0]), dense_output=dense)
    assert pull["stats"] == lib["stats"] or [{k: v for k, v in s.items() if k != "scatter_groups"} for s in pull["stats"]] == \
        [{k: v for k, v in s.items() if k != "scatter_groups"} for s in lib["stats"]]
    assert pull["ctx"].launch_count() < lib["ctx"].launch_count()


def test_push_form_of_ragged_pushes():
    V = 4_001
    w = replace(tg.scaled(tg.WORKLOADS["mid"], V, chunk=600), dims=(24, 40), fanout=(0,), pool_slots=V, hub_count=25)
    g, model = tg.make_graph(w), tg.make_model(w, bias_scale=0.3)
    x0 = tg.features(w.seed, 0, 0, V, 24)
    chunks = [(s, min(s + 457, V)) for s in range(0, V, 457)]
    a, b = (run_library(w, g, model, x0, chunk_plan=chunks, flags=f) for f in (PUSH, 4))   # 4: every push in CSR order
    assert a["stats"] == b["stats"]
    assert np.linalg.norm(a["outs"][0] - b["outs"][0]) <= 1e-5 * np.linalg.norm(b["outs"][0])


FAILING_MALLOC = r"""
#define _GNU_SOURCE
#include <dlfcn.h>
#include <stddef.h>
static long calls = 0, fail_at = -1;
void arm(long n) { calls = 0; fail_at = n; }      /* call n (0 = the next one) reports that memory is exhausted, once */
long seen(void) { return calls; }
int cudaMalloc(void** p, size_t n) {
  static int (*real)(void**, size_t) = 0;
  if (!real) real = (int (*)(void**, size_t))dlsym(dlopen("libcudart.so.12", RTLD_LAZY | RTLD_NOLOAD), "cudaMalloc");   /* not in the global scope */
  if (calls++ == fail_at) { *p = 0; return 2; }   /* cudaErrorMemoryAllocation */
  return real(p, n);
}
"""

CHILD = r"""
import ctypes, sys
from dataclasses import replace
import numpy as np
import paper_2607_17374_b200 as tb
import taurus_gen as tg

shim = ctypes.CDLL(sys.argv[1])
fanout, dims = int(sys.argv[2]), tuple(int(d) for d in sys.argv[3].split("-"))
V = 1_500
w = replace(tg.scaled(tg.WORKLOADS["mid"], V, chunk=384), dims=dims, fanout=(fanout,), pool_slots=V, hub_count=0)
g, model = tg.make_graph(w), tg.make_model(w, bias_scale=0.3)
assert g.in_degree.max() > 256
x = tg.features(w.seed, 0, 0, V, dims[0])

def context():
    return tb.Context(V, g.E, g.row_ptr, g.col_idx, g.in_degree, w.mode, dims, model.W_neigh, model.W_self, model.bias, model.act, w.chunk,
                      V, 0, w.fanout, w.seed, 0, V)

def one_pass(ctx):
    ctx.layer_begin(0)
    n0 = ctx.launch_count()
    for s in range(0, V, w.chunk):
        ctx.push_chunk(s, min(s + w.chunk, V), np.ascontiguousarray(x[s:s + w.chunk]))
    pushes = ctx.launch_count() - n0
    ids, rows = np.empty(V, np.int64), np.empty((V, dims[1]), np.float32)
    assert ctx.drain_completed(ids, rows, V) == V
    ctx.layer_end()
    ctx.destroy()
    return rows[np.argsort(ids)], pushes

want, pull_launches = one_pass(context())
shim.arm(ctypes.c_long(-1))
ctx = context()
allocations = shim.seen()
ctx.destroy()
ended = []
for n in range(allocations):
    shim.arm(ctypes.c_long(n))
    try:
        ctx = context()
    except tb.TaurusError as e:
        assert e.code == tb.ERROR_CODES["NOMEM"], (n, str(e))
        ended.append(None)
        continue
    rows, launches = one_pass(ctx)
    assert np.linalg.norm(rows - want) <= 1e-5 * np.linalg.norm(want), n
    ended.append(launches)
first = next(i for i, k in enumerate(ended) if k is not None)
# before the form is chosen nothing helps; behind it every failed allocation leads to the push form
assert all(k is not None and k > pull_launches for k in ended[first:]), (first, ended)
assert len(ended) - first >= 12, ended
print("fell back", len(ended) - first)
"""


@pytest.mark.parametrize("fanout,dims", [(0, "24-40"), (10, "24-40"), (0, "40-24")])
def test_a_failed_allocation_leads_to_the_push_form(tmp_path, fanout, dims):
    (tmp_path / "shim.c").write_text(FAILING_MALLOC)
    shim = str(tmp_path / "shim.so")
    subprocess.check_call(["gcc", "-O1", "-shared", "-fPIC", "-o", shim, str(tmp_path / "shim.c"), "-ldl"])
    root = os.path.dirname(os.path.dirname(os.path.abspath(__file__)))
    r = subprocess.run([sys.executable, "-c", CHILD, shim, str(fanout), dims], cwd=root, capture_output=True, text=True, timeout=600,
                       env=dict(os.environ, LD_PRELOAD=shim))
    assert r.returncode == 0 and "fell back" in r.stdout, r.stdout[-2000:] + r.stderr[-3000:]
