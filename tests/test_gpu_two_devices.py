"""What belongs to a device is kept by the context, not by the process: a context on a device whose kernels have no limits raised yet
has to raise them itself.  One device is enough to show it: in a process of its own, `cudaDeviceReset` between two contexts leaves
the second one with a device that has forgotten what the first one set."""
import os
import subprocess
import sys

import pytest

pytestmark = pytest.mark.gpu

CHILD = r"""
import ctypes
from dataclasses import replace
import numpy as np
import paper_2607_17374_b200 as tb
import taurus_gen as tg

width, hubs, pool = (int(a) for a in __import__("sys").argv[1:4])
w = replace(tg.scaled(tg.WORKLOADS["tiny"], 3_000, chunk=64), dims=(width, width), fanout=(0,), mode=tg.SAGE_MEAN)
g, model = tg.make_graph(w), tg.make_model(w, bias_scale=0.3)
x = tg.features(w.seed, 0, 0, g.V, width)

def one_pass():
    ctx = tb.Context(g.V, g.E, g.row_ptr, g.col_idx, g.in_degree, w.mode, w.dims, model.W_neigh, model.W_self, model.bias, model.act, w.chunk,
                     pool, hubs, w.fanout, w.seed, 0 if pool >= g.V else g.V, g.V)
    ctx.layer_begin(0)
    for s in range(0, g.V, w.chunk):
        ctx.push_chunk(s, min(s + w.chunk, g.V), np.ascontiguousarray(x[s:s + w.chunk]))
    ids, rows = np.empty(g.V, np.int64), np.empty((g.V, width), np.float32)
    assert ctx.drain_completed(ids, rows, g.V) == g.V
    ctx.layer_end()
    ctx.destroy()
    return rows[np.argsort(ids)]

first = one_pass()
assert ctypes.CDLL("libcudart.so.12").cudaDeviceReset() == 0
second = one_pass()
assert np.linalg.norm(first - second) <= 1e-5 * np.linalg.norm(first)
print("same rows")
"""


@pytest.mark.parametrize("width,hubs,pool", [(48, 0, 3_000), (1_024, 0, 3_000), (64, 5, 2_200)])   # rings of 16 KB and 66 KB; row transfers
def test_second_context_after_the_device_forgot(width, hubs, pool):
    root = os.path.dirname(os.path.dirname(os.path.abspath(__file__)))
    r = subprocess.run([sys.executable, "-c", CHILD, str(width), str(hubs), str(pool)], cwd=root, capture_output=True, text=True, timeout=300)
    assert r.returncode == 0 and "same rows" in r.stdout, r.stdout[-2000:] + r.stderr[-2000:]
