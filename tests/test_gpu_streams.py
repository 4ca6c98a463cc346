"""Calls of one context on several streams: what a caller puts on the stream of a layer that has ended is over before a layer begun on another stream
reads or writes anything; pushes in turn on two streams, rows from the host or from the device; what stands in front of a launch that may come up early."""
import os
import subprocess
import sys
from dataclasses import replace

import pytest

import taurus_gen as tg
from gpu_harness import row_error, run_oracle

pytestmark = pytest.mark.gpu


def _context(w, g, flags=0):
    import paper_2607_17374_b200 as tb
    m = tg.make_model(w, bias_scale=0.3)
    return m, tb.Context(g.V, g.E, g.row_ptr, g.col_idx, g.in_degree, w.mode, w.dims, m.W_neigh, m.W_self, m.bias, m.act, w.chunk, w.pool_slots, w.hub_count, w.fanout,
                         w.seed, 0, 2 * g.V, 0, flags, 0, w.gin_eps)


@pytest.mark.parametrize("dims", [(64, 64, 32), (20, 72, 40)])
def test_work_between_two_layers_on_the_stream_of_the_first(dims):
    """The caller writes the second layer's input on the first one's stream, behind a kernel that takes its time."""
    import torch
    V, chunk = 5_000, 1_024
    w = replace(tg.scaled(tg.WORKLOADS["large"], V, chunk=chunk), dims=dims, fanout=(0, 0), pool_slots=V, hub_count=5)
    g = tg.make_graph(w)
    m, ctx = _context(w, g)
    x0 = tg.features(w.seed, 0, 0, V, dims[0])
    want = run_oracle(w, g, m, x0)["outs"][1]
    x = torch.from_numpy(x0).cuda()
    first, second = torch.cuda.Stream(), torch.cuda.Stream()
    raw, between, out = (torch.empty(V, d, device="cuda") for d in (dims[1], dims[1], dims[2]))
    for _ in range(3):
        between.fill_(float("nan"))
        torch.cuda.synchronize()
        for l, (src, dst, st) in enumerate(((x, raw, first), (between, out, second))):
            ctx.layer_begin(l, st)
            ctx.layer_set_dense_output(dst, dst.shape[1])
            for b in range(0, V, chunk):
                ctx.push_chunk(b, min(b + chunk, V), src[b:b + chunk], st)
            assert ctx.layer_end()["completed"] == V
            if l == 0:
                with torch.cuda.stream(first):
                    torch.cuda._sleep(20_000_000)   # some 10 ms
                    between.copy_(raw)
        assert row_error(out.cpu().numpy(), want)[0] <= 1e-4


@pytest.mark.parametrize("rows", ["pinned", "device"])
@pytest.mark.parametrize("push_form", [False, True])
@pytest.mark.parametrize("mode,dims", [(tg.GIN_SUM, (32, 64)), (tg.GIN_SUM, (64, 32)), (tg.SAGE_MEAN, (33, 72))])
def test_pushes_in_turn_on_two_streams(mode, dims, push_form, rows):
    """(GIN 32 -> 64 in the push form scatters the caller's rows in place: no kernel of the push stands in front of its first one.)"""
    import torch
    import paper_2607_17374_b200 as tb
    V, chunk = 6_000, 500
    w = replace(tg.scaled(tg.WORKLOADS["large"], V, chunk=chunk), dims=dims, fanout=(0,), pool_slots=V, hub_count=9, mode=mode)
    g = tg.make_graph(w)
    m, ctx = _context(w, g, tb.FLAG_PUSH_FORM if push_form else 0)
    x0 = tg.features(w.seed, 0, 0, V, dims[0])
    want = run_oracle(w, g, m, x0)["outs"][0]
    x = torch.from_numpy(x0).pin_memory() if rows == "pinned" else torch.from_numpy(x0).cuda()
    streams = [torch.cuda.Stream(), torch.cuda.Stream()]
    out = torch.empty(V, dims[1], device="cuda")
    for _ in range(3):
        out.fill_(float("nan"))
        torch.cuda.synchronize()
        ctx.layer_begin(0, streams[0])
        ctx.layer_set_dense_output(out, dims[1])
        for i, b in enumerate(range(0, V, chunk)):
            ctx.push_chunk(b, b + chunk, x[b:b + chunk], streams[i & 1])
        assert ctx.layer_end()["completed"] == V
        assert row_error(out.cpu().numpy(), want)[0] <= 1e-4


SHIM = r"""
#define _GNU_SOURCE
#include <dlfcn.h>
#include <cuda_runtime_api.h>
/* What came last on every stream, and launches that may come up early right behind a wait for an event. */
static struct { cudaStream_t stream; int waited; } seen[256];
static int streams = 0;
static long early = 0, behind_wait = 0;
static void* real(const char* name) { return dlsym(dlopen("libcudart.so.12", RTLD_LAZY | RTLD_NOLOAD), name); }
static int* waited(cudaStream_t s) {
  int i = 0;
  while (i < streams && seen[i].stream != s) ++i;
  if (i == streams && streams < 255) seen[streams++].stream = s;
  return &seen[i].waited;
}
long early_launches(void) { return early; }
long early_behind_a_wait(void) { return behind_wait; }
cudaError_t cudaStreamWaitEvent(cudaStream_t s, cudaEvent_t e, unsigned flags) {
  static cudaError_t (*f)(cudaStream_t, cudaEvent_t, unsigned) = 0;
  if (!f) f = real("cudaStreamWaitEvent");
  *waited(s) = 1;
  return f(s, e, flags);
}
cudaError_t cudaLaunchKernel(const void* k, dim3 g, dim3 b, void** a, size_t m, cudaStream_t s) {
  static cudaError_t (*f)(const void*, dim3, dim3, void**, size_t, cudaStream_t) = 0;
  if (!f) f = real("cudaLaunchKernel");
  *waited(s) = 0;
  return f(k, g, b, a, m, s);
}
cudaError_t cudaLaunchKernelExC(const cudaLaunchConfig_t* c, const void* k, void** a) {
  static cudaError_t (*f)(const cudaLaunchConfig_t*, const void*, void**) = 0;
  if (!f) f = real("cudaLaunchKernelExC");
  for (unsigned i = 0; i < c->numAttrs; ++i)
    if (c->attrs[i].id == cudaLaunchAttributeProgrammaticStreamSerialization && c->attrs[i].val.programmaticStreamSerializationAllowed) {
      ++early;
      behind_wait += *waited(c->stream);
    }
  *waited(c->stream) = 0;
  return f(c, k, a);
}
"""

CHILD = r"""
import ctypes, sys
from dataclasses import replace
import torch
import paper_2607_17374_b200 as tb
import taurus_gen as tg

shim = ctypes.CDLL(sys.argv[1])
V, chunk = 4_000, 400
for mode, dims in ((tg.GIN_SUM, (32, 64)), (tg.GIN_SUM, (64, 32)), (tg.SAGE_MEAN, (33, 72)), (tg.GCN_SYM, (64, 40)), (tg.GAT, (64, 32))):
    for pool in (V, 3_000):
        for flags in (0, tb.FLAG_PUSH_FORM) if pool == V else (0,):
            for pinned in (False, True):
                for output in ("drain", "device", "pinned"):
                    w = replace(tg.scaled(tg.WORKLOADS["large"], V, chunk=chunk), dims=dims, fanout=(0,), pool_slots=pool, hub_count=9, mode=mode)
                    g, m = tg.make_graph(w), tg.make_model(w, bias_scale=0.3)
                    ctx = tb.Context(V, g.E, g.row_ptr, g.col_idx, g.in_degree, w.mode, w.dims, m.W_neigh, m.W_self, m.bias, m.act, chunk, pool, 9, w.fanout, w.seed,
                                     0 if pool == V else V, 2 * V, 0, flags, 0, w.gin_eps, m.att_src, m.att_dst, w.leaky_slope, w.gat_heads)
                    x = torch.zeros(V, dims[0])
                    x = x.pin_memory() if pinned else x.cuda()
                    out = torch.empty(V, dims[1])
                    out = out.pin_memory() if output == "pinned" else out.cuda()
                    streams = [torch.cuda.Stream(), torch.cuda.Stream()]
                    ctx.layer_begin(0, streams[0])
                    if mode == tg.GAT:
                        hp = torch.zeros(V, dims[1], device="cuda")
                        for b in range(0, V, chunk):
                            ctx.gat_project_chunk(b, b + chunk, x[b:b + chunk], hp[b:b + chunk], dims[1], streams[0])
                        ctx.gat_attention(streams[0])
                        x = torch.zeros(V, dims[1]).pin_memory() if pinned else hp
                    if output != "drain":
                        ctx.layer_set_dense_output(out, dims[1])
                    for i, b in enumerate(range(0, V, chunk)):
                        before = shim.early_behind_a_wait()
                        ctx.push_chunk(b, b + chunk, x[b:b + chunk], streams[i // 2 & 1])
                        assert shim.early_behind_a_wait() == before, (mode, dims, pool, flags, pinned, output, i)
                        if output == "drain":
                            ctx.drain_dense(out, dims[1], V)
                    assert ctx.layer_end()["completed"] == V
                    assert shim.early_behind_a_wait() == 0, (mode, dims, pool, flags, pinned, output)
print("early", shim.early_launches())
"""


def test_no_early_launch_right_behind_a_wait_of_the_library(tmp_path):
    """A kernel that may come up while the one before it on the stream still runs has a kernel in front of it.  Launches and waits are counted by a
    library in front of the CUDA runtime, in a process of its own."""
    (tmp_path / "shim.c").write_text(SHIM)
    shim = str(tmp_path / "shim.so")
    subprocess.check_call(["gcc", "-O1", "-shared", "-fPIC", "-I", "/usr/local/cuda/include", "-o", shim, str(tmp_path / "shim.c"), "-ldl"])
    root = os.path.dirname(os.path.dirname(os.path.abspath(__file__)))
    r = subprocess.run([sys.executable, "-c", CHILD, shim], cwd=root, capture_output=True, text=True, timeout=600, env=dict(os.environ, LD_PRELOAD=shim))
    assert r.returncode == 0 and int(r.stdout.split()[-1]) > 100, r.stdout[-2000:] + r.stderr[-3000:]
