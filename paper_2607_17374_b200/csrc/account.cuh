// The accounting of a push to a pool that holds every vertex, as code that a block of any kernel can run: kernels of its own
// (kernels_resident.cu) for large pushes, whose blocks run beside the projection of the rows on a stream of their own, and the first blocks of
// the launch that writes the rows for small ones, which are bound by launches and by the events between two streams.
#pragma once

#include "block_exit.h"
#include "taurus_internal.h"

#define FULL 0xffffffffu

// Items of a grid chunk: every vertex the chunk can touch, in ascending order, each once: destinations of the chunk's edges
// (begin, count: their entries in the destination's in-list) and the chunk's own vertices (self message; the count may
// be zero).  No two items share a vertex, so nothing here needs an atomic or an epoch stamp.
struct Items { const int32_t* v; const uint32_t* begin; const int32_t* count; };

struct AccountWork {
  ChunkArgs a;
  Items it;
  long long i0, n_items;       // the chunk's items
  const uint32_t* cmask;       // sampled layers: kept entries of the in-lists
  int4* heavy;                 // segments of long in-lists, NULL: none
  int32_t* heavy_left;
  int blocks;                  // blocks of the launch that do it
};

namespace {

__device__ __forceinline__ int rl() { return threadIdx.x & 31; }
// The first THREADS threads of a block (which may have more; they have gone).  It waits for that many, so none of them leaves early by itself.
template <int THREADS>
__device__ __forceinline__ void account_sync() { asm volatile("bar.sync 1, %0;" ::"n"(THREADS) : "memory"); }

__device__ __forceinline__ int mask_bits(const uint32_t* mask, unsigned long long b, int n) {   // set bits of [b, b + n)
  if (n <= 0) return 0;
  const unsigned long long e = b + (unsigned)n - 1;
  const long long w0 = (long long)(b >> 5), w1 = (long long)(e >> 5);
  const uint32_t first = 0xffffffffu << (b & 31), last = 0xffffffffu >> (31 - (e & 31));
  if (w0 == w1) return __popc(mask[w0] & first & last);
  int c = __popc(mask[w0] & first) + __popc(mask[w1] & last);
  for (long long w = w0 + 1; w < w1; ++w) c += __popc(mask[w]);
  return c;
}

// Pending counts, states, completion list, and the chunk's sums, which account_close folds into the layer's.  LISTED: the items are the touched vertices listed by account_edges_kernel, whose pending
// counts are already down.  Bound by the scattered words of a vertex (4 B count, 1 B state), which ascending items make
// nearly sequential; ITEMS per thread keep their reads in flight together.
enum { C_HS, C_NS, C_GS, C_MSGS, C_HUB, C_GROUPS, C_FREED, C_COUNT };
#define ITEMS 4

struct AccountShared {
  int cnt[2][8], base[2], go;
  unsigned int sum[C_COUNT];
};
// Edges and own vertices of a push that is not a grid cell: pending counts by atomics, first touches listed.
template <int THREADS>
__device__ __forceinline__ void account_edges_block(const ChunkArgs& a, AccountShared& s, int block, int blocks) {
  DevCtl* ctl = a.ctl;
  ChunkCtl* pc = a.pc;
  if (threadIdx.x == 0) s.sum[0] = s.sum[1] = 0;
  if (!block_goes_on((int)threadIdx.x, &ctl->error, &s.go, account_sync<THREADS>)) return;
  const long long e0 = a.row_ptr[a.src_begin], ne = a.row_ptr[a.src_end] - e0, total = ne + (a.src_end - a.src_begin);
  const long long stride = (long long)blocks * THREADS;
  unsigned msgs = 0, hub = 0;
  int bad = 0, par = 0;
  for (long long base = (long long)block * THREADS; base < total; base += stride, par ^= 1) {
    const long long i = base + threadIdx.x;
    int v = -1;
    if (i < ne) {
      const long long e = e0 + i;
      if (a.mask == nullptr || ((a.mask[e >> 5] >> (e & 31)) & 1u)) v = a.col[e];
      if (v >= 0) { msgs++; if (a.hub && a.hub[v]) hub++; }
    } else if (i < total) {
      v = (int)(a.src_begin + (i - ne));
    }
    bool first = false;
    if (v >= 0) {
      atomicAdd(&a.pend[v], -1);
      if (a.touch[v] != a.epoch) first = atomicMax(&a.touch[v], a.epoch) != a.epoch;
    }
    // appended per block: an address takes an atomic every 3 ns (120 k edges: 8.6 us a launch with one per warp, 6.5 now)
    const unsigned m = __ballot_sync(FULL, first);
    const int warp = threadIdx.x >> 5;
    if (rl() == 0) s.cnt[par][warp] = __popc(m);
    account_sync<THREADS>();
    if (threadIdx.x == 0) {
      int t = 0;
      for (int w = 0; w < THREADS / 32; ++w) { const int c = s.cnt[par][w]; s.cnt[par][w] = t; t += c; }
      s.base[par] = t ? atomicAdd(&pc->touched_count, t) : 0;
    }
    account_sync<THREADS>();
    if (first) {
      const int at = s.base[par] + s.cnt[par][warp] + __popc(m & ((1u << rl()) - 1));
      if (at < a.touched_capacity) a.touched_list[at] = v; else bad = 1;
    }
  }
  if (msgs) atomicAdd(&s.sum[0], msgs);
  if (hub) atomicAdd(&s.sum[1], hub);
  if (bad) atomicCAS(&ctl->error, 0, TAURUS_ERR_INTERNAL);
  account_sync<THREADS>();
  if (threadIdx.x == 0 && s.sum[0]) {
    atomicAdd((unsigned long long*)&ctl->total_messages, (unsigned long long)s.sum[0]);
    atomicAdd((unsigned long long*)&ctl->scatter_groups, (unsigned long long)s.sum[0]);   // no groups here: one per message
    if (s.sum[1]) atomicAdd((unsigned long long*)&ctl->hub_messages, (unsigned long long)s.sum[1]);
  }
}

template <bool LISTED, int THREADS>
__device__ __forceinline__ void account_block(const AccountWork& work, AccountShared& s, int block, int blocks) {
  const ChunkArgs& a = work.a;
  const Items& it = work.it;
  const uint32_t* const __restrict__ cmask = work.cmask;
  int4* const __restrict__ heavy = work.heavy;
  int32_t* const __restrict__ heavy_left = work.heavy_left;
  const long long i0 = work.i0, n_items = work.n_items;
  constexpr int WARPS = THREADS / 32;
  DevCtl* ctl = a.ctl;
  ChunkCtl* pc = a.pc;
  if (threadIdx.x < C_COUNT) s.sum[threadIdx.x] = 0;
  if (!block_goes_on((int)threadIdx.x, &ctl->error, &s.go, account_sync<THREADS>)) return;
  if (block == 0 && threadIdx.x == 0) pc->grad_base = a.dense_half >= 0 ? a.grad_off : ctl->grad_count;
  const long long n = LISTED ? (long long)pc->touched_count : n_items;
  const long long stride = (long long)blocks * THREADS * ITEMS;
  const int warp = threadIdx.x >> 5;
  const unsigned lt = (1u << rl()) - 1;
  unsigned sum[C_COUNT] = {0};
  int bad = 0, par = 0;
  for (long long base = (long long)block * THREADS * ITEMS; base < n; base += stride, par ^= 1) {
    int v[ITEMS], msgs[ITEMS], dec[ITEMS], p[ITEMS], st[ITEMS];
#pragma unroll
    for (int q = 0; q < ITEMS; ++q) {
      const long long i = base + q * THREADS + threadIdx.x;
      v[q] = -1; msgs[q] = dec[q] = 0;
      if (i < n) {
        if (LISTED) v[q] = a.touched_list[i];
        else {
          v[q] = it.v[i0 + i];
          msgs[q] = it.count[i0 + i];
          if (cmask) msgs[q] = mask_bits(cmask, it.begin[i0 + i], msgs[q]);
          dec[q] = msgs[q] + (v[q] >= a.src_begin && v[q] < a.src_end ? 1 : 0);
          if (dec[q] == 0) v[q] = -1;   // a sampled layer kept none of the group's messages
        }
      }
    }
#pragma unroll
    for (int q = 0; q < ITEMS; ++q)
      if (v[q] >= 0) { p[q] = a.pend[v[q]] - dec[q]; st[q] = a.state[v[q]]; }
    bool done[ITEMS];
    unsigned md[ITEMS];
    int wd = 0;
#pragma unroll
    for (int q = 0; q < ITEMS; ++q) {
      done[q] = false;
      if (v[q] >= 0) {
        const bool hub = a.hub && a.hub[v[q]];
        done[q] = p[q] == 0;
        if (p[q] < 0 || st[q] == TAURUS_COMPLETED) bad = 1;   // a completed vertex cannot receive a message
        if (!LISTED) a.pend[v[q]] = p[q];
        const int to = done[q] ? TAURUS_COMPLETED : hub ? TAURUS_ON_GPU : TAURUS_IN_BUFFER;
        if (to != st[q]) a.state[v[q]] = (uint8_t)to;
        if (hub) sum[C_GS]++;
        else if (st[q] == TAURUS_NOT_STARTED) sum[C_NS]++;
        else sum[C_HS]++;
        if (done[q] && !hub) sum[C_FREED]++;
        sum[C_MSGS] += (unsigned)msgs[q];
        if (msgs[q] > 0) sum[C_GROUPS]++;
        if (hub) sum[C_HUB] += (unsigned)msgs[q];
      }
      md[q] = __ballot_sync(FULL, done[q]);
      wd += __popc(md[q]);
    }
    // appended per block: single-address atomics would bound this kernel
    if (rl() == 0) s.cnt[par][warp] = wd;
    account_sync<THREADS>();
    if (threadIdx.x == 0) {
      int t = 0;
      for (int w = 0; w < WARPS; ++w) { const int c = s.cnt[par][w]; s.cnt[par][w] = t; t += c; }
      s.base[par] = t ? atomicAdd(&pc->done_count, t) : 0;
    }
    account_sync<THREADS>();
    int at = s.base[par] + s.cnt[par][warp];
#pragma unroll
    for (int q = 0; q < ITEMS; ++q) {
      if (done[q]) {
        const int i = at + __popc(md[q] & lt);
        if (i < a.grad_cap) a.done_list[i] = v[q]; else bad = 1;
        if (heavy && i < a.grad_cap) {
          const int d = a.din[v[q]];
          if (d > TAURUS_HEAVY_DEGREE) {
            const int segs = (d + TAURUS_HEAVY_SEGMENT - 1) / TAURUS_HEAVY_SEGMENT;
            const int row = atomicAdd(&ctl->heavy_rows, 1), e = atomicAdd(&pc->heavy_count, segs);
            heavy_left[row] = segs;
            for (int s = 0; s < segs; ++s) heavy[e + s] = make_int4(i, s, row, segs);
          }
        }
      }
      at += __popc(md[q]);
    }
  }
  if (bad) atomicCAS(&ctl->error, 0, TAURUS_ERR_INTERNAL);
#pragma unroll
  for (int c = 0; c < C_COUNT; ++c) {
    const unsigned x = __reduce_add_sync(FULL, sum[c]);
    if (rl() == 0 && x) atomicAdd(&s.sum[c], x);
  }
  account_sync<THREADS>();
  if (threadIdx.x < C_COUNT && s.sum[threadIdx.x]) atomicAdd(&pc->acc[threadIdx.x], (unsigned long long)s.sum[threadIdx.x]);
}

__device__ __forceinline__ void account_totals(const ChunkArgs& a, DevCtl* ctl, ChunkCtl* pc) {   // one thread
  long long c[C_COUNT];
  for (int k = 0; k < C_COUNT; ++k) c[k] = (long long)pc->acc[k];
  const long long done = pc->done_count;
  const long long F = ctl->free_top - c[C_NS], at = ctl->chunks, grad = ctl->grad_count, peak = ctl->peak_occupancy;
  if (a.pool_slots - F > peak) ctl->peak_occupancy = a.pool_slots - F;
  ctl->free_top = F + c[C_FREED];
  if (at < a.log_capacity) {
    long long* r = a.chunk_log + at * TAURUS_CK_COLUMNS;
    r[TAURUS_CK_HS] = c[C_HS]; r[TAURUS_CK_NS] = c[C_NS]; r[TAURUS_CK_EV] = 0; r[TAURUS_CK_GS] = c[C_GS];
    r[TAURUS_CK_NEED] = c[C_NS]; r[TAURUS_CK_EVICTED] = 0; r[TAURUS_CK_RELOADED] = 0;
    r[TAURUS_CK_COMPLETED] = done; r[TAURUS_CK_OCCUPANCY] = a.pool_slots - (F + c[C_FREED]);
  }
  ctl->chunks = at + 1;
  ctl->sum_hs += c[C_HS]; ctl->sum_ns += c[C_NS]; ctl->sum_gs += c[C_GS];
  ctl->completed += done;
  ctl->total_messages += c[C_MSGS]; ctl->scatter_groups += c[C_GROUPS]; ctl->hub_messages += c[C_HUB];   // (none where the edges were counted one by one)
  if (a.dense_direct) { /* rows go straight into the caller's matrix */ }
  else if (a.dense_half >= 0) ctl->out_count[a.dense_half] = done;
  else {
    if (grad + done > a.drain_rows) atomicCAS(&ctl->error, 0, TAURUS_ERR_INTERNAL);
    ctl->grad_count = grad + done;
  }
}
// After the accounting of a chunk, once, by one warp of the kernel behind it (the gather, which every push has): the chunk record, the layer's
// totals, the free-slot count and the count of waiting rows, and the counters of the next chunk (the other set; its last reader, the chunk
// before this one, is through) are cleared.  By the accounting's last block to finish it was 1.7 us on the way of every push.
__device__ __forceinline__ void account_close(const ChunkArgs& a, DevCtl* ctl, ChunkCtl* pc) {
  if (__shfl_sync(FULL, ctl->error, 0) == 0) {   // (one answer for the warp, which meets again below)
    ChunkCtl* next = pc == &ctl->pc[0] ? &ctl->pc[1] : &ctl->pc[0];
    for (int i = rl(); i < (int)(offsetof(ChunkCtl, sel_k) / 4); i += 32) reinterpret_cast<int32_t*>(next)[i] = 0;
    __syncwarp();
    if (rl() == 0) account_totals(a, ctl, pc);
  }
  if (a.report) {   // what layer_end would otherwise launch a kernel for
    __threadfence();
    __syncwarp();
    report_ctl(ctl, a.report, rl(), 32);
  }
}

// (Small pushes that are one cell of the chunk grid.)  What a kernel whose first blocks may do the accounting of the push is given; AccountArgs<false>: none.
template <bool ON> struct AccountArgs;
template <> struct AccountArgs<true> { AccountWork w; __device__ __forceinline__ int blocks() const { return w.blocks; } };
template <> struct AccountArgs<false> { __device__ __forceinline__ int blocks() const { return 0; } };
// True in the blocks that did it.  s: shared memory of the kernel to use.
template <int THREADS>
__device__ __forceinline__ bool account_here(const AccountArgs<false>&, AccountShared&) { early_start(); return false; }
template <int THREADS>
__device__ __forceinline__ bool account_here(const AccountArgs<true>& acc, AccountShared& s) {
  early_start();
  if ((int)blockIdx.x >= acc.w.blocks) return false;
  if (threadIdx.x < THREADS) account_block<false, THREADS>(acc.w, s, (int)blockIdx.x, acc.w.blocks);
  return true;
}

}  // namespace
