// Pools that hold every vertex (pool_slots >= V): the pull form of a layer.
//
// Nothing is ever evicted from such a pool, so no partial sum has to be kept between chunks: the memory of the
// accumulator rows keeps the rows that the sources send instead (projected rows, or input rows in aggregate-first layers),
// filed under their source, and a vertex's sum is formed once, when its last message has arrived, from its in-list
// (Sect. 3.1's messages, 3.4's counts and 3.6's graduation in another order of the same additions).  One message then
// costs one row read, where the push form reads the row and read-modify-writes the destination's row once per (chunk,
// destination) group.
//
// A push is
//   rows     : the chunk's rows into the store (by the projection, or a copy)
//   account  : pending counts, states, completion list and the chunk record, one item per (chunk, destination) group
//   gather   : one warp per completed vertex sums the rows of its in-list and finishes the row; long in-lists are cut
//              into segments that different warps sum
// Integer accounting (counts, states, chunk records) is that of the push form.
#include <cub/cub.cuh>

#include <algorithm>
#include <type_traits>
#include <vector>

#include "account.cuh"
#include "taurus_internal.h"

#define HEAVY_DEGREE TAURUS_HEAVY_DEGREE
#define HEAVY_SEGMENT TAURUS_HEAVY_SEGMENT

namespace {

__device__ __forceinline__ float r_lrelu(float x, float slope) { return x > 0.f ? x : slope * x; }
__device__ __forceinline__ void red_v4(float* addr, const float4& v) {
  asm volatile("red.global.add.v4.f32 [%0], {%1, %2, %3, %4};" ::"l"(addr), "f"(v.x), "f"(v.y), "f"(v.z), "f"(v.w) : "memory");
}
// Four floats as two packed pairs; each half of a packed operation is rounded like the scalar one.
struct Pairs { unsigned long long a, b; };
__device__ __forceinline__ float4 floats_of(const Pairs& p) {
  float4 v;
  asm("mov.b64 {%0, %1}, %2;" : "=f"(v.x), "=f"(v.y) : "l"(p.a));
  asm("mov.b64 {%0, %1}, %2;" : "=f"(v.z), "=f"(v.w) : "l"(p.b));
  return v;
}
__device__ __forceinline__ void add4(Pairs& s, const Pairs& r) {
  asm("add.rn.f32x2 %0, %0, %1;" : "+l"(s.a) : "l"(r.a));
  asm("add.rn.f32x2 %0, %0, %1;" : "+l"(s.b) : "l"(r.b));
}
__device__ __forceinline__ void mul4(Pairs& s, float w) {
  unsigned long long ww;
  asm("mov.b64 %0, {%1, %1};" : "=l"(ww) : "f"(w));
  asm("mul.rn.f32x2 %0, %0, %1;" : "+l"(s.a) : "l"(ww));
  asm("mul.rn.f32x2 %0, %0, %1;" : "+l"(s.b) : "l"(ww));
}
__device__ __forceinline__ void add4(float4& s, const float4& r) { s.x += r.x; s.y += r.y; s.z += r.z; s.w += r.w; }
__device__ __forceinline__ void fma4(float4& s, float w, const float4& r) {
  s.x = fmaf(w, r.x, s.x); s.y = fmaf(w, r.y, s.y); s.z = fmaf(w, r.z, s.z); s.w = fmaf(w, r.w, s.w);
}

// ------------------------------------------------------------------------------------------------ layer reset
__global__ void resident_reset_kernel(long long V, const int32_t* din, int fanout, int32_t* pend, uint8_t* state, int32_t* touch,
                                      int32_t* reload, long long pool_slots, DevCtl* ctl) {
  const long long stride = (long long)gridDim.x * blockDim.x, tid = (long long)blockIdx.x * blockDim.x + threadIdx.x;
  for (long long v = tid; v < V; v += stride) {
    const int d = din[v];
    pend[v] = ((fanout > 0 && d > fanout) ? fanout : d) + 1;
    state[v] = TAURUS_NOT_STARTED;
    touch[v] = 0;
    reload[v] = 0;
  }
  long long* words = reinterpret_cast<long long*>(ctl);
  for (long long i = tid; i < (long long)(sizeof(DevCtl) / 8); i += stride) words[i] = words + i == &ctl->free_top ? pool_slots : 0;
}

// ------------------------------------------------------------------------------------------------ account
// (account.cuh; the accounting of a small push runs in the launch that writes its rows)
static_assert(sizeof(AccountShared) <= TAURUS_ACCOUNT_SHARED, "a block fits beside a CTA of the projection,");
static_assert(4 * TAURUS_QUARTER_REGISTERS / (5 * TAURUS_ACCOUNT_THREADS) / 8 * 8 <= TAURUS_ACCOUNT_REGISTERS, "with the registers its launch bounds allow");
static_assert(TAURUS_ACCOUNT_THREADS <= 8 * 32, "eight warps (AccountShared::cnt)");

__global__ void __launch_bounds__(TAURUS_ACCOUNT_THREADS, 8) account_edges_kernel(const __grid_constant__ AccountWork w) {
  __shared__ AccountShared s;
  account_edges_block<TAURUS_ACCOUNT_THREADS>(w.a, s, (int)blockIdx.x, (int)gridDim.x);
}
template <bool LISTED>
__global__ void __launch_bounds__(TAURUS_ACCOUNT_THREADS, LISTED ? 6 : 5) account_kernel(const __grid_constant__ AccountWork w) {
  __shared__ AccountShared s;
  account_block<LISTED, TAURUS_ACCOUNT_THREADS>(w, s, (int)blockIdx.x, (int)gridDim.x);
}

// ------------------------------------------------------------------------------------------------ gather
struct GatherArgs {
  const float4* rows;        // the store: row of source u at u * pitch (float4 units)
  int pitch, vec;            // pitch and width of a gathered row in float4
  const int32_t* src;        // sources of the in-lists: entries [csc_ptr[v], csc_ptr[v + 1]), or, where a layer is
  int keep;                  //   sampled (keep > 0), the kept ones at v * keep
  const long long* csc_ptr;
  const int32_t* done_list;
  const int4* heavy;         // (index in done_list, segment, partial row, segments) of the long in-lists
  float4* heavy_rows;        // partial sums, zero between vertices
  int32_t* heavy_left;
  DevCtl* ctl;
  ChunkCtl* pc;
  const float4* bias;
  const float* att_s;
  const float2* att_tm;
  const double* att_z;
  float4* A;                 // aggregate-first: finished sums (SAGE: followed by the vertex's own row), pitch a_pitch float4; else NULL
  int a_pitch;
  float* dense;              // the caller's matrix, or NULL: graduation buffer
  long long dense_ld;
  float* grad_rows;
  long long* grad_ids;
  int d_out, act, mode, heads, head_vec;
  float gin_self, leaky;
  long long room;            // rows that the graduation buffer holds, where they go there behind others
};

#define G_WARPS 4            // warps per block
#define BATCH 8              // items a warp takes at a time
struct Item {                // fetched by one lane each: one chain of dependent reads for the whole batch
  int v, i, len, row;        // vertex, place in done_list, entries to sum (-1: nothing), partial row (-1: the whole in-list)
  uint32_t begin;            // first entry
  float scale, self, bw;     // factor of the finished row, weight of the own row, weight of the bias
};
struct HeadTerm { float t, top, scale, self, bw; };   // GAT: destination term and maximum of the scores; the same three per head

// A value that every lane of the warp holds alike, told to the compiler: the reduction's result is a uniform register, and
// branches on it need no reconvergence code (which was more than half of this kernel's instructions).
__device__ __forceinline__ int uniform(int x) { return __reduce_max_sync(FULL, x); }

__device__ __forceinline__ void copy16(void* dst, const void* src) {
  asm volatile("cp.async.cg.shared.global [%0], [%1], 16;" ::"r"((unsigned)__cvta_generic_to_shared(dst)), "l"(src) : "memory");
}
__device__ __forceinline__ void copy16_if(unsigned dst, const void* src, int yes) {   // dst: address in shared memory
  asm volatile("{\n.reg .pred p;\nsetp.ne.b32 p, %2, 0;\n@p cp.async.cg.shared.global [%0], [%1], 16;\n}" ::"r"(dst), "l"(src), "r"(yes) : "memory");
}
__device__ __forceinline__ void copy4(void* dst, const void* src) {
  asm volatile("cp.async.ca.shared.global [%0], [%1], 4;" ::"r"((unsigned)__cvta_generic_to_shared(dst)), "l"(src) : "memory");
}

// One warp per item (a completed vertex, or a segment of a long in-list), LPE lanes x VPL float4 per row and 32 / LPE rows
// side by side.  What bounds it is how many random row reads an SM has in flight, so the rows of a batch's in-lists run
// as one stream through a ring in shared memory: a step is U rows per lane group, D steps are always on their way, and
// the vertex's own row is the last step of its item.  Every lane copies and reads back its own 16 bytes: no barrier.
// With the same loads held in registers (4 rows per warp, 32 warps per SM) DRAM ran at 38 %, L2 at 27 %, the schedulers
// issued in 20 % of the cycles.  The U rows of a step are added up before they join the running sum and long in-lists
// are cut: fewer additions in sequence than the push form has.
// Issue slots are what is left beside the row reads, so control that is the same for the whole warp is told to the compiler as
// such (`uniform`), additions are packed in pairs, and lanes behind the end of a row are predicated off (copying its last 16
// bytes again instead halved the rate of 48-float rows that sit in L2).  Instructions per message of 256 / 100 floats on 800 k
// vertices, 40 M edges: 53 / 33 before, 43 / 24 now; all gathers of 2.45 M vertices, 124 M edges, three layers: 31.8 -> 27.1 ms.
// GAT: most heads the ring is sized for (0: no attention).  The scores of a block of 32 sources travel with the block's
// first step; the lanes turn them into coefficients, one source each, when the block is reached.
template <int VPL, int U, int D, int GAT>
struct Ring {
  float4 row[D + 1][U][VPL][32];
  float att[GAT ? D + 3 : 1][GAT ? 32 * GAT : 4];   // blocks between the producer and the consumer: at most one per step
  Item item[BATCH];
  HeadTerm head[GAT ? BATCH : 1][GAT ? GAT : 1];
};

template <int LPE, int VPL, int U, int D, int GAT>
__global__ void __launch_bounds__(32 * G_WARPS, VPL == 1 ? 6 : VPL == 2 ? 5 : VPL == 4 ? 4 : 2) gather_kernel(const __grid_constant__ GatherArgs g, const __grid_constant__ ChunkArgs chunk) {
  extern __shared__ __align__(16) unsigned char g_smem[];
  ChunkCtl* const pc = g.pc;
  early_start();
  if (blockIdx.x == 0) {   // a block for it: in the code of the others it would take registers
    if (threadIdx.x < 32) account_close(chunk, g.ctl, pc);
    return;
  }
  if (g.ctl->error) return;
  constexpr int EPS = 32 / LPE, STEP = U * EPS;
  static_assert(STEP <= 32 && 32 % STEP == 0, "a block of 32 sources is a whole number of steps");
  typedef Ring<VPL, U, D, GAT> R;
  const int lane = rl(), sub = lane / LPE, c4 = lane % LPE, wid = threadIdx.x >> 5;
  R& ring = reinterpret_cast<R*>(g_smem)[wid];
  const int warps = (int)(((gridDim.x - 1) * blockDim.x) >> 5), warp = (int)(((blockIdx.x - 1) * blockDim.x + threadIdx.x) >> 5);
  const int n = uniform(pc->done_count), nh = g.heavy ? uniform(pc->heavy_count) : 0;
  const int total = n + nh;
  if (g.room > 0 && uniform(pc->grad_base + n > g.room)) return;   // (the close has found the same)
  bool on[VPL];
  int hk[VPL];
#pragma unroll
  for (int k = 0; k < VPL; ++k) {
    on[k] = c4 + k * LPE < g.vec;
    hk[k] = 0;
    if (GAT && g.heads > 1) { hk[k] = (c4 + k * LPE) / g.head_vec; if (hk[k] >= g.heads) hk[k] = g.heads - 1; }
  }
  // lanes behind the end of a row copy nothing and add up what the ring happens to hold (never stored)
  const char* const rows = reinterpret_cast<const char*>(g.rows) + c4 * 16;
  constexpr unsigned SLOT = U * VPL * 512;
  const unsigned slots = (unsigned)__cvta_generic_to_shared(&ring.row[0][0][0][lane]);
  const unsigned pitch = (unsigned)g.pitch * 16u;
  const bool sage = g.mode == TAURUS_SAGE_MEAN;
  const int own_off = sage && !g.A ? g.vec * 16 : 0;   // SAGE, projected rows: the self message T_v sits behind P_v

  // Batches: the first of a warp is its own number, the others come from a counter, asked for while the batch before is summed
  // (dealt out in turn, the slowest warp of a launch of 10 ms finished 13 % after the average one).  Few items: up to four at
  // once, since a batch pays one chain of dependent reads whatever its size (12 548 items of 32 floats, 3 552 warps: one at
  // a time 18.9 us, four 13.8); more: two batches a warp or more, for the balance (338 884: eight at most 247 us, dealt out 277).
  const int once = (total + warps - 1) / warps < 4 ? (total + warps - 1) / warps : 4;
  int per = total / (warps * 2) < BATCH ? total / (warps * 2) : BATCH;
  per = per < once ? once : per;
  per = per < 1 ? 1 : per;
  const int n_batches = (total + per - 1) / per;
  int ticket = 0;
  for (int batch = uniform(warp); batch < n_batches; batch = uniform(lane == 0 ? ticket : 0)) {
    if (lane == 0) ticket = (int)atomicAdd(&pc->span_next, 1u) + warps;
    const int i0 = batch * per, cnt = total - i0 < per ? total - i0 : per;
    __syncwarp();
    if (lane < cnt) {
      Item x;
      int i = i0 + lane - nh, seg = 0;   // segments first
      x.row = -1;
      if (i < 0) { const int4 h = g.heavy[i0 + lane]; i = h.x; seg = h.y; x.row = h.z; }
      x.i = i;
      x.v = g.done_list[i];
      const long long b = g.csc_ptr[x.v];
      int d = (int)(g.csc_ptr[x.v + 1] - b);
      x.scale = x.self = x.bw = 1.f;
      if (g.mode == TAURUS_GCN_SYM) {
        x.bw = (float)sqrt((double)d + 1.0);
        x.scale = (float)(1.0 / sqrt((double)d + 1.0));
      } else if (g.mode == TAURUS_GIN_SUM) {
        x.self = g.gin_self;
      }
      x.begin = (uint32_t)b;
      if (g.keep) { x.begin = (uint32_t)x.v * (unsigned)g.keep; if (d > g.keep) d = g.keep; }
      if (sage) x.scale = 1.0f / (float)(d > 1 ? d : 1);
      x.len = d;
      if (x.row >= 0) { x.begin += (unsigned)(seg * HEAVY_SEGMENT); x.len = d - seg * HEAVY_SEGMENT < HEAVY_SEGMENT ? d - seg * HEAVY_SEGMENT : HEAVY_SEGMENT; }
      else if (g.heavy && d > HEAVY_DEGREE) x.len = -1;
      ring.item[lane] = x;
    }
    __syncwarp();
    if (GAT) {
      for (int x = lane; x < cnt * g.heads; x += 32) {
        const int j = x / g.heads, h = x - j * g.heads;
        const size_t at = (size_t)ring.item[j].v * g.heads + h;
        const float2 tm = g.att_tm[at];
        const double z = g.att_z[at];
        HeadTerm e;
        e.t = tm.x; e.top = tm.y;
        e.self = __expf(r_lrelu(g.att_s[at] + tm.x, g.leaky) - tm.y);
        e.bw = (float)z;
        e.scale = (float)(1.0 / z);
        ring.head[j][h] = e;
      }
      __syncwarp();
    }

    // sources, 32 at a time: `u` the block the producer is in, `un` the one after it (item fj, entries from fb on)
    int u = 0, un = 0, fj = 0, fb = -32, flen = uniform(ring.item[0].len);
    auto fetch = [&]() {
      fb += 32;
      while (fj < cnt && fb >= flen) {
        if (++fj < cnt) flen = uniform(ring.item[fj].len);
        fb = 0;
      }
      if (fj < cnt) un = fb + lane < flen ? g.src[ring.item[fj].begin + fb + lane] : 0;
    };
    // producer: next step to request (item pj, entries from pp on; pp at the end: the own row)
    int pj = -1, pp = 0, plen = 0;
    int pblk = 0, cblk = 0;     // GAT: block slots of the producer and the consumer
    auto next_block = [&]() {
      u = un;
      if (GAT) {
        pblk = pblk == D + 2 ? 0 : pblk + 1;
        if (pp + lane < plen) {
          const float* s = g.att_s + (size_t)(unsigned)u * g.heads;
          float* to = &ring.att[GAT ? pblk : 0][lane * g.heads];
          if ((g.heads & 3) == 0) for (int h = 0; h < g.heads; h += 4) copy16(to + h, s + h);
          else for (int h = 0; h < g.heads; ++h) copy4(to + h, s + h);
        }
      }
      fetch();
    };
    auto enter = [&]() {
      do {
        ++pj;
        if (pj < cnt) plen = uniform(ring.item[pj].len);
      } while (pj < cnt && plen < 0);
      if (pj < cnt) {
        pp = 0;
        if (plen > 0) next_block();
      }
    };
    auto produce = [&](unsigned to) {
      if (pj < cnt) {
        if (pp < plen) {
          const int at = (pp & 31) + sub, left = plen - pp;
          if (left >= STEP) {
#pragma unroll
            for (int q = 0; q < U; ++q) {
              const char* src = rows + (unsigned long long)(unsigned)__shfl_sync(FULL, u, at + q * EPS) * pitch;
#pragma unroll
              for (int k = 0; k < VPL; ++k) copy16_if(to + (q * VPL + k) * 512, src + k * LPE * 16, on[k]);
            }
          } else {
#pragma unroll
            for (int q = 0; q < U; ++q) {
              const char* src = rows + (unsigned long long)(unsigned)__shfl_sync(FULL, u, at + q * EPS) * pitch;
#pragma unroll
              for (int k = 0; k < VPL; ++k) copy16_if(to + (q * VPL + k) * 512, src + k * LPE * 16, on[k] && q * EPS + sub < left);
            }
          }
          pp += STEP;
          if (pp < plen && (pp & 31) == 0) next_block();
        } else {
          const bool whole = sub == 0 && ring.item[pj].row < 0;
          const char* src = rows + (size_t)ring.item[pj].v * pitch + own_off;
#pragma unroll
          for (int k = 0; k < VPL; ++k) copy16_if(to + k * 512, src + k * LPE * 16, on[k] && whole);
          enter();
        }
      }
      asm volatile("cp.async.commit_group;" ::: "memory");
    };
    fetch();
    enter();
#pragma unroll 1
    for (int d = 0; d < D; ++d) produce(slots + d * SLOT);
    unsigned now = slots, before = slots + D * SLOT;   // slots of this step and of the one before it
    auto advance = [&]() {
      produce(before);   // the step before this one: its rows have been added
      before = now;
      now = now == slots + D * SLOT ? slots : now + SLOT;
    };

#pragma unroll 1
    for (int j = 0; j < cnt; ++j) {
      const int len = uniform(ring.item[j].len);
      if (len < 0) continue;
      Pairs acc[VPL];
#pragma unroll
      for (int k = 0; k < VPL; ++k) acc[k].a = acc[k].b = 0ull;
#pragma unroll 1
      for (int p = 0; p < len; p += STEP) {
        asm volatile("cp.async.wait_group %0;" ::"n"(D - 1) : "memory");
        if (GAT && (p & 31) == 0) {   // scores of the block -> coefficients
          cblk = cblk == D + 2 ? 0 : cblk + 1;
          if (p + lane < len) {
            float* const w = &ring.att[GAT ? cblk : 0][lane * g.heads];
            for (int h = 0; h < g.heads; ++h) w[h] = __expf(r_lrelu(w[h] + ring.head[j][GAT ? h : 0].t, g.leaky) - ring.head[j][GAT ? h : 0].top);
          }
          __syncwarp();
        }
        auto add_step = [&](auto full) {
#pragma unroll
          for (int k = 0; k < VPL; ++k) {
            Pairs r[U];
#pragma unroll
            for (int q = 0; q < U; ++q) {
              r[q].a = r[q].b = 0ull;
              if (full || p + q * EPS + sub < len) {
                asm volatile("ld.shared.v2.b64 {%0, %1}, [%2];" : "=l"(r[q].a), "=l"(r[q].b) : "r"(now + (unsigned)((q * VPL + k) * 512)) : "memory");
                if (GAT) mul4(r[q], ring.att[GAT ? cblk : 0][((p & 31) + q * EPS + sub) * g.heads + hk[k]]);
              }
            }
#pragma unroll
            for (int o = 1; o < U; o <<= 1)
#pragma unroll
              for (int q = 0; q + o < U; q += 2 * o) add4(r[q], r[q + o]);
            add4(acc[k], r[0]);
          }
        };
        if (p + STEP <= len) add_step(std::true_type()); else add_step(std::false_type());
        advance();
      }
      // the sub-groups' sums
      float4 sum[VPL];
#pragma unroll
      for (int k = 0; k < VPL; ++k) {
#pragma unroll
        for (int o = LPE; o < 32; o <<= 1) {
          Pairs y;
          y.a = __shfl_xor_sync(FULL, acc[k].a, o); y.b = __shfl_xor_sync(FULL, acc[k].b, o);
          add4(acc[k], y);
        }
        sum[k] = floats_of(acc[k]);
      }
      // the own row
      asm volatile("cp.async.wait_group %0;" ::"n"(D - 1) : "memory");
      float4 x[VPL];
#pragma unroll
      for (int k = 0; k < VPL; ++k) {
        x[k] = make_float4(0.f, 0.f, 0.f, 0.f);
        if (sub == 0 && on[k]) asm volatile("ld.shared.v4.f32 {%0, %1, %2, %3}, [%4];" : "=f"(x[k].x), "=f"(x[k].y), "=f"(x[k].z), "=f"(x[k].w) : "r"(now + k * 512u) : "memory");
      }
      advance();

      const int v = ring.item[j].v, i = ring.item[j].i, row = uniform(ring.item[j].row);
      if (row >= 0) {
        // partial sums meet in a row of their own; the segment that arrives last finishes the vertex
        float4* const part = g.heavy_rows + (size_t)row * g.vec;
        if (sub == 0)
#pragma unroll
          for (int k = 0; k < VPL; ++k)
            if (on[k]) red_v4(reinterpret_cast<float*>(part + c4 + k * LPE), sum[k]);
        __threadfence();
        __syncwarp();
        int left = 0;
        if (lane == 0) left = atomicSub(&g.heavy_left[row], 1);
        left = __shfl_sync(FULL, left, 0);
        if (left != 1) continue;
        __threadfence();
        if (sub == 0)
#pragma unroll
          for (int k = 0; k < VPL; ++k)
            if (on[k]) {
              sum[k] = __ldcg(part + c4 + k * LPE);
              part[c4 + k * LPE] = make_float4(0.f, 0.f, 0.f, 0.f);
              x[k] = *reinterpret_cast<const float4*>(rows + (size_t)v * pitch + own_off + k * LPE * 16);
            }
      }
      // finished row
      if (sub == 0) {
        float scale = ring.item[j].scale, self = ring.item[j].self, bw = ring.item[j].bw;
        const long long base = g.A || g.dense ? 0 : pc->grad_base;
        const bool vec_ok = g.A || !g.dense || ((g.dense_ld & 3) == 0 && (reinterpret_cast<uintptr_t>(g.dense) & 15) == 0);
        float* const out = g.A ? reinterpret_cast<float*>(g.A + (size_t)i * g.a_pitch)
                               : g.dense ? g.dense + (size_t)v * g.dense_ld : g.grad_rows + (size_t)(base + i) * g.vec * 4;
        const int width = g.dense && !g.A ? g.d_out : g.vec * 4;
#pragma unroll
        for (int k = 0; k < VPL; ++k) {
          const int c = c4 + k * LPE;
          if (!on[k]) continue;
          if (GAT) { const HeadTerm& h = ring.head[j][hk[k]]; scale = h.scale; self = h.self; bw = h.bw; }
          float4 y = sum[k];
          if (g.A) {   // the weights, the bias and the activation are applied by the transform
            if (sage) reinterpret_cast<float4*>(out)[g.vec + c] = x[k];
            else fma4(y, self, x[k]);
            y.x *= scale; y.y *= scale; y.z *= scale; y.w *= scale;
          } else {
            if (sage) add4(y, x[k]);   // T_v: own row times W_self, plus bias, times the message count
            else {
              const float4 b = g.bias[c];
              add4(y, make_float4(x[k].x * self + b.x * bw, x[k].y * self + b.y * bw, x[k].z * self + b.z * bw, x[k].w * self + b.w * bw));
            }
            y.x *= scale; y.y *= scale; y.z *= scale; y.w *= scale;
            if (g.act) { y.x = fmaxf(y.x, 0.f); y.y = fmaxf(y.y, 0.f); y.z = fmaxf(y.z, 0.f); y.w = fmaxf(y.w, 0.f); }
          }
          const int c0 = c << 2;
          if (vec_ok && c0 + 3 < width) {
            reinterpret_cast<float4*>(out)[c] = y;
          } else {   // ragged last columns, or a matrix whose rows are not 16-byte aligned
            if (c0 < width) out[c0] = y.x;
            if (c0 + 1 < width) out[c0 + 1] = y.y;
            if (c0 + 2 < width) out[c0 + 2] = y.z;
            if (c0 + 3 < width) out[c0 + 3] = y.w;
          }
        }
        if (c4 == 0 && !g.dense && !g.A) g.grad_ids[base + i] = v;
      }
    }
  }
}

// per_sm: the context's record of the instantiation (blocks per SM, 0 = not launched yet).  The shared-memory limit belongs to
// the context's device, so nothing is kept process-wide.
template <int LPE, int VPL, int U, int D, int GAT>
int launch_g(taurus_ctx* c, const GatherArgs& g, const ChunkArgs& a, long long bound, int* per_sm, cudaStream_t st) {
  const size_t smem = sizeof(Ring<VPL, U, D, GAT>) * G_WARPS;
  if (*per_sm == 0) {
    int b = 0;
    cudaError_t e = cudaSuccess;
    if (smem > 48 * 1024) e = cudaFuncSetAttribute(gather_kernel<LPE, VPL, U, D, GAT>, cudaFuncAttributeMaxDynamicSharedMemorySize, (int)smem);
    if (e == cudaSuccess) e = cudaOccupancyMaxActiveBlocksPerMultiprocessor(&b, gather_kernel<LPE, VPL, U, D, GAT>, 32 * G_WARPS, smem);
    if (e != cudaSuccess) { taurus_note_cuda_error(e, "gather_kernel"); return TAURUS_ERR_CUDA; }
    *per_sm = b < 1 ? 1 : b;
  }
  // no more warps than items: a completed vertex each, and the segments of long in-lists
  const long long items = bound + c->n_heavy_segments;
  const int grid = (int)std::max<long long>(1, std::min<long long>((items + G_WARPS - 1) / G_WARPS, (long long)c->sm_count * *per_sm));
  const cudaError_t e = launch_early(c->early, gather_kernel<LPE, VPL, U, D, GAT>, grid + 1, 32 * G_WARPS, smem, st, g, a);   // the accounting has been enqueued: the push must not look as if nothing had happened
  if (e != cudaSuccess) { taurus_note_cuda_error(e, "gather_kernel"); return TAURUS_ERR_CUDA; }
  return TAURUS_OK;
}
template <int LPE, int VPL, int U, int D>
int launch_g2(taurus_ctx* c, const GatherArgs& g, const ChunkArgs& a, long long bound, int width_class, cudaStream_t st) {
  int* const per_sm = c->gather_per_sm[width_class];
  if (g.mode != TAURUS_GAT) return launch_g<LPE, VPL, U, D, 0>(c, g, a, bound, per_sm, st);
  constexpr int DG = D > 3 ? 3 : 2;   // the scores take room in the ring
  return g.heads <= 4 ? launch_g<LPE, VPL, U, DG, 4>(c, g, a, bound, per_sm + 1, st) : launch_g<LPE, VPL, U, DG, 16>(c, g, a, bound, per_sm + 2, st);
}

// ------------------------------------------------------------------------------------------------ rows into the store
// out[r] = scale * X[r], zero-padded from K columns to the pitch ldo, so that every sector of a row is written whole; scale = 1, or
// 1 / sqrt(out-degree + 1) with GCN.  A copy, bound by memory: 8 blocks per SM, all of the launch's grid at once (36 registers
// let only 6 of them in, and the last quarter of the grid ran by itself: 524 288 rows of 256 floats 222 us, now 178 = 6.0 TB/s; of 100
// floats 114 and 93).
__device__ __forceinline__ void store_rows(const float* __restrict__ X, long long ldx, int n, int K, long long src_begin, int gcn,
                                           const long long* __restrict__ row_ptr, float* __restrict__ out, int ldo, int block, int blocks) {
  const long long stride = (long long)blocks * blockDim.x;
  const int vec = ldo >> 2;
  const bool wide = (ldx & 3) == 0 && (reinterpret_cast<uintptr_t>(X) & 15) == 0;
  for (long long i = (long long)block * blockDim.x + threadIdx.x; i < (long long)n * vec; i += stride) {
    const long long r = i / vec;
    const int c = (int)(i - r * vec) * 4;
    const float* src = X + r * ldx + c;
    float4 x;
    if (wide && c + 3 < K) x = *reinterpret_cast<const float4*>(src);
    else x = make_float4(c < K ? src[0] : 0.f, c + 1 < K ? src[1] : 0.f, c + 2 < K ? src[2] : 0.f, c + 3 < K ? src[3] : 0.f);
    if (gcn) {
      const long long u = src_begin + r;
      const float s = (float)(1.0 / sqrt((double)(row_ptr[u + 1] - row_ptr[u]) + 1.0));
      x.x *= s; x.y *= s; x.z *= s; x.w *= s;
    }
    reinterpret_cast<float4*>(out)[i] = x;
  }
}

__global__ void __launch_bounds__(256, 8) store_rows_kernel(const float* X, long long ldx, int n, int K, long long src_begin, int gcn, const long long* row_ptr,
                                                            float* out, int ldo) {
  store_rows(X, ldx, n, K, src_begin, gcn, row_ptr, out, ldo, (int)blockIdx.x, (int)gridDim.x);
}
// The first blocks do the accounting of the push.
__global__ void __launch_bounds__(256, 4) store_and_account_kernel(const float* X, long long ldx, int n, int K, long long src_begin, int gcn, const long long* row_ptr,
                                                                   float* out, int ldo, const __grid_constant__ AccountArgs<true> acc) {
  __shared__ AccountShared s;
  if (account_here<256>(acc, s)) return;
  store_rows(X, ldx, n, K, src_begin, gcn, row_ptr, out, ldo, (int)blockIdx.x - acc.blocks(), (int)gridDim.x - acc.blocks());
}

// ------------------------------------------------------------------------------------------------ attention
// tm[v] = (t_v, LeakyReLU(max_u s_u + t_v)) and z[v] = sum over v itself and its in-list of exp(e_uv - max): two sweeps
// over the in-list, (entry, head) pairs across the lanes, the second one in double.  Bound by the latency of the scalars'
// reads (heads x 4 B per entry, from L2), so a lane holds the first HELD of its scores for the second sweep.  The push form
// of the same sweeps pays one atomic per edge, head and sweep: 4.7 ms for two layers of 400 k vertices, 20 M edges, four
// heads.  WARPS = 1: a warp per vertex, long in-lists left out; else a block of so many warps per listed vertex with an
// in-list of more than `above` and at most `upto` entries.
#define HELD 8
template <int WARPS>
__global__ void __launch_bounds__(WARPS == 1 ? 256 : 32 * WARPS)
attention_kernel(long long V, int heads, const long long* __restrict__ csc_ptr, const int32_t* __restrict__ csc_src, const uint32_t* __restrict__ cmask,
                 const float* __restrict__ att_s, const float* __restrict__ att_t, float slope, float2* __restrict__ tm, double* __restrict__ z,
                 const int32_t* __restrict__ list, int above, int upto) {
  constexpr bool LONG = WARPS > 1;
  __shared__ float s_max[LONG ? WARPS * 16 : 1];
  __shared__ double s_sum[LONG ? WARPS * 16 : 1];
  const int lane = rl(), wid = threadIdx.x >> 5;
  const int eps = 32 / heads, sub = lane / heads, h = lane - sub * heads;   // eps entries side by side; lanes behind them idle
  const bool live = sub < eps;
  int top = 1;                       // power of two >= eps
  while (top < eps) top <<= 1;
  const long long stride = LONG ? gridDim.x : ((long long)gridDim.x * blockDim.x) >> 5;
  const int step = WARPS * eps, first = LONG ? wid * eps + sub : sub;
  for (long long i = LONG ? blockIdx.x : ((long long)blockIdx.x * blockDim.x + threadIdx.x) >> 5; i < V; i += stride) {
    const long long v = LONG ? list[i] : i;
    const long long b = csc_ptr[v];
    const int d = (int)(csc_ptr[v + 1] - b);
    if (d <= above || d > upto) continue;
    const float own = live ? att_s[v * heads + h] : 0.f, t = live ? att_t[v * heads + h] : 0.f;
    float x[HELD];
    unsigned has = 0;                // which of the held scores are kept entries
    auto load = [&](int p0) {
      has = 0;
#pragma unroll
      for (int q = 0; q < HELD; ++q) {
        const int p = p0 + q * step + first;
        x[q] = own;
        if (live && p < d && (!cmask || ((cmask[(b + p) >> 5] >> ((b + p) & 31)) & 1u))) {
          x[q] = att_s[(long long)csc_src[b + p] * heads + h];
          has |= 1u << q;
        }
      }
    };
    float mx = own;   // the self message takes part in the maximum
    for (int p0 = 0; p0 < d; p0 += HELD * step) {
      load(p0);
#pragma unroll
      for (int q = 0; q < HELD; ++q) mx = fmaxf(mx, x[q]);
    }
    for (int o = top >> 1; o; o >>= 1) {
      const float y = __shfl_down_sync(FULL, mx, o * heads);
      if (sub + o < eps) mx = fmaxf(mx, y);
    }
    if (LONG) {
      if (lane < heads) s_max[wid * 16 + lane] = mx;
      __syncthreads();
      if (lane < heads) for (int w = 0; w < WARPS; ++w) mx = fmaxf(mx, s_max[w * 16 + lane]);
    }
    mx = __shfl_sync(FULL, mx, h);
    const float m = r_lrelu(mx + t, slope);
    double sum = 0.0;
    for (int p0 = 0; p0 < d; p0 += HELD * step) {
      if (d > HELD * step) load(p0);   // else the scores are still held
#pragma unroll
      for (int q = 0; q < HELD; ++q)
        if ((has >> q) & 1u) sum += (double)__expf(r_lrelu(x[q] + t, slope) - m);
    }
    for (int o = top >> 1; o; o >>= 1) {
      const double y = __shfl_down_sync(FULL, sum, o * heads);
      if (sub + o < eps) sum += y;
    }
    if (LONG) {
      if (lane < heads) s_sum[wid * 16 + lane] = sum;
      __syncthreads();
      if (wid == 0 && lane < heads) { sum = 0.0; for (int w = 0; w < WARPS; ++w) sum += s_sum[w * 16 + lane]; }
    }
    if (lane < heads && (!LONG || wid == 0)) {
      tm[v * heads + lane] = make_float2(t, m);
      z[v * heads + lane] = sum + (double)__expf(r_lrelu(own + t, slope) - m);
    }
    if (LONG) __syncthreads();   // the partial results are rewritten for the block's next vertex
  }
}

// The same for 1, 2, 4 or 8 heads, whose scores of an entry are one vector: a lane per entry, eight lanes per vertex, so four vertices' chains of
// dependent reads (offsets, sources, scores) run side by side in a warp, and a read brings in H times as many scores.  The vertices with
// long in-lists in the same launch, by the first blocks: a block each, then a warp each.  Two layers of 400 k vertices, 20 M edges, four
// heads: three launches of the kernel above 1.15 ms, this one 0.44 (a block for every vertex of the list 0.51; 4 or 16 lanes 0.59).
template <int H> struct Scores { float x[H]; };
template <int H>
__device__ __forceinline__ Scores<H> scores_of(const float* __restrict__ att, long long v) {
  Scores<H> s;
  const float* p = att + v * H;
  if constexpr (H == 1) s.x[0] = *p;
  else if constexpr (H == 2) { const float2 a = *reinterpret_cast<const float2*>(p); s.x[0] = a.x; s.x[1] = a.y; }
  else
#pragma unroll
    for (int h = 0; h < H; h += 4) {
      const float4 a = *reinterpret_cast<const float4*>(p + h);
      s.x[h] = a.x; s.x[h + 1] = a.y; s.x[h + 2] = a.z; s.x[h + 3] = a.w;
    }
  return s;
}
#define ATT_LANES 8          // lanes per vertex
#define ATT_BLOCK 4096       // in-lists of the list that are a whole block's
template <int H>
__global__ void __launch_bounds__(256) attention_vec_kernel(long long V, const long long* __restrict__ csc_ptr, const int32_t* __restrict__ csc_src,
                                                            const uint32_t* __restrict__ cmask, const float* __restrict__ att_s, const float* __restrict__ att_t,
                                                            float slope, float2* __restrict__ tm, double* __restrict__ z, const int32_t* __restrict__ list, long long n_list,
                                                            int list_blocks) {
  constexpr int KEEP = H == 8 ? 4 : 8;   // entries of a lane whose scores are held for the second sweep
  __shared__ float s_max[8][H];
  __shared__ double s_sum[8][H];
  // One vertex by G threads, of which this is number g.  All of them / the groups of a warp take the same path.
  auto vertex = [&](auto threads, long long v, bool live) {
    constexpr int G = decltype(threads)::value;
    constexpr bool BLOCK = G > 32;
    const int g = (int)threadIdx.x % G;
    const long long b = live ? csc_ptr[v] : 0;
    int d = live ? (int)(csc_ptr[v + 1] - b) : 0;
    if (G < 32 && d > HEAVY_DEGREE) { d = 0; live = false; }   // (on the list)
    const int most = G < 32 ? __reduce_max_sync(FULL, d) : d;
    Scores<H> own, t, x[KEEP];
#pragma unroll
    for (int h = 0; h < H; ++h) own.x[h] = t.x[h] = 0.f;
    if (live) { own = scores_of<H>(att_s, v); t = scores_of<H>(att_t, v); }
    unsigned has = 0;
    auto load = [&](int p0) {
      has = 0;
      int src[KEEP];
#pragma unroll
      for (int q = 0; q < KEEP; ++q) {
        const int p = p0 + q * G + g;
        src[q] = -1;
        if (p < d && (!cmask || ((cmask[(b + p) >> 5] >> ((b + p) & 31)) & 1u))) { src[q] = csc_src[b + p]; has |= 1u << q; }
      }
#pragma unroll
      for (int q = 0; q < KEEP; ++q) { if (src[q] >= 0) x[q] = scores_of<H>(att_s, src[q]); else x[q] = own; }
    };
    float mx[H];
#pragma unroll
    for (int h = 0; h < H; ++h) mx[h] = own.x[h];   // the self message takes part in the maximum
    for (int p0 = 0; p0 < most; p0 += KEEP * G) {
      load(p0);
#pragma unroll
      for (int q = 0; q < KEEP; ++q)
#pragma unroll
        for (int h = 0; h < H; ++h) mx[h] = fmaxf(mx[h], x[q].x[h]);
    }
#pragma unroll
    for (int o = (BLOCK ? 32 : G) / 2; o; o >>= 1)
#pragma unroll
      for (int h = 0; h < H; ++h) mx[h] = fmaxf(mx[h], __shfl_xor_sync(FULL, mx[h], o));
    if (BLOCK) {
      if (rl() == 0)
#pragma unroll
        for (int h = 0; h < H; ++h) s_max[threadIdx.x >> 5][h] = mx[h];
      __syncthreads();
#pragma unroll
      for (int h = 0; h < H; ++h)
#pragma unroll
        for (int w = 0; w < 8; ++w) mx[h] = fmaxf(mx[h], s_max[w][h]);
    }
    double sum[H];
#pragma unroll
    for (int h = 0; h < H; ++h) { mx[h] = r_lrelu(mx[h] + t.x[h], slope); sum[h] = 0.0; }
    for (int p0 = 0; p0 < most; p0 += KEEP * G) {
      if (most > KEEP * G) load(p0);   // else the scores are still held
#pragma unroll
      for (int q = 0; q < KEEP; ++q)
        if ((has >> q) & 1u)
#pragma unroll
          for (int h = 0; h < H; ++h) sum[h] += (double)__expf(r_lrelu(x[q].x[h] + t.x[h], slope) - mx[h]);
    }
#pragma unroll
    for (int o = (BLOCK ? 32 : G) / 2; o; o >>= 1)
#pragma unroll
      for (int h = 0; h < H; ++h) sum[h] += __shfl_xor_sync(FULL, sum[h], o);
    if (BLOCK) {
      if (rl() == 0)
#pragma unroll
        for (int h = 0; h < H; ++h) s_sum[threadIdx.x >> 5][h] = sum[h];
      __syncthreads();
      if (g < H) {
#pragma unroll
        for (int h = 0; h < H; ++h) { sum[h] = 0.0; for (int w = 0; w < 8; ++w) sum[h] += s_sum[w][h]; }
      }
    }
#pragma unroll
    for (int h = 0; h < H; ++h)
      if (live && g == h) {
        tm[v * H + h] = make_float2(t.x[h], mx[h]);
        z[v * H + h] = sum[h] + (double)__expf(r_lrelu(own.x[h] + t.x[h], slope) - mx[h]);
      }
    if (BLOCK) __syncthreads();   // the partial results are rewritten for the block's next vertex
  };
  if ((int)blockIdx.x < list_blocks) {
    for (long long i = blockIdx.x; i < n_list; i += list_blocks) {
      const long long v = list[i];
      if (csc_ptr[v + 1] - csc_ptr[v] > ATT_BLOCK) vertex(std::integral_constant<int, 256>(), v, true);
    }
    for (long long i = (long long)blockIdx.x * 8 + (threadIdx.x >> 5); i < n_list; i += (long long)list_blocks * 8) {
      const long long v = list[i];
      if (csc_ptr[v + 1] - csc_ptr[v] <= ATT_BLOCK) vertex(std::integral_constant<int, 32>(), v, true);
    }
    return;
  }
  const long long warps = (long long)(gridDim.x - list_blocks) * 8, per = 32 / ATT_LANES;
  for (long long v0 = ((long long)(blockIdx.x - list_blocks) * 8 + (threadIdx.x >> 5)) * per; v0 < V; v0 += warps * per) {
    const long long v = v0 + rl() / ATT_LANES;
    vertex(std::integral_constant<int, ATT_LANES>(), v, v < V);
  }
}

// ------------------------------------------------------------------------------------------------ build (init)
__global__ void edge_sources_kernel(long long V, const long long* __restrict__ row_ptr, int32_t* __restrict__ src) {
  const long long warps = ((long long)gridDim.x * blockDim.x) >> 5;
  for (long long u = ((long long)blockIdx.x * blockDim.x + threadIdx.x) >> 5; u < V; u += warps)
    for (long long k = row_ptr[u] + rl(); k < row_ptr[u + 1]; k += 32) src[k] = (int32_t)u;
}
__global__ void degrees_kernel(long long V, const int32_t* __restrict__ din, long long* __restrict__ out) {   // out[V] = 0: room for the total
  const long long stride = (long long)gridDim.x * blockDim.x;
  for (long long v = (long long)blockIdx.x * blockDim.x + threadIdx.x; v <= V; v += stride) out[v] = v < V ? din[v] : 0;
}

// Items of vertex v, ascending by chunk: one per chunk that holds a source of its in-list, and one for v's own chunk.
// Pass 0 counts them, pass 1 writes (chunk, vertex, first entry) from the vertex's offset on.
template <int PASS>
__global__ void items_kernel(long long V, unsigned cs, const long long* __restrict__ csc_ptr, const int32_t* __restrict__ csc_src,
                             long long* __restrict__ at, int32_t* __restrict__ chunk, int32_t* __restrict__ item_v, uint32_t* __restrict__ item_b,
                             unsigned long long* __restrict__ heavy) {   // heavy[0..1]: vertices with long in-lists, their segments
  const long long warps = ((long long)gridDim.x * blockDim.x) >> 5;
  const int lane = rl();
  for (long long v = ((long long)blockIdx.x * blockDim.x + threadIdx.x) >> 5; v < V; v += warps) {
    const long long b = csc_ptr[v], e = csc_ptr[v + 1];
    const unsigned own = (unsigned)v / cs;
    uint32_t put = PASS ? (uint32_t)at[v] : 0u, n = 0;
    unsigned prev = 0xffffffffu;    // chunk of the entry before the batch
    bool own_done = false;
    for (long long p0 = b; p0 < e; p0 += 32) {
      const long long p = p0 + lane;
      const unsigned k = p < e ? (unsigned)csc_src[p] / cs : 0xffffffffu;
      unsigned before = __shfl_up_sync(FULL, k, 1);
      if (lane == 0) before = prev;
      const bool head = p < e && k != before;
      const unsigned heads = __ballot_sync(FULL, head);
      const unsigned past = __ballot_sync(FULL, p < e && k >= own);   // the first such entry is where the own chunk's item starts
      int extra_lane = 32;
      if (!own_done && past) {
        own_done = true;
        const int f = __ffs(past) - 1;
        const unsigned kf = __shfl_sync(FULL, k, f);
        if (kf != own) {   // no source of the own chunk: an item without messages in front of this entry (a head, as its chunk is a later one)
          extra_lane = f;
          if (PASS && lane == f) {
            const uint32_t i = put + __popc(heads & ((1u << f) - 1));
            chunk[i] = (int32_t)own; item_v[i] = (int32_t)v; item_b[i] = (uint32_t)p;
          }
        }
      }
      if (PASS && head) {
        const uint32_t i = put + __popc(heads & ((1u << lane) - 1)) + (lane >= extra_lane ? 1u : 0u);
        chunk[i] = (int32_t)k; item_v[i] = (int32_t)v; item_b[i] = (uint32_t)p;
      }
      const uint32_t got = (uint32_t)__popc(heads) + (extra_lane < 32 ? 1u : 0u);
      put += got; n += got;
      prev = __shfl_sync(FULL, k, 31);
    }
    if (!own_done) {   // every source lies in an earlier chunk
      if (PASS && lane == 0) { chunk[put] = (int32_t)own; item_v[put] = (int32_t)v; item_b[put] = (uint32_t)e; }
      n += 1;
    }
    if (!PASS && lane == 0) {
      at[v] = n;
      if (e - b > HEAVY_DEGREE) {
        atomicAdd(&heavy[0], 1ull);
        atomicAdd(&heavy[1], (unsigned long long)((e - b + HEAVY_SEGMENT - 1) / HEAVY_SEGMENT));
      }
    }
  }
}
__global__ void items_order_kernel(long long M, const int32_t* __restrict__ order, const int32_t* __restrict__ v_in, const uint32_t* __restrict__ b_in,
                                   const long long* __restrict__ csc_ptr, int32_t* __restrict__ v_out, uint32_t* __restrict__ b_out,
                                   int32_t* __restrict__ n_out) {
  const long long stride = (long long)gridDim.x * blockDim.x;
  for (long long i = (long long)blockIdx.x * blockDim.x + threadIdx.x; i < M; i += stride) {
    const int32_t j = order[i];
    const int32_t v = v_in[j];
    const uint32_t b = b_in[j];
    const uint32_t e = (long long)j + 1 < M && v_in[(long long)j + 1] == v ? b_in[j + 1] : (uint32_t)csc_ptr[v + 1];
    v_out[i] = v; b_out[i] = b; n_out[i] = (int32_t)(e - b);
  }
}
__global__ void items_bounds_kernel(long long M, long long n_chunks, const int32_t* __restrict__ key, long long* __restrict__ ptr) {
  const long long k = (long long)blockIdx.x * blockDim.x + threadIdx.x;
  if (k > n_chunks) return;
  long long lo = 0, hi = M;   // first item of a chunk >= k
  while (lo < hi) { const long long mid = (lo + hi) >> 1; if ((long long)key[mid] < k) lo = mid + 1; else hi = mid; }
  ptr[k] = lo;
}
__global__ void iota32_kernel(long long n, int32_t* out) {
  const long long stride = (long long)gridDim.x * blockDim.x;
  for (long long i = (long long)blockIdx.x * blockDim.x + threadIdx.x; i < n; i += stride) out[i] = (int32_t)i;
}
// The vertices with long in-lists.
__global__ void heavy_kernel(long long V, const int32_t* __restrict__ din, int32_t* __restrict__ list, long long capacity, unsigned long long* __restrict__ count) {
  const long long stride = (long long)gridDim.x * blockDim.x;
  for (long long v = (long long)blockIdx.x * blockDim.x + threadIdx.x; v < V; v += stride)
    if (din[v] > HEAVY_DEGREE) {
      const long long i = (long long)atomicAdd(count, 1ull);
      if (i < capacity) list[i] = (int32_t)v;
    }
}

// One allocation handed out in pieces: the build is mostly allocations otherwise.
struct Arena {
  char* base = nullptr;
  size_t size = 0, used = 0;
  template <class T> void plan(size_t n) { size += (n * sizeof(T) + 255) / 256 * 256; }
  bool get() { return cudaMalloc((void**)&base, size > 0 ? size : 256) == cudaSuccess; }
  template <class T> T* take(size_t n) { T* p = reinterpret_cast<T*>(base + used); used += (n * sizeof(T) + 255) / 256 * 256; return p; }
  ~Arena() { cudaFree(base); }
};

template <class T>
bool take_mem(T** p, size_t n) { return cudaMalloc((void**)p, (n > 0 ? n : 1) * sizeof(T)) == cudaSuccess; }

}  // namespace

// Floats between rows of the store for layer l: whole 32-byte sectors.
int resident_row(const taurus_ctx* c, int l) {
  const int Kp = taurus_round_up(c->dims[l], 4), Hp = taurus_round_up(c->dims[l + 1], 4);
  return taurus_round_up(c->agg_first[l] ? Kp : c->mode == TAURUS_SAGE_MEAN ? 2 * Hp : Hp, 8);
}

// In-lists (csc_ptr, csc_src; with csc_eid where a layer is sampled: built already), items of the chunk grid, heavy vertices.
int build_resident(taurus_ctx* c) {
  const long long V = c->V, E = c->E, cs = c->chunk_sources, n_chunks = (V + cs - 1) / cs;
  const int grid = c->sm_count * 8;
  int v_bit = 1, k_bit = 1;
  while (v_bit < 31 && (1ll << v_bit) < V) ++v_bit;
  while (k_bit < 31 && (1ll << k_bit) < n_chunks) ++k_bit;
  const bool have = c->d_csc_eid != nullptr;
  int32_t* const none = nullptr;
  long long* const none64 = nullptr;
  size_t scan_b = 0, sort_b = 0;
  cub::DeviceScan::ExclusiveSum(nullptr, scan_b, none64, none64, V + 1);
  if (!have && E > 0) cub::DeviceRadixSort::SortPairs(nullptr, sort_b, none, none, none, none, E, 0, v_bit);
  Arena a;
  a.plan<long long>(V + 1); a.plan<unsigned long long>(3); a.plan<char>(scan_b);
  if (!have) { a.plan<int32_t>(E); a.plan<int32_t>(E); a.plan<char>(sort_b); }
  if (!take_mem(&c->d_csc_src, (size_t)E) || !a.get()) return TAURUS_ERR_NOMEM;
  long long* at = a.take<long long>(V + 1);
  unsigned long long* heavy = a.take<unsigned long long>(3);
  void* scan = a.take<char>(scan_b);
  if (have) {
    const int rc = build_csc_src_from_eid(c);
    if (rc) return rc;
  } else {
    if (!take_mem(&c->d_csc_ptr, (size_t)V + 1)) return TAURUS_ERR_NOMEM;
    degrees_kernel<<<grid, 256>>>(V, c->d_din, c->d_csc_ptr);
    if (cub::DeviceScan::ExclusiveSum(scan, scan_b, c->d_csc_ptr, c->d_csc_ptr, V + 1) != cudaSuccess) return TAURUS_ERR_CUDA;
    if (E > 0) {
      int32_t *src = a.take<int32_t>(E), *keys = a.take<int32_t>(E);
      edge_sources_kernel<<<grid, 256>>>(V, c->d_row_ptr, src);
      if (cub::DeviceRadixSort::SortPairs(a.take<char>(sort_b), sort_b, c->d_col, keys, src, c->d_csc_src, E, 0, v_bit) != cudaSuccess) return TAURUS_ERR_CUDA;
    }
  }
  cudaMemsetAsync(heavy, 0, 3 * sizeof(*heavy));
  cudaMemsetAsync(at + V, 0, sizeof(*at));
  items_kernel<0><<<grid, 256>>>(V, (unsigned)cs, c->d_csc_ptr, c->d_csc_src, at, nullptr, nullptr, nullptr, heavy);
  if (cub::DeviceScan::ExclusiveSum(scan, scan_b, at, at, V + 1) != cudaSuccess) return TAURUS_ERR_CUDA;
  long long M = 0;
  unsigned long long count[2] = {0, 0};
  if (cudaMemcpy(&M, at + V, sizeof(M), cudaMemcpyDeviceToHost) != cudaSuccess || cudaMemcpy(count, heavy, sizeof(count), cudaMemcpyDeviceToHost) != cudaSuccess)
    return TAURUS_ERR_CUDA;
  c->n_heavy = (long long)count[0];
  c->n_heavy_segments = (long long)count[1];
  cub::DeviceRadixSort::SortPairs(nullptr, sort_b, none, none, none, none, M, 0, k_bit);
  Arena t;
  for (int k = 0; k < 6; ++k) t.plan<int32_t>(M);
  t.plan<char>(sort_b);
  if (!t.get()) return TAURUS_ERR_NOMEM;
  int32_t *key_in = t.take<int32_t>(M), *key_out = t.take<int32_t>(M), *idx_in = t.take<int32_t>(M), *idx_out = t.take<int32_t>(M), *v_in = t.take<int32_t>(M);
  uint32_t* b_in = t.take<uint32_t>(M);
  // one block of memory for the items, one for the long in-lists (freed through their first members)
  int width = 4;
  for (int l = 0; l < c->L; ++l) width = std::max(width, taurus_round_up(c->agg_first[l] ? c->dims[l] : c->dims[l + 1], 4));
  if (!take_mem(&c->d_item_v, (size_t)M * 3) || !take_mem(&c->d_item_ptr, (size_t)n_chunks + 1)) return TAURUS_ERR_NOMEM;
  c->d_item_begin = reinterpret_cast<uint32_t*>(c->d_item_v + M);
  c->d_item_count = c->d_item_v + 2 * M;
  items_kernel<1><<<grid, 256>>>(V, (unsigned)cs, c->d_csc_ptr, c->d_csc_src, at, key_in, v_in, b_in, nullptr);
  iota32_kernel<<<grid, 256>>>(M, idx_in);
  if (cub::DeviceRadixSort::SortPairs(t.take<char>(sort_b), sort_b, key_in, key_out, idx_in, idx_out, M, 0, k_bit) != cudaSuccess) return TAURUS_ERR_CUDA;
  items_order_kernel<<<grid, 256>>>(M, idx_out, v_in, b_in, c->d_csc_ptr, c->d_item_v, c->d_item_begin, c->d_item_count);
  items_bounds_kernel<<<(int)((n_chunks + 1 + 255) / 256), 256>>>(M, n_chunks, key_out, c->d_item_ptr);
  if (c->n_heavy > 0) {
    if (!take_mem(&c->d_heavy_list, (size_t)c->n_heavy * 2) || !take_mem(&c->d_heavy, (size_t)c->n_heavy_segments) ||
        !take_mem(&c->d_heavy_rows, (size_t)c->n_heavy * width)) return TAURUS_ERR_NOMEM;
    c->d_heavy_left = c->d_heavy_list + c->n_heavy;
    cudaMemsetAsync(c->d_heavy_rows, 0, (size_t)c->n_heavy * width * sizeof(float));
    heavy_kernel<<<grid, 256>>>(V, c->d_din, c->d_heavy_list, c->n_heavy, heavy + 2);
  }
  c->item_ptr.resize((size_t)n_chunks + 1);
  c->launches += 8;
  return cudaMemcpy(c->item_ptr.data(), c->d_item_ptr, (size_t)(n_chunks + 1) * sizeof(long long), cudaMemcpyDeviceToHost) == cudaSuccess ? TAURUS_OK : TAURUS_ERR_CUDA;
}

void launch_resident_reset(taurus_ctx* c, int layer, cudaStream_t st) {
  const long long work = std::max<long long>(c->V, (long long)(sizeof(DevCtl) / 8));
  const int grid = (int)std::min<long long>((work + 255) / 256, (long long)c->sm_count * 8);
  resident_reset_kernel<<<grid, 256, 0, st>>>(c->V, c->d_din, c->fanout[layer], c->d_pend, c->d_state, c->d_touch, c->d_reload, c->pool_slots, c->d_ctl);
  c->launches += 1;
}

void launch_store_rows(taurus_ctx* c, const float* X, long long ldx, int n, int K, long long src_begin, bool gcn, float* out, int ldo, cudaStream_t st,
                       const AccountWork* acc) {
  const int grid = (int)std::min<long long>(((long long)n * (ldo >> 2) + 255) / 256, (long long)c->sm_count * 8);
  if (acc)
    launch_early(c->early, store_and_account_kernel, grid + acc->blocks, 256, 0, st, X, ldx, n, K, src_begin, gcn ? 1 : 0, (const long long*)c->d_row_ptr, out, ldo,
                 AccountArgs<true>{*acc});
  else
    store_rows_kernel<<<grid, 256, 0, st>>>(X, ldx, n, K, src_begin, gcn ? 1 : 0, c->d_row_ptr, out, ldo);
  c->launches += 1;
}

// Accounting of a push.  `cell`: the chunk's number when it is one cell of the chunk grid, else -1: then edge by edge first.
AccountWork account_work(const taurus_ctx* c, const ChunkArgs& a, long long cell) {
  AccountWork w;
  w.a = a;
  w.cmask = c->d_mask_cur ? c->d_cmask : nullptr;
  w.heavy = c->n_heavy > 0 && !w.cmask ? c->d_heavy : nullptr;
  w.heavy_left = c->d_heavy_left;
  w.it = Items{c->d_item_v, c->d_item_begin, c->d_item_count};
  w.i0 = cell >= 0 ? c->item_ptr[(size_t)cell] : 0;
  w.n_items = cell >= 0 ? c->item_ptr[(size_t)cell + 1] - w.i0 : 0;
  w.blocks = 0;
  return w;
}
void launch_account(taurus_ctx* c, const ChunkArgs& a, long long cell, cudaStream_t st) {
  const AccountWork w = account_work(c, a, cell);
  if (cell >= 0) {
    const int grid = (int)std::max<long long>(1, std::min<long long>((w.n_items + 256 * ITEMS - 1) / (256 * ITEMS), (long long)c->sm_count * 6));
    account_kernel<false><<<grid, TAURUS_ACCOUNT_THREADS, 0, st>>>(w);
    c->launches += 1;
    return;
  }
  account_edges_kernel<<<c->sm_count * 8, TAURUS_ACCOUNT_THREADS, 0, st>>>(w);
  const int grid = (int)std::max<long long>(1, std::min<long long>((a.touched_capacity + 256 * ITEMS - 1) / (256 * ITEMS), (long long)c->sm_count * 6));
  // Not early: its waiting blocks would take the room that the CTAs of the projection beside it come into.  ms a pass of 500 k vertices, 6 M edges, 40 000
  // sources a push, 128 -> 128: early 1.50, behind the edges 1.28; fanout 5 1.30 and 1.02; 120 k vertices, FFMA kernel, 1.74 and 1.71.
  account_kernel<true><<<grid, TAURUS_ACCOUNT_THREADS, 0, st>>>(w);
  c->launches += 2;
}

// Sums and finished rows of the vertices the push completed, at most `bound` (aggregate-first layers: sums into A).
int launch_gather(taurus_ctx* c, const ChunkArgs& a, const float* rows, int pitch, float* A, long long bound, cudaStream_t st) {
  GatherArgs g;
  const bool sampled = c->d_mask_cur != nullptr;
  g.rows = reinterpret_cast<const float4*>(rows); g.pitch = pitch >> 2; g.vec = a.Hp >> 2;
  g.csc_ptr = c->d_csc_ptr; g.src = sampled ? c->d_kept : c->d_csc_src; g.keep = sampled ? a.fanout : 0;
  g.done_list = a.done_list;
  g.heavy = c->n_heavy > 0 && !sampled ? c->d_heavy : nullptr;
  g.heavy_rows = reinterpret_cast<float4*>(c->d_heavy_rows); g.heavy_left = c->d_heavy_left;
  g.ctl = a.ctl; g.pc = a.pc;
  g.bias = reinterpret_cast<const float4*>(a.bias);
  g.att_s = a.att_s; g.att_tm = a.att_tm; g.att_z = a.att_z;
  g.A = reinterpret_cast<float4*>(A); g.a_pitch = (c->mode == TAURUS_SAGE_MEAN ? 2 * a.Hp : a.Hp) >> 2;
  g.dense = a.dense_direct; g.dense_ld = a.dense_ld; g.grad_rows = a.grad_rows; g.grad_ids = a.grad_ids;
  g.d_out = a.d_out; g.act = a.act; g.mode = a.mode; g.heads = a.heads; g.head_vec = a.head_vec;
  g.gin_self = a.gin_self; g.leaky = a.leaky;
  g.room = !A && !a.dense_direct && a.dense_half < 0 ? a.drain_rows : 0;
  c->launches += 1;
  // Rows split over as many lanes as they have float4, steps of about 2 KB per warp.  Measured (ms of all launches of a pass):
  // 48 floats, 2.45 M vertices, 124 M edges: 16 lanes x 1 float4, 4 rows a step, 3 steps 3.9; 8 x 2 4.6 to 5.2.  64 floats, 500 k
  // vertices, 12.5 M edges: 4 rows, 3 steps 0.47; 2 rows, 4 steps 0.50; 8 x 2 0.54.  100 floats (first graph): 32 x 1, 4 rows, 3 steps
  // 7.5; 16 x 2 7.7.  256 floats: 2 rows, 4 steps 15.8; 4 rows, 3 steps 15.8, slower where in-lists are short.  GATConv (a step
  // less, for the scores), 64 floats, one head: 4 rows, 2 steps 0.66; 2 rows, 3 steps 0.71.
  const int Hp = a.Hp;
  if (Hp <= 16) return launch_g2<4, 1, 2, 4>(c, g, a, bound, 0, st);
  if (Hp <= 32) return launch_g2<8, 1, 2, 4>(c, g, a, bound, 1, st);
  if (Hp <= 64) return launch_g2<16, 1, 4, 3>(c, g, a, bound, 2, st);
  if (Hp <= 128) return launch_g2<32, 1, 4, 3>(c, g, a, bound, 3, st);
  if (Hp <= 256) return launch_g2<32, 2, 2, 4>(c, g, a, bound, 4, st);
  if (Hp <= 512) return launch_g2<32, 4, 1, 4>(c, g, a, bound, 5, st);
  return launch_g2<32, 8, 1, 3>(c, g, a, bound, 6, st);
}

void launch_resident_attention(taurus_ctx* c, cudaStream_t st) {
  const uint32_t* cmask = c->d_mask_cur ? c->d_cmask : nullptr;
  if (c->heads == 1 || c->heads == 2 || c->heads == 4 || c->heads == 8) {
    const int list_blocks = (int)std::min<long long>(c->n_heavy, (long long)c->sm_count * 4);
    const int blocks = list_blocks + (int)std::min<long long>((c->V + 31) / 32, (long long)c->sm_count * 8);
    auto run = [&](auto kernel) {
      kernel<<<blocks, 256, 0, st>>>(c->V, c->d_csc_ptr, c->d_csc_src, cmask, c->d_att_s, c->d_att_t, c->leaky, c->d_att_tm, c->d_att_z, c->d_heavy_list, c->n_heavy,
                                     list_blocks);
    };
    if (c->heads == 1) run(attention_vec_kernel<1>); else if (c->heads == 2) run(attention_vec_kernel<2>);
    else if (c->heads == 4) run(attention_vec_kernel<4>); else run(attention_vec_kernel<8>);
    c->launches += 1;
    return;
  }
  const int grid = (int)std::min<long long>((c->V + 7) / 8, (long long)c->sm_count * 8);
  attention_kernel<1><<<grid, 256, 0, st>>>(c->V, c->heads, c->d_csc_ptr, c->d_csc_src, cmask, c->d_att_s, c->d_att_t, c->leaky, c->d_att_tm, c->d_att_z,
                                            nullptr, -1, HEAVY_DEGREE);
  c->launches += 1;
  if (c->n_heavy > 0) {
    attention_kernel<8><<<(int)std::min<long long>(c->n_heavy, (long long)c->sm_count * 8), 256, 0, st>>>(
        c->n_heavy, c->heads, c->d_csc_ptr, c->d_csc_src, cmask, c->d_att_s, c->d_att_t, c->leaky, c->d_att_tm, c->d_att_z, c->d_heavy_list, HEAVY_DEGREE, 4096);
    attention_kernel<32><<<(int)std::min<long long>(c->n_heavy, (long long)c->sm_count), 1024, 0, st>>>(
        c->n_heavy, c->heads, c->d_csc_ptr, c->d_csc_src, cmask, c->d_att_s, c->d_att_t, c->leaky, c->d_att_tm, c->d_att_z, c->d_heavy_list, 4096, 0x7fffffff);
    c->launches += 2;
  }
}
