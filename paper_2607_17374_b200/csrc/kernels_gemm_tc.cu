// Projection step (S2) on the 5th-generation tensor cores: [P | T] = X . [W_neigh | W_self] with the per-row
// epilogue, for one pushed chunk (Sect. 3.6 puts the layer transform on the GPU; here it runs before the
// aggregation, which is legal by linearity, SAGEConv paragraph of Sect. 3.9).
//
// Persistent kernel: one CTA per SM walks (128-row tile of X, block of up to 256 output columns) units.  Roles (14 warps):
//   warp 0        TMA producer: cp.async.bulk.tensor loads of the raw fp32 X tile and the W operand tiles
//   warp 1        MMA issuer: tcgen05.mma, accumulators in TMEM (two buffers of up to 256 columns)
//   warps 2..5    converter: turns the raw fp32 X tile in shared memory into tensor-core operands
//                   fp32 mode : hi = x with the low 13 mantissa bits cleared (in place), lo = x - hi (exact);
//                               acc += lo.Whi + hi.Wlo + hi.Whi   (three kind::tf32 MMAs, small terms first)
//                   bf16 mode : bf16(x) in place, one kind::f16 MMA
//   warps 6..13   epilogue, two per quadrant of TMEM lanes: tcgen05.ld of the accumulator, per-row scaling / bias, 32 x 32
//                 tiles transposed through shared memory and written four rows at a time (full 128-byte lines)
// The output columns of a tile are processed in blocks of up to 256; (tile, block) units alternate between two
// TMEM accumulator buffers, so the epilogue of one unit overlaps the main loop of the next, also across tiles.
//
// fp32 mode: why two TF32 values.  Each of them has an exponent of its own, so every element of X and of W keeps 22 bits, whatever stands
// beside it in its row or column.  Two fp16 values hold as many bits and their products take two thirds of the time (65 536 rows, 256 -> 2 x 256:
// 61 us a launch against 85), but fp16's range wants one power of two for a whole row, and then an element is off by up to 2^-33 of the row's
// largest: with one raw column of 1e6 among N(0, 1), by 3.7e-5 of the result where that column has no weight.  Finding such rows ahead of their
// conversion costs 12 to 27 us a launch.
//
// Every wait on an mbarrier is bounded: after WAIT_LIMIT polls the kernel raises a CTA-wide abort flag,
// records TAURUS_ERR_INTERNAL in the control block, waits (bounded) for its TMA copies and MMAs in flight, frees its
// TMEM and returns.  Every TMA load is a plain load of the issuing CTA alone.
#include <cuda.h>
#include <cuda_bf16.h>

#include <algorithm>
#include <vector>

#include "account.cuh"
#include "stage_waits.h"
#include "taurus_internal.h"

namespace {

constexpr int BM = 128;            // rows per CTA tile (UMMA M)
constexpr int BN_MAX = 256;        // output columns per block (UMMA N)
// A product of more columns is cut into blocks of nearly the same width: a CTA keeps to one block (its bias, its weights' tiles), so a
// narrow last block (256 + 256 + 16 columns) leaves the CTAs that have it idle most of the time.  Eight launches of 65 536 rows,
// 132 -> 264 columns: 256 + 16 463 us, 144 + 128 362; 516 -> 520: 256 + 256 + 16 1 850, 3 x 176 1 610 to 1 650 (2 x 192 + 144 1 740).
constexpr int block_columns(int Np) {
  const int blocks = (Np + BN_MAX - 1) / BN_MAX;
  return ((Np + blocks - 1) / blocks + 15) / 16 * 16;
}
constexpr int OPERAND_BYTES = 192 * 1024;   // shared memory of the operand stages
constexpr int MAX_STAGES = 8;        // most of them: shorter operand rows and narrower weight tiles leave room for more (set_stages)
constexpr int TILE_A_BYTES = BM * 128;           // 128 rows x 128 B
constexpr int TILE_B_BYTES = BN_MAX * 128;       // 256 rows x 128 B
// fp32 mode: KS, the K columns per stage, is 32 (128-byte operand rows, 128-byte swizzle) or 16 (64-byte rows and swizzle: stages
// half as large, twice as many in flight).  Both are exact.  The three TF32 MMAs of a K step read their operands from shared
// memory without reuse between them (12 KB per 128 x 256 x 8 MMA, one MMA per 128 cycles at the pipe's rate), and the TMA fill and
// the operand split come on top: 272 KB of shared memory per 32 columns, 2 176 cycles at 128 B per cycle to 1 536 of the pipe.
// Counters of a launch of 65 536 rows, 256 -> 512, have the pipe at 63 % of the active cycles, shared-memory banks at 30 % (reads) and 22 %
// (writes) of their peaks, L2 at 37 %, DRAM at 20 %: nothing is full, the rest are hand-offs (load, split, MMA, release).
// Stages of 32 mean half as many of them and are the better ones while three of them fit (blocks of up to 128 columns);
// with two, wide rows want the deeper pipeline, and K up to 64 does not fill it.  us a launch of 65 536 rows, 32 / 16:
//   columns    16           96           128          160          192          256          2 x 192       2 x 256
//   K = 128    17.2 / 21.2  20.3 / 23.1  22.2 / 24.3  27.2 / 26.6
//   K = 256    27.5 / 36.3  32.8 / 38.3  35.0 / 39.1  44.7 / 41.9  47.6 / 47.3  54.3 / 52.4
//   K = 512    47.1 / 65.0  57.1 / 68.1  59.2 / 69.8  79.8 / 73.3  84.1 / 82.5  95.9 / 88.3  134.9 / 140.2  156.2 / 145.6
constexpr int stage_columns(int K, int block) { return K <= 64 || block <= 128 ? 32 : 16; }
constexpr unsigned WAIT_LIMIT = 1u << 24;
constexpr int EPI_WARPS = 8;         // two per quadrant of TMEM lanes, which take turns with the columns
constexpr int NUM_THREADS = 32 * (6 + EPI_WARPS);
constexpr int OUT_TILE_BYTES = 32 * 128;        // epilogue staging tile: 32 rows x 32 fp32, 128B-swizzled
constexpr int OUT_STAGING_BYTES = EPI_WARPS * OUT_TILE_BYTES;

struct __align__(8) Barriers {
  unsigned long long full[MAX_STAGES], conv[MAX_STAGES], empty[MAX_STAGES], acc_full[2], acc_empty[2];
  __align__(16) float bias[BN_MAX];   // of the CTA's columns (a CTA keeps to one block of columns)
  unsigned int tmem_base;
  int abort_flag;
  int loads, mmas;   // uses of the operand ring whose copies / whose MMAs have been issued (written when their warp is through)
};

// shared memory per stage: fp32 mode  X raw, then hi in place 16K | lo 16K | W hi 32K | W lo 32K    = 96 KB (KS = 32)
//                          bf16 mode  X raw in two halves, then bf16 in the first 32K | W bf16 32K   = 64 KB (64 K-columns)
// with weight tiles of 256 columns; a launch whose weight tiles are narrower runs as many stages as fit (GemmArgs::stages, stage_bytes).
constexpr int stage_bytes(bool bf16, int ks, int b_box_bytes) { return bf16 ? 2 * TILE_A_BYTES + b_box_bytes : 2 * BM * ks * 4 + 2 * b_box_bytes; }
static_assert(2 * stage_bytes(false, 32, TILE_B_BYTES) <= OPERAND_BYTES, "fp32 mode: two stages with the widest tiles,");
static_assert(3 * stage_bytes(false, 32, 128 * 128) <= OPERAND_BYTES, "three stages of 32 columns with blocks of 128 (stage_columns);");
static_assert(3 * stage_bytes(true, 64, TILE_B_BYTES) <= OPERAND_BYTES, "bf16 mode: three with any");

__device__ __forceinline__ unsigned smem_u32(const void* p) { return (unsigned)__cvta_generic_to_shared(p); }

__device__ __forceinline__ void mbar_init(unsigned long long* bar, unsigned count) {
  asm volatile("mbarrier.init.shared::cta.b64 [%0], %1;" ::"r"(smem_u32(bar)), "r"(count));
}
__device__ __forceinline__ void mbar_arrive(unsigned long long* bar) {
  asm volatile("mbarrier.arrive.shared::cta.b64 _, [%0];" ::"r"(smem_u32(bar)) : "memory");
}
__device__ __forceinline__ void mbar_expect_tx(unsigned long long* bar, unsigned bytes) {
  asm volatile("mbarrier.arrive.expect_tx.shared::cta.b64 _, [%0], %1;" ::"r"(smem_u32(bar)), "r"(bytes) : "memory");
}
__device__ __forceinline__ bool mbar_try(unsigned long long* bar, unsigned parity) {
  unsigned ok;
  asm volatile("{\n.reg .pred p;\nmbarrier.try_wait.parity.shared::cta.b64 p, [%1], %2;\nselp.u32 %0, 1, 0, p;\n}"
               : "=r"(ok) : "r"(smem_u32(bar)), "r"(parity) : "memory");
  return ok != 0;
}
// Bounded wait.  Returns false when the CTA is aborting (this wait or another one ran out).
__device__ __forceinline__ bool mbar_wait(unsigned long long* bar, unsigned parity, volatile int* abort_flag) {
  for (unsigned i = 0; i < WAIT_LIMIT; ++i) {
    if (mbar_try(bar, parity)) return true;
    if ((i & 63u) == 63u && *abort_flag) return false;
  }
  *abort_flag = 1;
  return false;
}

// The same for a whole warp: all of its lanes go on, or none (they meet again in collective instructions).
__device__ __forceinline__ bool mbar_wait_warp(unsigned long long* bar, unsigned parity, volatile int* abort_flag) {
  return __all_sync(0xffffffffu, mbar_wait(bar, parity, abort_flag));
}

__device__ __forceinline__ void tma_load_2d(void* dst, const CUtensorMap* map, int x, int y, unsigned long long* bar) {
  asm volatile("cp.async.bulk.tensor.2d.shared::cluster.global.mbarrier::complete_tx::bytes [%0], [%1, {%2, %3}], [%4];"
               ::"r"(smem_u32(dst)), "l"(map), "r"(x), "r"(y), "r"(smem_u32(bar)) : "memory");
}

// K-major operand tile with ROW-byte rows (128: 128-byte swizzle; 64: 64-byte swizzle), 8-row groups 8 * ROW bytes apart.
template <int ROW>
__device__ __forceinline__ unsigned long long umma_desc(unsigned smem_addr) {
  static_assert(ROW == 128 || ROW == 64, "operand rows of 128 or 64 bytes");
  unsigned long long d = 0;
  d |= (unsigned long long)((smem_addr & 0x3FFFFu) >> 4);   // start address
  d |= 1ull << 16;                                           // leading byte offset (unused for swizzled K-major)
  d |= (unsigned long long)((8 * ROW) >> 4) << 32;           // stride byte offset: next 8-row group
  d |= 1ull << 46;                                           // descriptor version of this architecture
  d |= (ROW == 128 ? 2ull : 4ull) << 61;                     // SWIZZLE_128B / SWIZZLE_64B
  return d;
}

__device__ __forceinline__ void umma(unsigned tmem_d, unsigned long long a, unsigned long long b, unsigned idesc,
                                     unsigned accumulate, bool tf32) {
  if (tf32)
    asm volatile("{\n.reg .pred p;\nsetp.ne.b32 p, %4, 0;\ntcgen05.mma.cta_group::1.kind::tf32 [%0], %1, %2, %3, p;\n}"
                 ::"r"(tmem_d), "l"(a), "l"(b), "r"(idesc), "r"(accumulate) : "memory");
  else
    asm volatile("{\n.reg .pred p;\nsetp.ne.b32 p, %4, 0;\ntcgen05.mma.cta_group::1.kind::f16 [%0], %1, %2, %3, p;\n}"
                 ::"r"(tmem_d), "l"(a), "l"(b), "r"(idesc), "r"(accumulate) : "memory");
}
__device__ __forceinline__ void umma_commit(unsigned long long* bar) {
  asm volatile("tcgen05.commit.cta_group::1.mbarrier::arrive::one.shared::cluster.b64 [%0];" ::"r"(smem_u32(bar)) : "memory");
}
// 32 columns of the accumulator, one row per lane.
__device__ __forceinline__ void tmem_ld32(unsigned (&v)[32], unsigned taddr) {
  asm volatile(
      "tcgen05.ld.sync.aligned.32x32b.x32.b32 {%0, %1, %2, %3, %4, %5, %6, %7, %8, %9, %10, %11, %12, %13, %14, %15, "
      "%16, %17, %18, %19, %20, %21, %22, %23, %24, %25, %26, %27, %28, %29, %30, %31}, [%32];"
      : "=r"(v[0]), "=r"(v[1]), "=r"(v[2]), "=r"(v[3]), "=r"(v[4]), "=r"(v[5]), "=r"(v[6]), "=r"(v[7]), "=r"(v[8]),
        "=r"(v[9]), "=r"(v[10]), "=r"(v[11]), "=r"(v[12]), "=r"(v[13]), "=r"(v[14]), "=r"(v[15]), "=r"(v[16]),
        "=r"(v[17]), "=r"(v[18]), "=r"(v[19]), "=r"(v[20]), "=r"(v[21]), "=r"(v[22]), "=r"(v[23]), "=r"(v[24]),
        "=r"(v[25]), "=r"(v[26]), "=r"(v[27]), "=r"(v[28]), "=r"(v[29]), "=r"(v[30]), "=r"(v[31])
      : "r"(taddr) : "memory");
  asm volatile("tcgen05.wait::ld.sync.aligned;" ::: "memory");
}
__device__ __forceinline__ void tc_fence_before() { asm volatile("tcgen05.fence::before_thread_sync;" ::: "memory"); }
__device__ __forceinline__ void tc_fence_after() { asm volatile("tcgen05.fence::after_thread_sync;" ::: "memory"); }

struct GemmArgs {
  float* PT;            // [n x N], pitch ldo
  long long ldo;
  int n, N, Np;         // rows, output columns, columns padded to a multiple of 16
  int bn;               // columns per block (the last one may have fewer)
  int k_stages;         // K in stages of KS (fp32 mode) or 64 (bf16 mode) columns
  int b_box_bytes;      // bytes one W-operand TMA box delivers (box rows x operand row bytes)
  int stages;           // operand stages in flight (2 .. MAX_STAGES)
  int stage_bytes;
  int Hp, mode, fanout;
  const float* bias;
  const long long* row_ptr;
  const int32_t* din;
  long long src_begin;
  DevCtl* ctl;
  const int32_t* done_count;   // non-null: the rows that matter are the first *done_count ones (read on the device): row tiles behind them are skipped
  int finish;           // epilogue of finished rows: act(row + fin.bias) into fin.dense[fin.done_list[row]], no store to PT
  GemmFinish fin;
};

// A CTA leaves room for a block of the accounting on its SM, and with it for the small kernels of the output stream: without it the two
// took turns.  Passes of 1.5 M vertices, 128-256-256-256, fanout 15-10-5: 12.9 -> 12.1 ms; of 2.45 M, 100-256-256-47: 36.9 -> 36.2;
// eight pushes of 65 536 rows, 256 -> 2 x 48: 823 -> 720 us.  (96 registers measure the same; at 112 the scheduler with four of the
// CTA's warps has no room for the two of the other block, although the SM as a whole has.)
constexpr int PROJECT_REGISTERS = 104;
constexpr int SHARED_BYTES = OPERAND_BYTES + OUT_STAGING_BYTES + (int)sizeof(Barriers);
static_assert(SHARED_BYTES + TAURUS_BLOCK_SHARED + TAURUS_ACCOUNT_SHARED + TAURUS_BLOCK_SHARED <= TAURUS_SM_SHARED, "shared memory for a block of the accounting");
static_assert(taurus_quarter_registers(NUM_THREADS, PROJECT_REGISTERS) + taurus_quarter_registers(TAURUS_ACCOUNT_THREADS, TAURUS_ACCOUNT_REGISTERS) <=
              TAURUS_QUARTER_REGISTERS, "registers for a block of the accounting");

// ACCOUNT: the first CTAs do the accounting of the push.
template <bool BF16, int KS, bool ACCOUNT>
__global__ void __maxnreg__(PROJECT_REGISTERS)
project_tc_kernel(const __grid_constant__ CUtensorMap map_x, const __grid_constant__ CUtensorMap map_b0, const __grid_constant__ CUtensorMap map_b1,
                  const __grid_constant__ GemmArgs g, const __grid_constant__ AccountArgs<ACCOUNT> account) {
  extern __shared__ __align__(1024) unsigned char smem[];   // (the swizzled operand tiles want 1 024)
  if ((smem_u32(smem) & 1023u) != 0) {
    if (threadIdx.x == 0) atomicCAS(&g.ctl->error, 0, TAURUS_ERR_INTERNAL);
    return;
  }
  if (account_here<TAURUS_ACCOUNT_THREADS>(account, *reinterpret_cast<AccountShared*>(smem))) return;
  // Written out in every role instead of kept in variables: those sit in the registers of threads, and with them the single thread that issues MMAs or
  // copies takes 0.1 us longer for a K step (65 536 rows, 512 -> 16: 47.8 and 54.0 us).
  auto first_unit = [&] { return (int)blockIdx.x - account.blocks(); };
  auto unit_step = [&] { return (int)gridDim.x - account.blocks(); };
  constexpr int ROW = KS * 4, A32_BYTES = BM * ROW;   // fp32 mode: bytes of an operand row, of a feature tile (raw / hi, or lo)
  const int n_stages = g.stages;
  unsigned char* out_staging = smem + OPERAND_BYTES;
  Barriers* bars = reinterpret_cast<Barriers*>(out_staging + OUT_STAGING_BYTES);
  volatile int* abort_flag = &bars->abort_flag;
  const int warp = threadIdx.x >> 5, lane = threadIdx.x & 31;
  int n_rows = g.n;
  if (g.done_count) { const int nd = *g.done_count; n_rows = nd < g.n ? nd : g.n; }   // same value in every thread
  const int n_tiles = (n_rows + BM - 1) / BM;
  const int n_blocks = (g.Np + g.bn - 1) / g.bn;
  const int tmem_cols = 512;   // two accumulator buffers of 256 columns; one CTA per SM

  if (threadIdx.x == 0) {
    for (int s = 0; s < MAX_STAGES; ++s) { mbar_init(&bars->full[s], 1); mbar_init(&bars->conv[s], 128); mbar_init(&bars->empty[s], 1); }
    for (int b = 0; b < 2; ++b) { mbar_init(&bars->acc_full[b], 1); mbar_init(&bars->acc_empty[b], EPI_WARPS); }
    bars->abort_flag = 0;
    asm volatile("fence.mbarrier_init.release.cluster;" ::: "memory");
  }
  if (warp == 1) {   // TMEM allocation by one full warp
    asm volatile("tcgen05.alloc.cta_group::1.sync.aligned.shared::cta.b32 [%0], %1;" ::"r"(smem_u32(&bars->tmem_base)), "r"(tmem_cols) : "memory");
    asm volatile("tcgen05.relinquish_alloc_permit.cta_group::1.sync.aligned;" ::: "memory");
  }
  // Bias of the CTA's columns (the grid is a multiple of n_blocks).  Read from memory where it is added, between stores to shared
  // memory, it was eight round trips in a row per 32 columns.
  for (int j = threadIdx.x; j < BN_MAX; j += NUM_THREADS) {
    const int c = first_unit() % n_blocks * g.bn + j;
    bars->bias[j] = j >= g.bn || c >= g.N || g.mode == TAURUS_GAT ? 0.f : g.finish ? g.fin.bias[c] : g.bias && c >= g.Hp ? g.bias[c - g.Hp] : 0.f;
  }
  tc_fence_before();
  __syncthreads();
  tc_fence_after();
  const unsigned tmem_base = bars->tmem_base;

  auto stage_ptr = [&](int s) { return smem + s * g.stage_bytes; };

  if (warp == 0) {
    // ---------------------------------------------------------------- TMA producer
    if (lane == 0) {
      int it = 0;
      for (int w = first_unit(); w < n_tiles * n_blocks && !*abort_flag; w += unit_step()) {
        const int tile = w / n_blocks, nb = w % n_blocks;
        const int row0 = tile * BM;
        const int col0 = nb * g.bn;
        for (int ks = 0; ks < g.k_stages; ++ks, ++it) {
          const int s = it % n_stages;
          const unsigned ph = (it / n_stages) & 1;
          if (it >= n_stages && !mbar_wait(&bars->empty[s], ph ^ 1, abort_flag)) break;
          unsigned char* st = stage_ptr(s);
          if (BF16) {
            mbar_expect_tx(&bars->full[s], 2 * TILE_A_BYTES + g.b_box_bytes);
            tma_load_2d(st, &map_x, ks * 64, row0, &bars->full[s]);
            tma_load_2d(st + TILE_A_BYTES, &map_x, ks * 64 + 32, row0, &bars->full[s]);
            tma_load_2d(st + 2 * TILE_A_BYTES, &map_b0, ks * 64, col0, &bars->full[s]);
          } else {
            mbar_expect_tx(&bars->full[s], A32_BYTES + 2 * g.b_box_bytes);
            tma_load_2d(st, &map_x, ks * KS, row0, &bars->full[s]);
            tma_load_2d(st + 2 * A32_BYTES, &map_b0, ks * KS, col0, &bars->full[s]);
            tma_load_2d(st + 2 * A32_BYTES + g.b_box_bytes, &map_b1, ks * KS, col0, &bars->full[s]);
          }
        }
      }
      bars->loads = it;
    }
  } else if (warp == 1) {
    // ---------------------------------------------------------------- MMA issuer
    if (lane == 0) {
      int it = 0, unit = 0;
      for (int w = first_unit(); w < n_tiles * n_blocks && !*abort_flag; w += unit_step(), ++unit) {
        const int nb = w % n_blocks;
        const int bw = (g.Np - nb * g.bn) < g.bn ? (g.Np - nb * g.bn) : g.bn;
        const int buf = unit & 1;
        if (unit >= 2 && !mbar_wait(&bars->acc_empty[buf], ((unit >> 1) & 1) ^ 1, abort_flag)) break;
        tc_fence_after();
        const unsigned tmem_d = tmem_base + (unsigned)(buf * BN_MAX);
        const unsigned idesc = (1u << 4) | ((BF16 ? 1u : 2u) << 7) | ((BF16 ? 1u : 2u) << 10) |
                               ((unsigned)(bw >> 3) << 17) | ((unsigned)(BM >> 4) << 24);
        bool ok = true;
        for (int ks = 0; ks < g.k_stages; ++ks, ++it) {
          const int s = it % n_stages;
          const unsigned ph = (it / n_stages) & 1;
          if (!mbar_wait(&bars->conv[s], ph, abort_flag)) { ok = false; break; }
          tc_fence_after();
          const unsigned base = smem_u32(stage_ptr(s));
          if (BF16) {
            const unsigned long long da = umma_desc<128>(base), db = umma_desc<128>(base + 2 * TILE_A_BYTES);
#pragma unroll
            for (int kk = 0; kk < 4; ++kk) umma(tmem_d, da + 2 * kk, db + 2 * kk, idesc, (ks | kk) != 0, false);
          } else {
            const unsigned long long a_hi = umma_desc<ROW>(base), a_lo = umma_desc<ROW>(base + A32_BYTES);
            const unsigned long long b_hi = umma_desc<ROW>(base + 2 * A32_BYTES), b_lo = umma_desc<ROW>(base + 2 * A32_BYTES + g.b_box_bytes);
#pragma unroll
            for (int kk = 0; kk < KS / 8; ++kk) {
              umma(tmem_d, a_lo + 2 * kk, b_hi + 2 * kk, idesc, (ks | kk) != 0, true);
              umma(tmem_d, a_hi + 2 * kk, b_lo + 2 * kk, idesc, 1u, true);
              umma(tmem_d, a_hi + 2 * kk, b_hi + 2 * kk, idesc, 1u, true);
            }
          }
          umma_commit(&bars->empty[s]);    // stage reusable once these MMAs have read it
        }
        if (!ok) break;
        umma_commit(&bars->acc_full[buf]);  // accumulator of this block complete
      }
      bars->mmas = it;
    }
  } else if (warp < 6) {
    // ---------------------------------------------------------------- converter (128 threads)
    const int t = threadIdx.x - 64;
    int it = 0;
    for (int w = first_unit(); w < n_tiles * n_blocks && !*abort_flag; w += unit_step()) {
      bool ok = true;
      for (int ks = 0; ks < g.k_stages; ++ks, ++it) {
        const int s = it % n_stages;
        const unsigned ph = (it / n_stages) & 1;
        if (!mbar_wait(&bars->full[s], ph, abort_flag)) { ok = false; break; }
        unsigned char* st = stage_ptr(s);
        if (BF16) {
          // A thread to a row.  Raw half h holds columns 32h .. 32h + 31; a row is 128 bytes before and after, and logical 16-byte chunk c
          // of row r sits at chunk c ^ (r & 7).
          unsigned char* const row = st + t * 128;
          uint4 o[8];
#pragma unroll
          for (int c = 0; c < 8; ++c) {
            const unsigned char* const raw = row + (c >> 2) * TILE_A_BYTES;
            const float4 v0 = *reinterpret_cast<const float4*>(raw + (((2 * (c & 3)) ^ (t & 7)) << 4));
            const float4 v1 = *reinterpret_cast<const float4*>(raw + (((2 * (c & 3) + 1) ^ (t & 7)) << 4));
            __nv_bfloat162 b0 = __floats2bfloat162_rn(v0.x, v0.y), b1 = __floats2bfloat162_rn(v0.z, v0.w);
            __nv_bfloat162 b2 = __floats2bfloat162_rn(v1.x, v1.y), b3 = __floats2bfloat162_rn(v1.z, v1.w);
            o[c].x = *reinterpret_cast<unsigned*>(&b0); o[c].y = *reinterpret_cast<unsigned*>(&b1);
            o[c].z = *reinterpret_cast<unsigned*>(&b2); o[c].w = *reinterpret_cast<unsigned*>(&b3);
          }
#pragma unroll
          for (int c = 0; c < 8; ++c) *reinterpret_cast<uint4*>(row + ((c ^ (t & 7)) << 4)) = o[c];
        } else {
          // element-wise and layout-preserving: the swizzle does not matter
          float4* hi = reinterpret_cast<float4*>(st);
          float4* lo = reinterpret_cast<float4*>(st + A32_BYTES);
#pragma unroll
          for (int i = 0; i < A32_BYTES / 16 / 128; ++i) {
            const int idx = t + i * 128;
            float4 x = hi[idx], h4, l4;
            h4.x = __uint_as_float(__float_as_uint(x.x) & 0xFFFFE000u); l4.x = x.x - h4.x;
            h4.y = __uint_as_float(__float_as_uint(x.y) & 0xFFFFE000u); l4.y = x.y - h4.y;
            h4.z = __uint_as_float(__float_as_uint(x.z) & 0xFFFFE000u); l4.z = x.z - h4.z;
            h4.w = __uint_as_float(__float_as_uint(x.w) & 0xFFFFE000u); l4.w = x.w - h4.w;
            hi[idx] = h4; lo[idx] = l4;
          }
        }
        asm volatile("fence.proxy.async.shared::cta;" ::: "memory");   // generic-proxy writes -> visible to the tensor core
        mbar_arrive(&bars->conv[s]);
      }
      if (!ok) break;
    }
  } else {
    // ---------------------------------------------------------------- epilogue (warps 6..13, TMEM lanes 32 * (warp % 4))
    const int q = warp & 3, half = (warp - 6) >> 2;
    // this warp's staging tile: 32 rows (lane = row) x 32 columns, 16-byte chunk c of row r at chunk c ^ (r & 7)
    unsigned char* const tile_smem = out_staging + (warp - 6) * OUT_TILE_BYTES;
    int unit = 0;
    for (int w = first_unit(); w < n_tiles * n_blocks; w += unit_step(), ++unit) {   // (an abort ends it in the wait, for the warp as one)
    const int tile = w / n_blocks, nb = w % n_blocks;
    const int r = tile * BM + q * 32 + lane;
    float c_out = 1.f, self_mul = 1.f;
    int vrow = -1;        // finish mode: the vertex this lane's row belongs to
    if (g.finish) {
      if (r < g.n && r < *g.done_count && !g.ctl->error) {
        vrow = g.fin.done_list[r];
        if (nb == 0 && half == 0) g.fin.state[vrow] = TAURUS_COMPLETED;
      }
    } else if (r < g.n) {
      const long long u = g.src_begin + r;
      if (g.mode == TAURUS_GCN_SYM) {
        c_out = (float)(1.0 / sqrt((double)(g.row_ptr[u + 1] - g.row_ptr[u]) + 1.0));
      } else if (g.mode == TAURUS_SAGE_MEAN) {
        const int d = g.din[u];
        const int m = (g.fanout > 0 && d > g.fanout) ? g.fanout : d;
        self_mul = (float)(m > 1 ? m : 1);
      }
    }
    {
      const int buf = unit & 1;
      if (!mbar_wait_warp(&bars->acc_full[buf], (unit >> 1) & 1, abort_flag)) break;
      tc_fence_after();
      const int columns = g.bn < g.N - nb * g.bn ? g.bn : g.N - nb * g.bn;   // without the padding of the last block
#pragma unroll 1
      for (int c0 = half * 32; c0 < columns; c0 += 64) {
        unsigned v[32];
        tmem_ld32(v, tmem_base + ((unsigned)(q * 32) << 16) + (unsigned)(buf * BN_MAX + c0));
        const int cbase = nb * g.bn + c0;
        float o[32];
        if (cbase + 32 <= g.Hp && !g.finish) {   // P columns: c_out(u) * (x W_neigh)
#pragma unroll
          for (int j = 0; j < 32; ++j) o[j] = __uint_as_float(v[j]) * c_out;
        } else {
#pragma unroll
          for (int j = 0; j < 32; j += 4) {
            const float4 b = *reinterpret_cast<const float4*>(&bars->bias[c0 + j]);   // zero in P columns
            // T columns: (x W_self + b) * max(|M(u)|, 1); finished rows: act(x W + b); GAT: the attention scalars as they are
            const float mul = g.finish ? 1.f : cbase + j >= g.Hp ? self_mul : c_out;
            o[j] = (__uint_as_float(v[j]) + b.x) * mul; o[j + 1] = (__uint_as_float(v[j + 1]) + b.y) * mul;
            o[j + 2] = (__uint_as_float(v[j + 2]) + b.z) * mul; o[j + 3] = (__uint_as_float(v[j + 3]) + b.w) * mul;
          }
          if (g.finish && g.fin.act)
#pragma unroll
            for (int j = 0; j < 32; ++j) o[j] = fmaxf(o[j], 0.f);
        }
#pragma unroll
        for (int j = 0; j < 32; j += 4)
          *reinterpret_cast<float4*>(tile_smem + lane * 128 + (((j >> 2) ^ (lane & 7)) << 4)) = make_float4(o[j], o[j + 1], o[j + 2], o[j + 3]);
        // Transposed through the staging tile: the warp writes four rows per step, each as one 128-byte piece.  (TMA stores of the
        // tile queue up behind the operand loads.)
        __syncwarp();
        const int ch = lane & 7;
        const bool in = c0 + ch * 4 < columns;
#pragma unroll
        for (int it = 0; it < 8; ++it) {
          const int rr = it * 4 + (lane >> 3);
          const float4 y = *reinterpret_cast<const float4*>(tile_smem + rr * 128 + ((ch ^ (rr & 7)) << 4));
          if (g.finish) {
            const int vv = __shfl_sync(0xffffffffu, vrow, rr);
            if (vv >= 0 && in) *reinterpret_cast<float4*>(g.fin.dense + (size_t)vv * g.fin.dense_ld + cbase + ch * 4) = y;
          } else {
            const int row = tile * BM + q * 32 + rr;
            if (row < n_rows && in) *reinterpret_cast<float4*>(g.PT + (size_t)row * g.ldo + cbase + ch * 4) = y;
          }
        }
        __syncwarp();   // the tile is rewritten in the next round
      }
      tc_fence_before();
      __syncwarp();
      if (lane == 0) mbar_arrive(&bars->acc_empty[buf]);   // one arrival a warp: they are taken one after the other
    }
    }
  }

  // ---------------------------------------------------------------- teardown
  __syncthreads();
  if (*abort_flag) {
    if (threadIdx.x == 0) {
      atomicCAS(&g.ctl->error, 0, TAURUS_ERR_INTERNAL);
      // the copies and MMAs on their way get a bounded time to end before shared memory and TMEM are released
      wait_last_phases(bars->loads, n_stages, 1u << 16, [&](int s, unsigned parity) { return mbar_try(&bars->full[s], parity); });
      wait_last_phases(bars->mmas, n_stages, 1u << 16, [&](int s, unsigned parity) { return mbar_try(&bars->empty[s], parity); });
    }
    __syncthreads();
  }
  if (warp == 1) {
    tc_fence_after();
    asm volatile("tcgen05.dealloc.cta_group::1.sync.aligned.b32 %0, %1;" ::"r"(tmem_base), "r"(tmem_cols) : "memory");
  }
}

// ------------------------------------------------------------------------------------------------ host side
typedef CUresult (*EncodeTiledFn)(CUtensorMap*, CUtensorMapDataType, cuuint32_t, void*, const cuuint64_t*, const cuuint64_t*,
                                  const cuuint32_t*, const cuuint32_t*, CUtensorMapInterleave, CUtensorMapSwizzle,
                                  CUtensorMapL2promotion, CUtensorMapFloatOOBfill);

EncodeTiledFn encode_fn() {
  static EncodeTiledFn fn = nullptr;
  static bool tried = false;
  if (!tried) {
    tried = true;
    void* p = nullptr;
    cudaDriverEntryPointQueryResult qres;
    if (cudaGetDriverEntryPoint("cuTensorMapEncodeTiled", &p, cudaEnableDefault, &qres) == cudaSuccess &&
        qres == cudaDriverEntryPointSuccess)
      fn = reinterpret_cast<EncodeTiledFn>(p);
    else
      cudaGetLastError();
  }
  return fn;
}

// 2-D row-major tensor [rows x cols] of `elem` bytes, box [box_rows x box_cols], 128-byte swizzle, zero fill
// on loads.
bool make_map(CUtensorMap* m, const void* base, CUtensorMapDataType dt, int elem, long long rows, long long cols,
              long long ld_elems, int box_rows, int box_cols) {
  EncodeTiledFn fn = encode_fn();
  if (!fn) return false;
  cuuint64_t dims[2] = {(cuuint64_t)cols, (cuuint64_t)rows};
  cuuint64_t strides[1] = {(cuuint64_t)ld_elems * elem};
  cuuint32_t box[2] = {(cuuint32_t)box_cols, (cuuint32_t)box_rows};
  cuuint32_t estr[2] = {1, 1};
  const CUtensorMapSwizzle swz = box_cols * elem == 64 ? CU_TENSOR_MAP_SWIZZLE_64B : CU_TENSOR_MAP_SWIZZLE_128B;   // box rows of 64 or 128 bytes
  return fn(m, dt, 2, const_cast<void*>(base), dims, strides, box, estr, CU_TENSOR_MAP_INTERLEAVE_NONE,
            swz, CU_TENSOR_MAP_L2_PROMOTION_L2_128B, CU_TENSOR_MAP_FLOAT_OOB_FILL_NONE) == CUDA_SUCCESS;
}

// Stages that fit the shared memory of the operands.
void set_stages(GemmArgs& g, bool bf16, int ks) {
  g.stage_bytes = stage_bytes(bf16, ks, g.b_box_bytes);
  g.stages = std::min(OPERAND_BYTES / g.stage_bytes, MAX_STAGES);
}

// A product's operands on the device: the tensor maps of X and W (fp32 mode: W's high and low parts).
struct Maps { CUtensorMap x, hi, lo; };

template <bool BF16, int KS, bool ACCOUNT>
int launch_tc2(taurus_ctx* c, int grid, cudaStream_t st, const Maps& m, const GemmArgs& g, const AccountArgs<ACCOUNT>& acc) {
  bool& set = c->tc_smem_set[(ACCOUNT ? 1 : 0) + (KS == 16 ? 2 : 0)];   // once per context (the attribute belongs to the context's device)
  if (!set) {
    if (cudaFuncSetAttribute(project_tc_kernel<BF16, KS, ACCOUNT>, cudaFuncAttributeMaxDynamicSharedMemorySize, SHARED_BYTES) != cudaSuccess) {
      cudaGetLastError();
      return TAURUS_ERR_CUDA;
    }
    set = true;
  }
  launch_early(c->early, project_tc_kernel<BF16, KS, ACCOUNT>, grid, NUM_THREADS, SHARED_BYTES, st, m.x, m.hi, m.lo, g, acc);
  return TAURUS_OK;
}
template <bool ACCOUNT>
int launch_tc1(taurus_ctx* c, int grid, cudaStream_t st, const Maps& m, const GemmArgs& g, bool bf16, int ks, const AccountArgs<ACCOUNT>& acc) {
  if (bf16) return launch_tc2<true, 32, ACCOUNT>(c, grid, st, m, g, acc);
  return ks == 32 ? launch_tc2<false, 32, ACCOUNT>(c, grid, st, m, g, acc) : launch_tc2<false, 16, ACCOUNT>(c, grid, st, m, g, acc);
}
int launch_tc(taurus_ctx* c, int grid, cudaStream_t st, const Maps& m, const GemmArgs& g, bool bf16, int ks, const AccountWork* acc = nullptr) {
  if (acc) return launch_tc1<true>(c, grid + acc->blocks, st, m, g, bf16, ks, AccountArgs<true>{*acc});
  return launch_tc1<false>(c, grid, st, m, g, bf16, ks, AccountArgs<false>());
}

// Per-layer tensor-core images of Wcat, K-major: [Np x Kp].
struct WImage {
  void* hi = nullptr;   // fp32 mode: tf32-exact high part; bf16 mode: bf16 weights
  void* lo = nullptr;   // fp32 mode: residual
  int Np = 0, Kp = 0, ks = 0;   // ks: K columns per stage
  CUtensorMap map_hi, map_lo;
};

}  // namespace

int prepare_tc_weights(taurus_ctx* c, void** slot, const std::vector<float>& cat, int K, int N) {
  const bool bf16 = c->gemm_mode == TAURUS_GEMM_BF16;
  WImage* w = new WImage();
  *slot = w;
  w->Np = taurus_round_up(N, 16);
  const int bw = block_columns(w->Np);
  w->ks = bf16 ? 64 : stage_columns(K, bw);
  w->Kp = taurus_round_up(K, w->ks);
  const size_t cnt = (size_t)w->Np * w->Kp;
  if (bf16) {
    std::vector<__nv_bfloat16> img(cnt, __float2bfloat16(0.f));
    for (int k = 0; k < K; ++k)
      for (int j = 0; j < N; ++j) img[(size_t)j * w->Kp + k] = __float2bfloat16(cat[(size_t)k * N + j]);
    if (cudaMalloc(&w->hi, cnt * 2) != cudaSuccess) return TAURUS_ERR_NOMEM;
    if (cudaMemcpy(w->hi, img.data(), cnt * 2, cudaMemcpyHostToDevice) != cudaSuccess) return TAURUS_ERR_CUDA;
    if (!make_map(&w->map_hi, w->hi, CU_TENSOR_MAP_DATA_TYPE_BFLOAT16, 2, w->Np, w->Kp, w->Kp, bw, 64)) return TAURUS_ERR_CUDA;
    w->map_lo = w->map_hi;
  } else {
    std::vector<float> hi(cnt, 0.f), lo(cnt, 0.f);
    for (int k = 0; k < K; ++k)
      for (int j = 0; j < N; ++j) {
        float x = cat[(size_t)k * N + j];
        uint32_t b; memcpy(&b, &x, 4); b &= 0xFFFFE000u;
        float h; memcpy(&h, &b, 4);
        float l = x - h;
        uint32_t lb; memcpy(&lb, &l, 4); lb &= 0xFFFFE000u; memcpy(&l, &lb, 4);
        hi[(size_t)j * w->Kp + k] = h;
        lo[(size_t)j * w->Kp + k] = l;
      }
    if (cudaMalloc(&w->hi, cnt * 4) != cudaSuccess || cudaMalloc(&w->lo, cnt * 4) != cudaSuccess) return TAURUS_ERR_NOMEM;
    if (cudaMemcpy(w->hi, hi.data(), cnt * 4, cudaMemcpyHostToDevice) != cudaSuccess ||
        cudaMemcpy(w->lo, lo.data(), cnt * 4, cudaMemcpyHostToDevice) != cudaSuccess) return TAURUS_ERR_CUDA;
    if (!make_map(&w->map_hi, w->hi, CU_TENSOR_MAP_DATA_TYPE_FLOAT32, 4, w->Np, w->Kp, w->Kp, bw, w->ks) ||
        !make_map(&w->map_lo, w->lo, CU_TENSOR_MAP_DATA_TYPE_FLOAT32, 4, w->Np, w->Kp, w->Kp, bw, w->ks)) return TAURUS_ERR_CUDA;
  }
  return TAURUS_OK;
}

void free_tc_weights(taurus_ctx* c) {
  for (int l = 0; l < 2 * TAURUS_MAX_LAYERS; ++l) {
    void** slot = l < TAURUS_MAX_LAYERS ? &c->tc_image[l] : &c->tc_image_af[l - TAURUS_MAX_LAYERS];
    WImage* w = static_cast<WImage*>(*slot);
    if (!w) continue;
    cudaFree(w->hi); cudaFree(w->lo);
    delete w;
    *slot = nullptr;
  }
}

// Shapes the tensor-core kernel takes: feature rows that TMA can address (16-byte aligned base and pitch).
bool project_tc_usable(const taurus_ctx* c, int layer, const float* X, int ldx) {
  if (c->flags & TAURUS_FLAG_SIMT_GEMM) return false;
  if (!c->tc_image[layer] || !encode_fn()) return false;
  if ((ldx & 3) != 0 || (reinterpret_cast<uintptr_t>(X) & 15) != 0) return false;
  return true;
}

int project_tc_units(const taurus_ctx* c, int layer, int n) {
  const int Np = static_cast<const WImage*>(c->tc_image[layer])->Np, bn = block_columns(Np);
  return (n + BM - 1) / BM * ((Np + bn - 1) / bn);
}

int launch_project_tc(taurus_ctx* c, int layer, const float* X, int ldx, long long src_begin, int n, float* out, int ldo, cudaStream_t st,
                      const AccountWork* acc) {
  const bool bf16 = c->gemm_mode == TAURUS_GEMM_BF16;
  WImage* w = static_cast<WImage*>(c->tc_image[layer]);
  const int K = c->dims[layer], Hp = taurus_round_up(c->dims[layer + 1], 4);
  const int N = taurus_proj_width(c->mode, Hp, c->heads);
  Maps m;
  m.hi = w->map_hi; m.lo = w->map_lo;
  if (!make_map(&m.x, X, CU_TENSOR_MAP_DATA_TYPE_FLOAT32, 4, n, K, ldx, BM, bf16 ? 32 : w->ks)) return TAURUS_ERR_CUDA;
  GemmArgs g;
  g.PT = out; g.ldo = ldo; g.n = n; g.N = N; g.Np = w->Np; g.k_stages = w->Kp / w->ks;
  g.bn = block_columns(w->Np);
  g.b_box_bytes = g.bn * (bf16 ? 128 : w->ks * 4);
  set_stages(g, bf16, w->ks);
  g.Hp = Hp; g.mode = c->mode; g.fanout = c->fanout[layer]; g.bias = c->d_bias[layer];
  g.row_ptr = c->d_row_ptr; g.din = c->d_din; g.src_begin = src_begin; g.ctl = c->d_ctl;
  g.finish = 0; g.fin = GemmFinish(); g.done_count = nullptr;
  const int n_tiles = (n + BM - 1) / BM;
  const int n_blocks = (w->Np + g.bn - 1) / g.bn, n_units = n_tiles * n_blocks;
  const int sms = c->sm_count - c->xfer_blocks;   // the SMs of the row transfers have no shared memory left
  const int grid = n_units < sms ? n_units : std::max(1, sms / n_blocks) * n_blocks;   // a CTA keeps to one block of columns
  const int rc = launch_tc(c, grid, st, m, g, bf16, w->ks, acc);
  if (rc) return rc;
  c->launches += 1;
  return TAURUS_OK;
}

// Plain product on the tensor cores: out[n x N] (pitch ld_out floats) = X[n x K] (pitch ldx) . columns
// [col0, col0 + N) of the layer's weight image, no epilogue scaling (used when a layer aggregates raw rows
// first and transforms the finished rows afterwards).  col0 and N are multiples of 4.
bool gemm_plain_tc_usable(const taurus_ctx* c, const void* image, const float* X, int ldx, const float* out, long long ld_out) {
  if (c->flags & TAURUS_FLAG_SIMT_GEMM) return false;
  if (!image || !encode_fn()) return false;
  if ((ldx & 3) != 0 || (reinterpret_cast<uintptr_t>(X) & 15) != 0) return false;
  if ((ld_out & 3) != 0 || (reinterpret_cast<uintptr_t>(out) & 15) != 0) return false;
  return true;
}

int launch_gemm_plain_tc(taurus_ctx* c, void* image, int col0, int N, const float* X, int ldx, int K, int n, float* out, long long ld_out,
                         cudaStream_t st, const GemmFinish* finish, const int32_t* done_count) {
  if (n <= 0) return TAURUS_OK;
  if (finish && ((N & 3) != 0 || (finish->dense_ld & 3) != 0 || (reinterpret_cast<uintptr_t>(finish->dense) & 15) != 0)) return TAURUS_ERR_INTERNAL;
  const bool bf16 = c->gemm_mode == TAURUS_GEMM_BF16;
  WImage* w = static_cast<WImage*>(image);
  const int rows_left = w->Np - col0;                       // image rows (= output columns) from col0 on
  const int Np = std::min(taurus_round_up(N, 16), rows_left);
  const int bw = block_columns(Np);
  const int elem = bf16 ? 2 : 4;
  Maps m;
  if (!make_map(&m.x, X, CU_TENSOR_MAP_DATA_TYPE_FLOAT32, 4, n, K, ldx, BM, bf16 ? 32 : w->ks)) return TAURUS_ERR_CUDA;
  const char* hi = static_cast<const char*>(w->hi) + (size_t)col0 * w->Kp * elem;
  if (!make_map(&m.hi, hi, bf16 ? CU_TENSOR_MAP_DATA_TYPE_BFLOAT16 : CU_TENSOR_MAP_DATA_TYPE_FLOAT32, elem, rows_left, w->Kp, w->Kp, bw,
                w->ks))
    return TAURUS_ERR_CUDA;
  m.lo = m.hi;
  if (!bf16) {
    const char* lo = static_cast<const char*>(w->lo) + (size_t)col0 * w->Kp * elem;
    if (!make_map(&m.lo, lo, CU_TENSOR_MAP_DATA_TYPE_FLOAT32, 4, rows_left, w->Kp, w->Kp, bw, w->ks)) return TAURUS_ERR_CUDA;
  }
  GemmArgs g;
  g.PT = out; g.ldo = ld_out; g.n = n; g.N = N; g.Np = Np; g.k_stages = w->Kp / w->ks;
  g.bn = bw;
  g.b_box_bytes = bw * (bf16 ? 128 : w->ks * 4);
  set_stages(g, bf16, w->ks);
  g.Hp = N; g.mode = TAURUS_GIN_SUM; g.fanout = 0; g.bias = nullptr;
  g.row_ptr = c->d_row_ptr; g.din = c->d_din; g.src_begin = 0; g.ctl = c->d_ctl;
  g.finish = finish ? 1 : 0; g.fin = finish ? *finish : GemmFinish();
  g.done_count = done_count;
  const int n_tiles = (n + BM - 1) / BM;
  const int n_blocks = (Np + bw - 1) / bw, n_units = n_tiles * n_blocks;
  const int sms = c->sm_count - c->xfer_blocks;   // the SMs of the row transfers have no shared memory left
  const int grid = n_units < sms ? n_units : std::max(1, sms / n_blocks) * n_blocks;   // a CTA keeps to one block of columns
  const int rc = launch_tc(c, grid, st, m, g, bf16, w->ks);
  if (rc) return rc;
  c->launches += 1;
  return TAURUS_OK;
}
