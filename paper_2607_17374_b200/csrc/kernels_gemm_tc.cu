// Projection step (S2) on the 5th-generation tensor cores: [P | T] = X . [W_neigh | W_self] with the per-row
// epilogue, for one pushed chunk (Sect. 3.6 puts the layer transform on the GPU; here it runs before the
// aggregation, which is legal by linearity, SAGEConv paragraph of Sect. 3.9).
//
// Persistent kernel: one CTA per SM walks (128-row tile of X, block of up to 256 output columns) units.  Roles (15 warps):
//   warp 0        TMA loads of the raw fp32 X tile, a ring of its own: a tile waits for memory, then for its conversion
//   warp 14       TMA loads of the W operand tiles (from L2, as they are)
//   warp 1        MMA issuer: tcgen05.mma, accumulators in TMEM (two buffers of up to 256 columns)
//   warps 2..5    converter, a thread to a row: turns the raw fp32 X tile in shared memory into tensor-core operands, in place
//                   fp32 mode : x times a power of two of its row = hi + lo, two fp16 values rounded to nearest;
//                               acc += lo.Whi + hi.Wlo + hi.Whi   (three kind::f16 MMAs, small terms first)
//                   bf16 mode : bf16(x), one kind::f16 MMA
//   warps 6..13   epilogue, two per quadrant of TMEM lanes: tcgen05.ld of the accumulator, per-row scaling / bias, 32 x 32
//                 tiles transposed through shared memory and written four rows at a time (full 128-byte lines)
// The output columns of a tile are processed in blocks of up to 256; (tile, block) units alternate between two
// TMEM accumulator buffers, so the epilogue of one unit overlaps the main loop of the next, also across tiles.
//
// fp32 mode: why two fp16 values.  fp16 and tf32 both hold 11 bits, so hi + lo carry the same 22 bits of x either way, but fp16
// operands take half the shared memory and run at twice the rate.  What fp16 lacks is range, hence the powers of two: W is scaled
// at init so that its largest magnitude lies in [2^14, 2^15), a row of X so that the largest magnitude of its first K step with a
// nonzero value lies in [2^7, 2^8).  A later value that would not fit (2^15: more than 128 times that one) lowers the row's power
// of two, and the converter brings what the row has accumulated so far to the new one in TMEM.  The epilogue takes all of them out
// again, exactly.  Elements down to 2^-21 of a row's largest keep all their bits, smaller ones are off by at most 2^-33 of it.
// Rows with infinities or NaN give NaN.  (Finding a row's largest value before its first conversion costs 12 to 27 us a launch of
// 65 536 rows, more than half of what the cheaper operands win.)  Errors against 64 bits, norm of a row: N(0, 1) rows 256 -> 256
// 2.2e-6 as two tf32 values that the tensor core truncates, 0.9e-6 now; a third to a half as large on every kind of row tried.
// us a launch of 65 536 rows, two tf32 values / now:
//   K -> N    64 -> 64    100 -> 64   128 -> 128  256 -> 96   256 -> 192  256 -> 256  256 -> 512  512 -> 64   512 -> 256
//             14.5/14.3   19.1/17.8   22.6/20.8   34.0/28.2   47.1/32.8   52.1/37.4   85.3/61.1   49.5/43.7   88.3/57.6
// What bounds it: narrow products the row pieces of 128 B that a K step reads (4.5 TB/s: with nothing else in the kernel 35 of the
// 43.7 us of 512 -> 64).  Wide ones: nothing is full.  256 -> 512: a K step of a block takes 1 660 cycles, 768 of them MMAs (the pipe is busy 46 % of
// the active cycles); the L1 pipeline, which the conversion and the epilogue's transposition and stores share, is at 61 %, shared-memory
// banks at 25 % (reads) and 20 % (writes), L2 at 28 %, DRAM at 27 %.  Without the epilogue a launch takes 47.6 of 63.5 us, without its
// stores 55.5, without the conversion 56.6, without all but loads and MMAs 40.  Tried and slower: two threads to a row in eight warps
// (70 us), the epilogue's rows straight from registers in 32-byte pieces (78), the next accumulator piece loaded ahead of the stores and L2 promotion
// of 256 B (the same); one ring for X and W was 0.5 to 3 us a launch slower than the two.
//
// Every wait on an mbarrier is bounded: after WAIT_LIMIT polls the kernel raises a CTA-wide abort flag,
// records TAURUS_ERR_INTERNAL in the control block, waits (bounded) for its TMA copies and MMAs in flight, frees its
// TMEM and returns.  Every TMA load is a plain load of the issuing CTA alone.
#include <cuda.h>
#include <cuda_bf16.h>
#include <cuda_fp16.h>

#include <algorithm>
#include <cmath>
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
constexpr int OPERAND_BYTES = 192 * 1024;        // shared memory of the operand stages
constexpr int MAX_X = 8, MAX_W = 5;             // stages of the two rings; narrower weight tiles leave room for more (set_stages)
constexpr int TILE_A_BYTES = BM * 128;           // 128 rows x 128 B
constexpr int TILE_B_BYTES = BN_MAX * 128;       // 256 rows x 128 B
constexpr int KS = 32;                           // fp32 mode: K columns per stage; an operand row is [hi | lo], 64 B each (bf16 mode: 64 columns)
constexpr unsigned WAIT_LIMIT = 1u << 24;
constexpr int EPI_WARPS = 8;         // two per quadrant of TMEM lanes, which take turns with the columns
constexpr int CONV_WARPS = 4, EPI_FIRST = 2 + CONV_WARPS, W_WARP = EPI_FIRST + EPI_WARPS;
constexpr int NUM_THREADS = 32 * (W_WARP + 1);
constexpr int OUT_TILE_BYTES = 32 * 128;        // epilogue staging tile: 32 rows x 32 fp32, 128B-swizzled
constexpr int OUT_STAGING_BYTES = EPI_WARPS * OUT_TILE_BYTES;

struct __align__(8) Barriers {
  unsigned long long full[MAX_X], conv[MAX_X], empty[MAX_X], w_full[MAX_W], w_empty[MAX_W], acc_full[2], acc_empty[2];
  __align__(16) float bias[BN_MAX];   // of the CTA's columns (a CTA keeps to one block of columns)
  unsigned char row_exp[2][BM];       // fp32 mode: exponent fields of the factors that take the rows' powers of two out again, for two units,
  __align__(16) unsigned char col_exp[BN_MAX];   //   and of the square roots of those of the CTA's columns (applied twice: no overflow in between)
  unsigned int tmem_base;
  int abort_flag;
  int loads, w_loads, mmas;   // uses of the operand rings whose copies / whose MMAs have been issued (written when their warp is through)
};

// shared memory per stage: fp32 mode  A raw, then [hi | lo] in place 16K      | B [hi | lo] 32K   (32 K-columns)
//                          bf16 mode  A raw in two halves, then bf16 in the first 32K | B bf16 32K      (64 K-columns)
// with weight tiles of 256 columns.

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

// K-major operand tile with 128-byte rows and 128-byte swizzle, 8-row groups 1 024 bytes apart.
__device__ __forceinline__ unsigned long long umma_desc(unsigned smem_addr) {
  unsigned long long d = 0;
  d |= (unsigned long long)((smem_addr & 0x3FFFFu) >> 4);   // start address
  d |= 1ull << 16;                                           // leading byte offset (unused for swizzled K-major)
  d |= (unsigned long long)(1024 >> 4) << 32;                // stride byte offset: next 8-row group
  d |= 1ull << 46;                                           // descriptor version of this architecture
  d |= 2ull << 61;                                           // SWIZZLE_128B
  return d;
}

__device__ __forceinline__ void umma(unsigned tmem_d, unsigned long long a, unsigned long long b, unsigned idesc, unsigned accumulate) {
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
__device__ __forceinline__ float power_of_two(unsigned field) { return __uint_as_float(field << 23); }   // 2^(field - 127)
// One row of the accumulator per lane, `columns` (a multiple of 8) of them, times a * b.
__device__ __forceinline__ void tmem_scale(unsigned taddr, int columns, float a, float b) {
#pragma unroll 1
  for (int c = 0; c < columns; c += 8) {
    unsigned v[8];
    asm volatile("tcgen05.ld.sync.aligned.32x32b.x8.b32 {%0, %1, %2, %3, %4, %5, %6, %7}, [%8];"
                 : "=r"(v[0]), "=r"(v[1]), "=r"(v[2]), "=r"(v[3]), "=r"(v[4]), "=r"(v[5]), "=r"(v[6]), "=r"(v[7]) : "r"(taddr + (unsigned)c) : "memory");
    asm volatile("tcgen05.wait::ld.sync.aligned;" ::: "memory");
#pragma unroll
    for (int i = 0; i < 8; ++i) v[i] = __float_as_uint(__uint_as_float(v[i]) * a * b);
    asm volatile("tcgen05.st.sync.aligned.32x32b.x8.b32 [%0], {%1, %2, %3, %4, %5, %6, %7, %8};"
                 ::"r"(taddr + (unsigned)c), "r"(v[0]), "r"(v[1]), "r"(v[2]), "r"(v[3]), "r"(v[4]), "r"(v[5]), "r"(v[6]), "r"(v[7]) : "memory");
  }
  asm volatile("tcgen05.wait::st.sync.aligned;" ::: "memory");
}
// Two floats as the fp16 pairs hi and lo, each rounded to nearest.
__device__ __forceinline__ void split2(float x, float y, unsigned& hi, unsigned& lo) {
  const __half2 h = __floats2half2_rn(x, y);
  const float2 f = __half22float2(h);
  const __half2 l = __floats2half2_rn(x - f.x, y - f.y);
  hi = *reinterpret_cast<const unsigned*>(&h);
  lo = *reinterpret_cast<const unsigned*>(&l);
}
__device__ __forceinline__ void tc_fence_before() { asm volatile("tcgen05.fence::before_thread_sync;" ::: "memory"); }
__device__ __forceinline__ void tc_fence_after() { asm volatile("tcgen05.fence::after_thread_sync;" ::: "memory"); }

// Where a role stands in the ring of operand stages: stage, and parity of the phase it is in there.
struct Ring {
  int s = 0;
  unsigned phase = 0;
  __device__ __forceinline__ void next(int stages) { if (++s == stages) { s = 0; phase ^= 1; } }
};

struct GemmArgs {
  float* PT;            // [n x N], pitch ldo
  long long ldo;
  int n, N, Np;         // rows, output columns, columns padded to a multiple of 16
  int bn;               // columns per block (the last one may have fewer)
  int k_stages;         // K in stages of 32 (fp32 mode) or 64 (bf16 mode) columns
  int b_box_bytes;      // bytes one W-operand TMA box delivers (box rows x 128 B)
  int x_stages, w_stages;   // stages of the two rings
  float w_down;         // fp32 mode: takes the power of two of W out again, where all its columns have the same one,
  const unsigned char* col_exp;   //   else NULL here: [Np] exponent fields of the columns (Barriers::col_exp), and 1
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
static_assert(3 * (2 * TILE_A_BYTES + TILE_B_BYTES) <= OPERAND_BYTES, "three stages of the widest tiles with either operand type");
static_assert(taurus_quarter_registers(NUM_THREADS, PROJECT_REGISTERS) + taurus_quarter_registers(TAURUS_ACCOUNT_THREADS, TAURUS_ACCOUNT_REGISTERS) <=
              TAURUS_QUARTER_REGISTERS, "registers for a block of the accounting");

// ACCOUNT: the first CTAs do the accounting of the push.
template <bool BF16, bool ACCOUNT>
__global__ void __maxnreg__(PROJECT_REGISTERS)
project_tc_kernel(const __grid_constant__ CUtensorMap map_x, const __grid_constant__ CUtensorMap map_b, const __grid_constant__ GemmArgs g,
                  const __grid_constant__ AccountArgs<ACCOUNT> account) {
  extern __shared__ __align__(1024) unsigned char smem[];   // (the swizzled operand tiles want 1 024)
  if ((smem_u32(smem) & 1023u) != 0) {
    if (threadIdx.x == 0) atomicCAS(&g.ctl->error, 0, TAURUS_ERR_INTERNAL);
    return;
  }
  if (account_here<TAURUS_ACCOUNT_THREADS>(account, *reinterpret_cast<AccountShared*>(smem))) return;
  const int cta = (int)blockIdx.x - account.blocks(), ctas = (int)gridDim.x - account.blocks();
  constexpr int X_BYTES = BF16 ? 2 * TILE_A_BYTES : TILE_A_BYTES;
  const int x_stages = g.x_stages, w_stages = g.w_stages;
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
    for (int s = 0; s < MAX_X; ++s) { mbar_init(&bars->full[s], 1); mbar_init(&bars->conv[s], CONV_WARPS); mbar_init(&bars->empty[s], 1); }
    for (int s = 0; s < MAX_W; ++s) { mbar_init(&bars->w_full[s], 1); mbar_init(&bars->w_empty[s], 1); }
    for (int b = 0; b < 2; ++b) { mbar_init(&bars->acc_full[b], BF16 ? 1 : 1 + CONV_WARPS); mbar_init(&bars->acc_empty[b], EPI_WARPS); }
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
    const int c = cta % n_blocks * g.bn + j;
    bars->bias[j] = j >= g.bn || c >= g.N || g.mode == TAURUS_GAT ? 0.f : g.finish ? g.fin.bias[c] : g.bias && c >= g.Hp ? g.bias[c - g.Hp] : 0.f;
    if (!BF16 && g.col_exp) bars->col_exp[j] = j >= g.bn || c >= g.N ? 127 : g.col_exp[c];
  }
  tc_fence_before();
  __syncthreads();
  tc_fence_after();
  const unsigned tmem_base = bars->tmem_base;

  auto x_ptr = [&](int s) { return smem + s * X_BYTES; };
  unsigned char* const w_smem = smem + x_stages * X_BYTES;

  if (warp == 0 || warp == W_WARP) {
    // ---------------------------------------------------------------- TMA producers
    if (lane == 0) {
      const bool x = warp == 0;
      const int stages = x ? x_stages : w_stages;
      int it = 0;
      Ring ring;
      for (int w = cta; w < n_tiles * n_blocks && !*abort_flag; w += ctas) {
        const int row0 = w / n_blocks * BM, col0 = w % n_blocks * g.bn;
        for (int ks = 0; ks < g.k_stages; ++ks, ++it, ring.next(stages)) {
          const int s = ring.s;
          unsigned long long* const full = x ? &bars->full[s] : &bars->w_full[s];
          if (it >= stages && !mbar_wait(x ? &bars->empty[s] : &bars->w_empty[s], ring.phase ^ 1, abort_flag)) break;
          mbar_expect_tx(full, x ? X_BYTES : g.b_box_bytes);
          if (!x) {
            tma_load_2d(w_smem + s * g.b_box_bytes, &map_b, ks * 64, col0, full);
          } else if (BF16) {
            tma_load_2d(x_ptr(s), &map_x, ks * 64, row0, full);
            tma_load_2d(x_ptr(s) + TILE_A_BYTES, &map_x, ks * 64 + 32, row0, full);
          } else {
            tma_load_2d(x_ptr(s), &map_x, ks * KS, row0, full);
          }
        }
      }
      if (x) bars->loads = it; else bars->w_loads = it;
    }
  } else if (warp == 1) {
    // ---------------------------------------------------------------- MMA issuer
    if (lane == 0) {
      int it = 0, unit = 0;
      Ring ring, wring;
      for (int w = cta; w < n_tiles * n_blocks && !*abort_flag; w += ctas, ++unit) {
        const int nb = w % n_blocks;
        const int bw = (g.Np - nb * g.bn) < g.bn ? (g.Np - nb * g.bn) : g.bn;
        const int buf = unit & 1;
        if (unit >= 2 && !mbar_wait(&bars->acc_empty[buf], ((unit >> 1) & 1) ^ 1, abort_flag)) break;
        tc_fence_after();
        const unsigned tmem_d = tmem_base + (unsigned)(buf * BN_MAX);
        const unsigned idesc = (1u << 4) | ((BF16 ? 1u : 0u) << 7) | ((BF16 ? 1u : 0u) << 10) |
                               ((unsigned)(bw >> 3) << 17) | ((unsigned)(BM >> 4) << 24);
        bool ok = true;
        for (int ks = 0; ks < g.k_stages; ++ks, ++it, ring.next(x_stages), wring.next(w_stages)) {
          if (!mbar_wait(&bars->w_full[wring.s], wring.phase, abort_flag) || !mbar_wait(&bars->conv[ring.s], ring.phase, abort_flag)) { ok = false; break; }
          tc_fence_after();
          const unsigned long long a = umma_desc(smem_u32(x_ptr(ring.s))), b = umma_desc(smem_u32(w_smem) + wring.s * g.b_box_bytes);
          if (BF16) {
#pragma unroll
            for (int kk = 0; kk < 4; ++kk) umma(tmem_d, a + 2 * kk, b + 2 * kk, idesc, (ks | kk) != 0);
          } else {   // lo: 64 B behind hi
#pragma unroll
            for (int kk = 0; kk < KS / 16; ++kk) {
              umma(tmem_d, a + 4 + 2 * kk, b + 2 * kk, idesc, (ks | kk) != 0);
              umma(tmem_d, a + 2 * kk, b + 4 + 2 * kk, idesc, 1u);
              umma(tmem_d, a + 2 * kk, b + 2 * kk, idesc, 1u);
            }
          }
          umma_commit(&bars->empty[ring.s]);      // stages reusable once these MMAs have read them
          umma_commit(&bars->w_empty[wring.s]);
        }
        if (!ok) break;
        umma_commit(&bars->acc_full[buf]);  // accumulator of this block complete
      }
      bars->mmas = it;
    }
  } else if (warp < EPI_FIRST) {
    // ---------------------------------------------------------------- converter
    const int q = warp & 3, row = q * 32 + lane, swz = row & 7;   // the row is one of the TMEM lanes the warp can reach
    int unit = 0;
    Ring ring;
    for (int w = cta; w < n_tiles * n_blocks; w += ctas, ++unit) {   // (an abort ends it in a wait, for the warp as one)
      bool ok = true;
      int field = 0;   // fp32 mode: exponent field of the row's power of two; 0: nothing but zeros so far
      for (int ks = 0; ks < g.k_stages; ++ks, ring.next(x_stages)) {
        const int s = ring.s;
        const unsigned ph = ring.phase;
        if (!mbar_wait_warp(&bars->full[s], ph, abort_flag)) { ok = false; break; }
        // a tile row is 128 bytes before and after; logical 16-byte chunk c of it sits at chunk c ^ (row & 7)
        unsigned char* const at = x_ptr(s) + row * 128;
        if (BF16) {
          uint4 o[8];
#pragma unroll
          for (int c = 0; c < 8; ++c) {   // tile h holds columns 32h .. 32h + 31
            const unsigned char* const raw = at + (c >> 2) * TILE_A_BYTES;
            const float4 v0 = *reinterpret_cast<const float4*>(raw + (((2 * (c & 3)) ^ swz) << 4));
            const float4 v1 = *reinterpret_cast<const float4*>(raw + (((2 * (c & 3) + 1) ^ swz) << 4));
            __nv_bfloat162 b0 = __floats2bfloat162_rn(v0.x, v0.y), b1 = __floats2bfloat162_rn(v0.z, v0.w);
            __nv_bfloat162 b2 = __floats2bfloat162_rn(v1.x, v1.y), b3 = __floats2bfloat162_rn(v1.z, v1.w);
            o[c].x = *reinterpret_cast<unsigned*>(&b0); o[c].y = *reinterpret_cast<unsigned*>(&b1);
            o[c].z = *reinterpret_cast<unsigned*>(&b2); o[c].w = *reinterpret_cast<unsigned*>(&b3);
          }
#pragma unroll
          for (int c = 0; c < 8; ++c) *reinterpret_cast<uint4*>(at + ((c ^ swz) << 4)) = o[c];
        } else {
          float x[KS];
#pragma unroll
          for (int c = 0; c < 8; ++c) {
            const float4 v = *reinterpret_cast<const float4*>(at + ((c ^ swz) << 4));
            x[4 * c] = v.x; x[4 * c + 1] = v.y; x[4 * c + 2] = v.z; x[4 * c + 3] = v.w;
          }
          float top[4] = {0.f, 0.f, 0.f, 0.f};
#pragma unroll
          for (int j = 0; j < KS; ++j) top[j & 3] = fmaxf(top[j & 3], fabsf(x[j]));
          top[0] = fmaxf(fmaxf(top[0], top[1]), fmaxf(top[2], top[3]));
          const int e = (int)(__float_as_uint(top[0]) >> 23);   // 255: the row is lost to an infinity, whatever its power of two
          const int want = e == 255 ? 127 : min(max(261 - e, 7), 247);
          const bool shrink = field != 0 && e != 255 && e + field >= 269;   // some |x| 2^(field - 127) >= 2^15
          if (__any_sync(0xffffffffu, shrink)) {
            // sums of this unit so far, once the MMAs of the stage before this one are through (the first stage has no field yet)
            if (!mbar_wait_warp(&bars->empty[s == 0 ? x_stages - 1 : s - 1], s == 0 ? ph ^ 1 : ph, abort_flag)) { ok = false; break; }
            tc_fence_after();
            const int d = shrink ? want - field : 0, nb = w % n_blocks;
            tmem_scale(tmem_base + ((unsigned)(q * 32) << 16) + (unsigned)((unit & 1) * BN_MAX), min(g.bn, g.Np - nb * g.bn), power_of_two(127 + d / 2),
                       power_of_two(127 + d - d / 2));
            tc_fence_before();
            if (shrink) field = want;
          }
          if (field == 0 && top[0] != 0.f) field = want;
          const float up = power_of_two(field);
#pragma unroll
          for (int c = 0; c < 4; ++c) {
            uint4 hi, lo;
            split2(x[8 * c] * up, x[8 * c + 1] * up, hi.x, lo.x);
            split2(x[8 * c + 2] * up, x[8 * c + 3] * up, hi.y, lo.y);
            split2(x[8 * c + 4] * up, x[8 * c + 5] * up, hi.z, lo.z);
            split2(x[8 * c + 6] * up, x[8 * c + 7] * up, hi.w, lo.w);
            *reinterpret_cast<uint4*>(at + ((c ^ swz) << 4)) = hi;
            *reinterpret_cast<uint4*>(at + (((c + 4) ^ swz) << 4)) = lo;
          }
          if (ks == g.k_stages - 1) {   // what the epilogue multiplies with
            if (unit >= 2 && !mbar_wait_warp(&bars->acc_empty[unit & 1], ((unit >> 1) & 1) ^ 1, abort_flag)) { ok = false; break; }
            bars->row_exp[unit & 1][row] = (unsigned char)(254 - (field == 0 ? 127 : field));
            __syncwarp();
            if (lane == 0) mbar_arrive(&bars->acc_full[unit & 1]);
          }
        }
        asm volatile("fence.proxy.async.shared::cta;" ::: "memory");   // generic-proxy writes -> visible to the tensor core
        __syncwarp();
        if (lane == 0) mbar_arrive(&bars->conv[s]);   // one arrival a warp: they are taken one after the other
      }
      if (!ok) break;
    }
  } else {
    // ---------------------------------------------------------------- epilogue (warps 6..13, TMEM lanes 32 * (warp % 4))
    const int q = warp & 3, half = (warp - EPI_FIRST) >> 2;
    // this warp's staging tile: 32 rows (lane = row) x 32 columns, 16-byte chunk c of row r at chunk c ^ (r & 7)
    unsigned char* const tile_smem = out_staging + (warp - EPI_FIRST) * OUT_TILE_BYTES;
    int unit = 0;
    for (int w = cta; w < n_tiles * n_blocks; w += ctas, ++unit) {   // (an abort ends it in the wait, for the warp as one)
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
      const float row_down = BF16 ? 1.f : power_of_two(bars->row_exp[buf][q * 32 + lane]) * g.w_down;   // (both exact)
      const float down = BF16 || g.col_exp ? 1.f : row_down;
      const int columns = g.bn < g.N - nb * g.bn ? g.bn : g.N - nb * g.bn;   // without the padding of the last block
#pragma unroll 1
      for (int c0 = half * 32; c0 < columns; c0 += 64) {
        unsigned v[32];
        tmem_ld32(v, tmem_base + ((unsigned)(q * 32) << 16) + (unsigned)(buf * BN_MAX + c0));
        const int cbase = nb * g.bn + c0;
        float o[32];
        if (!BF16 && g.col_exp) {   // out with the powers of two of the columns
#pragma unroll
          for (int j = 0; j < 32; j += 4) {
            const unsigned f = *reinterpret_cast<const unsigned*>(&bars->col_exp[c0 + j]);
#pragma unroll
            for (int i = 0; i < 4; ++i) {
              const float h = power_of_two((f >> (8 * i)) & 255u);
              v[j + i] = __float_as_uint(__uint_as_float(v[j + i]) * h * row_down * h);   // (the row's in between: no overflow on the way)
            }
          }
        }
        if (cbase + 32 <= g.Hp && !g.finish) {   // P columns: c_out(u) * (x W_neigh)
#pragma unroll
          for (int j = 0; j < 32; ++j) o[j] = __uint_as_float(v[j]) * down * c_out;
        } else {
#pragma unroll
          for (int j = 0; j < 32; j += 4) {
            const float4 b = *reinterpret_cast<const float4*>(&bars->bias[c0 + j]);   // zero in P columns
            // T columns: (x W_self + b) * max(|M(u)|, 1); finished rows: act(x W + b); GAT: the attention scalars as they are
            const float mul = g.finish ? 1.f : cbase + j >= g.Hp ? self_mul : c_out;
            o[j] = fmaf(__uint_as_float(v[j]), down, b.x) * mul; o[j + 1] = fmaf(__uint_as_float(v[j + 1]), down, b.y) * mul;
            o[j + 2] = fmaf(__uint_as_float(v[j + 2]), down, b.z) * mul; o[j + 3] = fmaf(__uint_as_float(v[j + 3]), down, b.w) * mul;
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
      if (lane == 0) mbar_arrive(&bars->acc_empty[buf]);
    }
    }
  }

  // ---------------------------------------------------------------- teardown
  __syncthreads();
  if (*abort_flag) {
    if (threadIdx.x == 0) {
      atomicCAS(&g.ctl->error, 0, TAURUS_ERR_INTERNAL);
      // the copies and MMAs on their way get a bounded time to end before shared memory and TMEM are released
      wait_last_phases(bars->loads, x_stages, 1u << 16, [&](int s, unsigned parity) { return mbar_try(&bars->full[s], parity); });
      wait_last_phases(bars->w_loads, w_stages, 1u << 16, [&](int s, unsigned parity) { return mbar_try(&bars->w_full[s], parity); });
      wait_last_phases(bars->mmas, x_stages, 1u << 16, [&](int s, unsigned parity) { return mbar_try(&bars->empty[s], parity); });
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

// 2-D row-major tensor [rows x cols] of `elem` bytes, box [box_rows x box_cols] of 128-byte rows, 128-byte swizzle, zero fill
// on loads.
bool make_map(CUtensorMap* m, const void* base, CUtensorMapDataType dt, int elem, long long rows, long long cols,
              long long ld_elems, int box_rows, int box_cols) {
  EncodeTiledFn fn = encode_fn();
  if (!fn) return false;
  cuuint64_t dims[2] = {(cuuint64_t)cols, (cuuint64_t)rows};
  cuuint64_t strides[1] = {(cuuint64_t)ld_elems * elem};
  cuuint32_t box[2] = {(cuuint32_t)box_cols, (cuuint32_t)box_rows};
  cuuint32_t estr[2] = {1, 1};
  return fn(m, dt, 2, const_cast<void*>(base), dims, strides, box, estr, CU_TENSOR_MAP_INTERLEAVE_NONE,
            CU_TENSOR_MAP_SWIZZLE_128B, CU_TENSOR_MAP_L2_PROMOTION_L2_128B, CU_TENSOR_MAP_FLOAT_OOB_FILL_NONE) == CUDA_SUCCESS;
}

// Stages that fit the shared memory of the operands: three of W, or as many as half of what eight of X leave takes, the rest for X.
void set_stages(GemmArgs& g, bool bf16) {
  const int x_bytes = bf16 ? 2 * TILE_A_BYTES : TILE_A_BYTES;
  g.w_stages = std::min(std::max((OPERAND_BYTES - MAX_X * TILE_A_BYTES) / g.b_box_bytes, 3), MAX_W);
  g.x_stages = std::min((OPERAND_BYTES - g.w_stages * g.b_box_bytes) / x_bytes, MAX_X);
}

template <bool BF16, bool ACCOUNT>
int launch_tc2(taurus_ctx* c, int grid, cudaStream_t st, const CUtensorMap& map_x, const CUtensorMap& map_b, const GemmArgs& g, const AccountArgs<ACCOUNT>& acc) {
  bool& set = c->tc_smem_set[ACCOUNT ? 1 : 0];   // once per context (the attribute belongs to the context's device)
  if (!set) {
    if (cudaFuncSetAttribute(project_tc_kernel<BF16, ACCOUNT>, cudaFuncAttributeMaxDynamicSharedMemorySize, SHARED_BYTES) != cudaSuccess) {
      cudaGetLastError();
      return TAURUS_ERR_CUDA;
    }
    set = true;
  }
  launch_early(c->early, project_tc_kernel<BF16, ACCOUNT>, grid, NUM_THREADS, SHARED_BYTES, st, map_x, map_b, g, acc);
  return TAURUS_OK;
}
int launch_tc(taurus_ctx* c, int grid, cudaStream_t st, const CUtensorMap& map_x, const CUtensorMap& map_b, const GemmArgs& g, bool bf16,
              const AccountWork* acc = nullptr) {
  if (acc) {
    const AccountArgs<true> with{*acc};
    return bf16 ? launch_tc2<true, true>(c, grid + acc->blocks, st, map_x, map_b, g, with) : launch_tc2<false, true>(c, grid + acc->blocks, st, map_x, map_b, g, with);
  }
  const AccountArgs<false> without;
  return bf16 ? launch_tc2<true, false>(c, grid, st, map_x, map_b, g, without) : launch_tc2<false, false>(c, grid, st, map_x, map_b, g, without);
}

// Per-layer tensor-core images of Wcat, K-major: a row per output column.
struct WImage {
  void* data = nullptr;            // bf16 mode: [Np x Kp] bf16 weights; fp32 mode: [Np x 2 Kp] fp16, per 32 K-columns [hi | lo] of w times a power of two:
  float down = 1.f;                //   1 / that power, where the columns share one,
  unsigned char* exp = nullptr;    //   else [Np] exponent fields of the square roots of 1 / the columns' powers
  int Np = 0, Kp = 0, ks = 0;      // ks: K columns per stage
  int row() const { return ks == 64 ? Kp : 2 * Kp; }   // values per row
  CUtensorMap map;
};
bool make_w_map(CUtensorMap* m, const WImage* w, bool bf16, int col0, int box_rows) {   // columns from col0 on
  return make_map(m, static_cast<const char*>(w->data) + (size_t)col0 * w->row() * 2, bf16 ? CU_TENSOR_MAP_DATA_TYPE_BFLOAT16 : CU_TENSOR_MAP_DATA_TYPE_FLOAT16, 2,
                  w->Np - col0, w->row(), w->row(), box_rows, 64);
}

}  // namespace

int prepare_tc_weights(taurus_ctx* c, void** slot, const std::vector<float>& cat, int K, int N) {
  const bool bf16 = c->gemm_mode == TAURUS_GEMM_BF16;
  WImage* w = new WImage();
  *slot = w;
  w->Np = taurus_round_up(N, 16);
  const int bw = block_columns(w->Np);
  w->ks = bf16 ? 64 : KS;
  w->Kp = taurus_round_up(K, w->ks);
  const size_t cnt = (size_t)w->Np * w->row();
  if (cudaMalloc(&w->data, cnt * 2) != cudaSuccess) return TAURUS_ERR_NOMEM;
  if (bf16) {
    std::vector<__nv_bfloat16> img(cnt, __float2bfloat16(0.f));
    for (int k = 0; k < K; ++k)
      for (int j = 0; j < N; ++j) img[(size_t)j * w->Kp + k] = __float2bfloat16(cat[(size_t)k * N + j]);
    if (cudaMemcpy(w->data, img.data(), cnt * 2, cudaMemcpyHostToDevice) != cudaSuccess) return TAURUS_ERR_CUDA;
  } else {
    std::vector<__half> img(cnt, __float2half_rn(0.f));
    std::vector<unsigned char> fields((size_t)w->Np, 127);
    // One power of two for all columns, which takes the largest magnitude to [2^14, 2^15), where that leaves every column its 22 bits
    // (2^-10 of the largest: off by at most 2^-29 of its own) and its product with a row's is a float; else one a column, even,
    // so that the epilogue can apply its square root on either side of the row's.
    std::vector<float> top((size_t)N, 0.f), up((size_t)N, 1.f);
    bool shared = true;
    for (int k = 0; k < K; ++k)
      for (int j = 0; j < N; ++j) {
        const float x = std::fabs(cat[(size_t)k * N + j]);
        if (x > top[(size_t)j] || std::isnan(x)) top[(size_t)j] = x;   // (a NaN stays)
      }
    float most = 0.f;
    for (int j = 0; j < N; ++j) { shared = shared && std::isfinite(top[(size_t)j]); most = std::max(most, top[(size_t)j]); }
    const int all = shared && most > 0.f ? 14 - std::ilogb(most) : 0;
    shared = shared && all >= -6 && all <= 28;
    for (int j = 0; j < N; ++j) shared = shared && (top[(size_t)j] == 0.f || std::ilogb(top[(size_t)j]) >= 4 - all);
    for (int j = 0; j < N; ++j) {
      int f = shared ? all : 0;
      if (!shared && top[(size_t)j] > 0.f && std::isfinite(top[(size_t)j])) f = std::min(std::max(14 - std::ilogb(top[(size_t)j]), -120), 120) & ~1;
      fields[(size_t)j] = (unsigned char)(127 - f / 2);
      up[(size_t)j] = std::ldexp(1.f, f);
    }
    for (int k = 0; k < K; ++k)
      for (int j = 0; j < N; ++j) {
        const float x = cat[(size_t)k * N + j] * up[(size_t)j];
        const __half h = __float2half_rn(x);
        __half* to = &img[(size_t)j * w->row() + (size_t)(k / KS) * (2 * KS) + k % KS];
        to[0] = h; to[KS] = __float2half_rn(x - __half2float(h));
      }
    w->down = shared ? std::ldexp(1.f, -all) : 1.f;
    if (!shared && cudaMalloc((void**)&w->exp, fields.size()) != cudaSuccess) return TAURUS_ERR_NOMEM;
    if (cudaMemcpy(w->data, img.data(), cnt * 2, cudaMemcpyHostToDevice) != cudaSuccess ||
        (w->exp && cudaMemcpy(w->exp, fields.data(), fields.size(), cudaMemcpyHostToDevice) != cudaSuccess)) return TAURUS_ERR_CUDA;
  }
  return make_w_map(&w->map, w, bf16, 0, bw) ? TAURUS_OK : TAURUS_ERR_CUDA;
}

void free_tc_weights(taurus_ctx* c) {
  for (int l = 0; l < 2 * TAURUS_MAX_LAYERS; ++l) {
    void** slot = l < TAURUS_MAX_LAYERS ? &c->tc_image[l] : &c->tc_image_af[l - TAURUS_MAX_LAYERS];
    WImage* w = static_cast<WImage*>(*slot);
    if (!w) continue;
    cudaFree(w->data); cudaFree(w->exp);
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
  CUtensorMap map_x;
  if (!make_map(&map_x, X, CU_TENSOR_MAP_DATA_TYPE_FLOAT32, 4, n, K, ldx, BM, 32)) return TAURUS_ERR_CUDA;
  GemmArgs g;
  g.PT = out; g.ldo = ldo; g.n = n; g.N = N; g.Np = w->Np; g.k_stages = w->Kp / w->ks;
  g.bn = block_columns(w->Np);
  g.b_box_bytes = g.bn * 128;
  set_stages(g, bf16);
  g.w_down = w->down; g.col_exp = w->exp;
  g.Hp = Hp; g.mode = c->mode; g.fanout = c->fanout[layer]; g.bias = c->d_bias[layer];
  g.row_ptr = c->d_row_ptr; g.din = c->d_din; g.src_begin = src_begin; g.ctl = c->d_ctl;
  g.finish = 0; g.fin = GemmFinish(); g.done_count = nullptr;
  const int n_tiles = (n + BM - 1) / BM;
  const int n_blocks = (w->Np + g.bn - 1) / g.bn, n_units = n_tiles * n_blocks;
  const int sms = c->sm_count - c->xfer_blocks;   // the SMs of the row transfers have no shared memory left
  const int grid = n_units < sms ? n_units : std::max(1, sms / n_blocks) * n_blocks;   // a CTA keeps to one block of columns
  const int rc = launch_tc(c, grid, st, map_x, w->map, g, bf16, acc);
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
  const int Np = std::min(taurus_round_up(N, 16), w->Np - col0);
  const int bw = block_columns(Np);
  CUtensorMap map_x, map_b;
  if (!make_map(&map_x, X, CU_TENSOR_MAP_DATA_TYPE_FLOAT32, 4, n, K, ldx, BM, 32) || !make_w_map(&map_b, w, bf16, col0, bw)) return TAURUS_ERR_CUDA;
  GemmArgs g;
  g.PT = out; g.ldo = ld_out; g.n = n; g.N = N; g.Np = Np; g.k_stages = w->Kp / w->ks;
  g.bn = bw;
  g.b_box_bytes = bw * 128;
  set_stages(g, bf16);
  g.w_down = w->down; g.col_exp = w->exp ? w->exp + col0 : nullptr;
  g.Hp = N; g.mode = TAURUS_GIN_SUM; g.fanout = 0; g.bias = nullptr;
  g.row_ptr = c->d_row_ptr; g.din = c->d_din; g.src_begin = 0; g.ctl = c->d_ctl;
  g.finish = finish ? 1 : 0; g.fin = finish ? *finish : GemmFinish();
  g.done_count = done_count;
  const int n_tiles = (n + BM - 1) / BM;
  const int n_blocks = (Np + bw - 1) / bw, n_units = n_tiles * n_blocks;
  const int sms = c->sm_count - c->xfer_blocks;   // the SMs of the row transfers have no shared memory left
  const int grid = n_units < sms ? n_units : std::max(1, sms / n_blocks) * n_blocks;   // a CTA keeps to one block of columns
  const int rc = launch_tc(c, grid, st, map_x, map_b, g, bf16);
  if (rc) return rc;
  c->launches += 1;
  return TAURUS_OK;
}
