// Projection step (S2) as a plain fp32 FFMA GEMM: [P | T] = X . [W_neigh | W_self] with the per-row
// epilogue.  Exact fp32 arithmetic; kept as the reference shim for the tensor-core kernel and as the
// fallback for shapes that kernel does not take (TAURUS_FLAG_SIMT_GEMM selects it explicitly).
//
// Epilogue (project-then-aggregate is legal by linearity, SAGEConv paragraph of Sect. 3.9):
//   P_u = c_out(u) * (x_u W_neigh)                        message every out-neighbour receives
//   T_u = (x_u W_self + b) * max(|M(u)|, 1)     (SAGE)    self message, pre-multiplied by 1 / c_in(u) so
//                                                          that finalise is one multiply by c_in
//   (GCN has no T columns: its self message P_u + b / c_in(u) is formed by the scatter kernel.)
#include "account.cuh"
#include "taurus_internal.h"

#define BM 32
#define BN 64
#define BK 32
#define SIMT_STAGES 3

// A block of 128 threads takes 32 rows x 64 columns, a thread 4 x 4 of them.  Panels of 32 K-columns arrive by cp.async (4 bytes
// at a time from X, whose rows need no alignment), three in flight: one panel after the other, loaded and waited for, was 3.9 us
// each, most of a small launch.  Additions are packed in pairs of columns, fma by fma in the order of K.  With blocks of 64 x 64, a
// panel of 16 at a time, and now: 10 007 rows, 130 -> 48: 35 and 14.3 us; 700 rows, 47 -> 72: 9.5 and 4.8 us.  65 536 rows (a layer
// whose width is no multiple of 4 comes here with its full chunks): 130 -> 264 259 and 193 us, 47 -> 72 50 and 42.
// ACCOUNT: the first blocks do the accounting of the push.  A block's tile is one of `across` side by side.
template <bool ACCOUNT>
__global__ void __launch_bounds__(128) project_simt_kernel(const float* __restrict__ X, int ldx, int K, const float* __restrict__ W,
                                                           int ldw, int N, float* __restrict__ PT, long long ldo, int n, int Hp, int mode,
                                                           const float* __restrict__ bias, const long long* __restrict__ row_ptr,
                                                           const int32_t* __restrict__ din, int fanout, long long src_begin, int across,
                                                           const __grid_constant__ AccountArgs<ACCOUNT> account) {
  __shared__ __align__(16) float sA[SIMT_STAGES][BM][BK + 4];   // [row][k]
  if (account_here<128>(account, *reinterpret_cast<AccountShared*>(sA))) return;
  const int tile = (int)blockIdx.x - account.blocks();
  __shared__ __align__(16) float sB[SIMT_STAGES][BK][BN];
  const int t = threadIdx.x, tx = t % 16, ty = t / 16;
  const int row0 = tile / across * BM, col0 = tile % across * BN;
  auto load = [&](int s, int k0) {   // zero behind the ends
    if (k0 < K) {
#pragma unroll
      for (int i = 0; i < BM * BK / 128; ++i) {
        const int r = (t >> 5) + i * 4, k = t & 31;
        const bool in = row0 + r < n && k0 + k < K;
        const float* src = in ? X + (size_t)(row0 + r) * ldx + k0 + k : X;
        asm volatile("cp.async.ca.shared.global [%0], [%1], 4, %2;" ::"r"((unsigned)__cvta_generic_to_shared(&sA[s][r][k])), "l"(src), "r"(in ? 4 : 0) : "memory");
      }
#pragma unroll
      for (int i = 0; i < BK * BN / 4 / 128; ++i) {   // (N, ldw and the columns are multiples of 4)
        const int k = (t >> 4) + i * 8, c = (t & 15) * 4;
        const bool in = k0 + k < K && col0 + c < N;
        const float* src = in ? W + (size_t)(k0 + k) * ldw + col0 + c : W;
        asm volatile("cp.async.cg.shared.global [%0], [%1], 16, %2;" ::"r"((unsigned)__cvta_generic_to_shared(&sB[s][k][c])), "l"(src), "r"(in ? 16 : 0) : "memory");
      }
    }
    asm volatile("cp.async.commit_group;" ::: "memory");
  };
  unsigned long long sum[4][2];   // pairs of neighbouring columns
#pragma unroll
  for (int i = 0; i < 4; ++i) sum[i][0] = sum[i][1] = 0ull;
#pragma unroll
  for (int s = 0; s < SIMT_STAGES - 1; ++s) load(s, s * BK);
  int s = 0;
  for (int k0 = 0; k0 < K; k0 += BK) {
    asm volatile("cp.async.wait_group %0;" ::"n"(SIMT_STAGES - 2) : "memory");
    __syncthreads();   // this panel is there, and the one before it has been used up by all
    load(s == 0 ? SIMT_STAGES - 1 : s - 1, k0 + (SIMT_STAGES - 1) * BK);
#pragma unroll
    for (int k = 0; k < BK; k += 4) {
      float4 a[4];
      ulonglong2 b[4];
#pragma unroll
      for (int i = 0; i < 4; ++i) a[i] = *reinterpret_cast<const float4*>(&sA[s][ty * 4 + i][k]);
#pragma unroll
      for (int j = 0; j < 4; ++j) b[j] = *reinterpret_cast<const ulonglong2*>(&sB[s][k + j][tx * 4]);
#pragma unroll
      for (int j = 0; j < 4; ++j)
#pragma unroll
        for (int i = 0; i < 4; ++i) {
          const float x = j == 0 ? a[i].x : j == 1 ? a[i].y : j == 2 ? a[i].z : a[i].w;
          unsigned long long xx;
          asm("mov.b64 %0, {%1, %1};" : "=l"(xx) : "f"(x));
          asm("fma.rn.f32x2 %0, %1, %2, %0;" : "+l"(sum[i][0]) : "l"(xx), "l"(b[j].x));
          asm("fma.rn.f32x2 %0, %1, %2, %0;" : "+l"(sum[i][1]) : "l"(xx), "l"(b[j].y));
        }
    }
    s = s == SIMT_STAGES - 1 ? 0 : s + 1;
  }
  float acc[4][4];
#pragma unroll
  for (int i = 0; i < 4; ++i)
#pragma unroll
    for (int j = 0; j < 2; ++j) asm("mov.b64 {%0, %1}, %2;" : "=f"(acc[i][2 * j]), "=f"(acc[i][2 * j + 1]) : "l"(sum[i][j]));
#pragma unroll
  for (int i = 0; i < 4; ++i) {
    int r = row0 + ty * 4 + i;
    if (r >= n) continue;
    long long u = src_begin + r;
    float c_out = 1.f, self_mul = 1.f;
    if (mode == TAURUS_GCN_SYM) {
      c_out = (float)(1.0 / sqrt((double)(row_ptr[u + 1] - row_ptr[u]) + 1.0));
    } else if (mode == TAURUS_SAGE_MEAN) {
      int d = din[u];
      int m = (fanout > 0 && d > fanout) ? fanout : d;
      self_mul = (float)(m > 1 ? m : 1);
    }
#pragma unroll
    for (int j = 0; j < 4; ++j) {
      int cidx = col0 + tx * 4 + j;
      if (cidx >= N) continue;
      float x = acc[i][j];
      if (cidx < Hp) x *= c_out;
      else if (mode != TAURUS_GAT) x = (x + bias[cidx - Hp]) * self_mul;   // GAT: the attention scalars as they are
      PT[(size_t)r * ldo + cidx] = x;
    }
  }
}

void launch_project_simt(taurus_ctx* c, int layer, const float* X, int ldx, long long src_begin, int n, float* out, int ldo, cudaStream_t st,
                         const AccountWork* acc) {
  const int Hp = taurus_round_up(c->dims[layer + 1], 4);
  const int N = taurus_proj_width(c->mode, Hp, c->heads);
  const int across = (N + BN - 1) / BN, tiles = (n + BM - 1) / BM * across;
  if (acc)
    launch_early(c->early, project_simt_kernel<true>, tiles + acc->blocks, 128, 0, st, X, ldx, c->dims[layer], (const float*)c->d_Wcat[layer], N, N, out, (long long)ldo, n, Hp,
                 c->mode, (const float*)c->d_bias[layer], (const long long*)c->d_row_ptr, (const int32_t*)c->d_din, c->fanout[layer], src_begin, across,
                 AccountArgs<true>{*acc});
  else
    launch_early(c->early, project_simt_kernel<false>, tiles, 128, 0, st, X, ldx, c->dims[layer], (const float*)c->d_Wcat[layer], N, N, out, (long long)ldo, n, Hp,
                 c->mode, (const float*)c->d_bias[layer], (const long long*)c->d_row_ptr, (const int32_t*)c->d_din, c->fanout[layer], src_begin, across,
                 AccountArgs<false>());
  c->launches += 1;
}

// out[n x N] (pitch ld_out) = X[n x K] (pitch ldx) . W[:, 0..N) (row-major, pitch ldw), no epilogue.
void launch_gemm_plain_simt(taurus_ctx* c, const float* W, int ldw, int N, const float* X, int ldx, int K, int n, float* out,
                            long long ld_out, cudaStream_t st) {
  if (n <= 0) return;
  const int across = (N + BN - 1) / BN;
  project_simt_kernel<false><<<(n + BM - 1) / BM * across, 128, 0, st>>>(X, ldx, K, W, ldw, N, out, ld_out, n, N, TAURUS_GIN_SUM, nullptr, c->d_row_ptr, c->d_din,
                                                                         0, 0, across, AccountArgs<false>());
  c->launches += 1;
}
