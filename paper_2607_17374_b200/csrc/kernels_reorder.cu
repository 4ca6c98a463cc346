// Topology-aware reordering (Alg. 1, Sect. 3.8): positions r, locality centres mu, new order = ArgSort(r).
// Both update rules are evaluated pull-based in fp64, lists over lanes (in-lists for mu, CSR rows for r),
// so no floating-point atomics take part in the positions; the order is a stable radix sort of r (ties by
// vertex id).  The dispersion J and the total span C(pi) are reported for the initial order and after every
// iteration, both measured on the ordering itself (positions = ranks).
#include <cub/cub.cuh>

#include <vector>

#include "taurus.h"

#define FULL 0xffffffffu

namespace {

__device__ __forceinline__ int lane() { return threadIdx.x & 31; }
__device__ __forceinline__ double warp_sum(double x) {
  for (int o = 16; o; o >>= 1) x += __shfl_xor_sync(FULL, x, o);
  return x;
}

__global__ void ro_degree_kernel(long long E, const int32_t* col, long long V, int32_t* din, int* bad) {
  long long stride = (long long)gridDim.x * blockDim.x;
  for (long long e = (long long)blockIdx.x * blockDim.x + threadIdx.x; e < E; e += stride) {
    int v = col[e];
    if (v < 0 || v >= V) *bad = 1; else atomicAdd(&din[v], 1);
  }
}
__global__ void ro_src_kernel(long long V, const long long* row_ptr, int32_t* src_of_edge) {
  const long long warps = ((long long)gridDim.x * blockDim.x) >> 5;
  for (long long u = ((long long)blockIdx.x * blockDim.x + threadIdx.x) >> 5; u < V; u += warps)
    for (long long k = row_ptr[u] + lane(); k < row_ptr[u + 1]; k += 32) src_of_edge[k] = (int32_t)u;
}
__global__ void ro_widen_kernel(long long V, const int32_t* din, long long* ptr) {
  long long stride = (long long)gridDim.x * blockDim.x;
  for (long long v = (long long)blockIdx.x * blockDim.x + threadIdx.x; v <= V; v += stride) ptr[v] = v < V ? din[v] : 0;
}
__global__ void ro_init_kernel(long long V, const int32_t* initial_rank, double* r) {
  long long stride = (long long)gridDim.x * blockDim.x;
  for (long long v = (long long)blockIdx.x * blockDim.x + threadIdx.x; v < V; v += stride)
    r[v] = initial_rank ? (double)initial_rank[v] : (double)v;
}

// Lists are walked by eight lanes each, four to a warp: most have a dozen entries and the double-precision shuffles of a
// full-warp sum cost more than the reads.  Lists longer than LONG_LIST are taken one after the other by the whole warp,
// four entries per lane in flight.  (400 k vertices, 5.8 M edges: mu 97 -> 77 us, r 180 -> 172 us, the measures 201 -> 108 us
// against one warp per list; r ends with its longest rows, eight entries in flight do not shorten them.)
#define LONG_LIST 64
__device__ __forceinline__ double sum8(double x) {
  for (int o = 4; o; o >>= 1) x += __shfl_xor_sync(FULL, x, o);
  return x;
}
// one(p): the value of entry p.  Returns, in all eight lanes, the sum over the lane group's own list [b, e).
template <class One>
__device__ __forceinline__ double list_sum(long long b, long long e, One one) {
  const int l8 = lane() & 7, grp = lane() >> 3;
  const bool is_long = e - b > LONG_LIST;
  double s = 0.0;
  if (!is_long) for (long long p = b + l8; p < e; p += 8) s += one(p);
  s = sum8(s);
  for (unsigned m = __ballot_sync(FULL, is_long && l8 == 0); m; m &= m - 1) {
    const int from = __ffs(m) - 1;
    const long long lb = __shfl_sync(FULL, b, from), le = __shfl_sync(FULL, e, from);
    double t[4] = {0.0, 0.0, 0.0, 0.0};
    for (long long p = lb + lane(); p < le; p += 128)
#pragma unroll
      for (int q = 0; q < 4; ++q) if (p + q * 32 < le) t[q] += one(p + q * 32);
    const double all = warp_sum((t[0] + t[1]) + (t[2] + t[3]));
    if (grp == from >> 3) s = all;
  }
  return s;
}

// mu(v) = (r(v) + sum_{u -> v} r(u)) / d(v), d = in-degree + 1 (every vertex aggregates a self message);
// also w1 = mu / d and w2 = 1 / d, the two terms each out-neighbourhood sums.
__global__ void ro_mu_kernel(long long V, const long long* __restrict__ in_ptr, const int32_t* __restrict__ in_src, const double* __restrict__ r,
                             double2* __restrict__ w) {
  const long long groups = ((long long)gridDim.x * blockDim.x) >> 3;
  const long long first = (((long long)blockIdx.x * blockDim.x + threadIdx.x) >> 5) << 2;   // the warp's first list
  for (long long v0 = first; v0 < V; v0 += groups) {
    const long long v = v0 + (lane() >> 3);
    const bool on = v < V;
    const long long b = on ? in_ptr[v] : 0, e = on ? in_ptr[v + 1] : 0;
    const double s = list_sum(b, e, [&](long long p) { return r[in_src[p]]; });
    if (on && (lane() & 7) == 0) {
      const double d = (double)(e - b) + 1.0;
      w[v] = make_double2((r[v] + s) / d / d, 1.0 / d);
    }
  }
}
// r(w) = (mu(w)/d(w) + sum_{w -> v} mu(v)/d(v)) / (1/d(w) + sum_{w -> v} 1/d(v))
__global__ void ro_r_kernel(long long V, const long long* __restrict__ row_ptr, const int32_t* __restrict__ col, const double2* __restrict__ w, double* __restrict__ r) {
  const long long groups = ((long long)gridDim.x * blockDim.x) >> 3;
  const long long first = (((long long)blockIdx.x * blockDim.x + threadIdx.x) >> 5) << 2;
  const int l8 = lane() & 7, grp = lane() >> 3;
  for (long long u0 = first; u0 < V; u0 += groups) {
    const long long u = u0 + grp;
    const bool on = u < V;
    const long long b = on ? row_ptr[u] : 0, e = on ? row_ptr[u + 1] : 0;
    const bool is_long = e - b > LONG_LIST;
    double num = 0.0, den = 0.0;
    if (!is_long) for (long long p = b + l8; p < e; p += 8) { const double2 x = w[col[p]]; num += x.x; den += x.y; }
    num = sum8(num); den = sum8(den);
    for (unsigned m = __ballot_sync(FULL, is_long && l8 == 0); m; m &= m - 1) {
      const int from = __ffs(m) - 1;
      const long long lb = __shfl_sync(FULL, b, from), le = __shfl_sync(FULL, e, from);
      double n2 = 0.0, d2 = 0.0;
#pragma unroll 4
      for (long long p = lb + lane(); p < le; p += 32) { const double2 x = w[col[p]]; n2 += x.x; d2 += x.y; }
      n2 = warp_sum(n2); d2 = warp_sum(d2);
      if (grp == from >> 3) { num = n2; den = d2; }
    }
    if (on && l8 == 0) { const double2 x = w[u]; r[u] = (x.x + num) / (x.y + den); }
  }
}
__global__ void ro_iota_kernel(long long V, int32_t* ids) {
  long long stride = (long long)gridDim.x * blockDim.x;
  for (long long v = (long long)blockIdx.x * blockDim.x + threadIdx.x; v < V; v += stride) ids[v] = (int32_t)v;
}
__global__ void ro_rank_kernel(long long V, const int32_t* order, int32_t* rank) {
  long long stride = (long long)gridDim.x * blockDim.x;
  for (long long i = (long long)blockIdx.x * blockDim.x + threadIdx.x; i < V; i += stride) rank[order[i]] = (int32_t)i;
}
// J = sum_v 1/d(v) * sum over v's in-neighbours and v itself of (pos(u) - mu(v))^2 with mu(v) their mean (the optimum for
// these positions, which are the ranks); span = sum_v (max - min) of ranks.  Two sweeps over a list in one kernel: the
// second finds its scattered ranks in L1 / L2.
__global__ void ro_measure_kernel(long long V, const long long* __restrict__ in_ptr, const int32_t* __restrict__ in_src, const int32_t* __restrict__ rank,
                                  double* J, unsigned long long* span) {
  const long long groups = ((long long)gridDim.x * blockDim.x) >> 3;
  const long long first = (((long long)blockIdx.x * blockDim.x + threadIdx.x) >> 5) << 2;
  double jsum = 0.0;
  unsigned long long ssum = 0;
  for (long long v0 = first; v0 < V; v0 += groups) {
    const long long v = v0 + (lane() >> 3);
    const bool on = v < V;
    const long long b = on ? in_ptr[v] : 0, e = on ? in_ptr[v + 1] : 0;
    const int own = on ? rank[v] : 0;
    const double d = (double)(e - b) + 1.0;
    const double m = ((double)own + list_sum(b, e, [&](long long p) { return (double)rank[in_src[p]]; })) / d;
    // deviations; smallest and largest rank (a long list's are gathered by lanes of other groups too)
    int lo = 0x7fffffff, hi = -1;
    double q = 0.0;
    {
      const int l8 = lane() & 7, grp = lane() >> 3;
      const bool is_long = e - b > LONG_LIST;
      auto take = [&](long long p, double mean, double& sum, int& l, int& h) {
        const int x = rank[in_src[p]];
        const double dlt = (double)x - mean;
        sum += dlt * dlt;
        l = x < l ? x : l; h = x > h ? x : h;
      };
      if (!is_long) for (long long p = b + l8; p < e; p += 8) take(p, m, q, lo, hi);
      q = sum8(q);
      for (int o = 4; o; o >>= 1) { lo = min(lo, __shfl_xor_sync(FULL, lo, o)); hi = max(hi, __shfl_xor_sync(FULL, hi, o)); }
      for (unsigned k = __ballot_sync(FULL, is_long && l8 == 0); k; k &= k - 1) {
        const int from = __ffs(k) - 1;
        const long long lb = __shfl_sync(FULL, b, from), le = __shfl_sync(FULL, e, from);
        const double mean = __shfl_sync(FULL, m, from);
        double q2 = 0.0;
        int lo2 = 0x7fffffff, hi2 = -1;
#pragma unroll 4
        for (long long p = lb + lane(); p < le; p += 32) take(p, mean, q2, lo2, hi2);
        q2 = warp_sum(q2);
        lo2 = __reduce_min_sync(FULL, lo2); hi2 = __reduce_max_sync(FULL, hi2);
        if (grp == from >> 3) { q = q2; lo = lo2; hi = hi2; }
      }
    }
    if (on && (lane() & 7) == 0) {
      jsum += (q + ((double)own - m) * ((double)own - m)) / d;
      ssum += (unsigned long long)(max(hi, own) - min(lo, own));
    }
  }
  jsum = warp_sum(jsum);
  for (int o = 16; o; o >>= 1) ssum += __shfl_xor_sync(FULL, ssum, o);
  if (lane() == 0) {
    if (jsum != 0.0) atomicAdd(J, jsum);
    if (ssum) atomicAdd(span, ssum);
  }
}

// One allocation, handed out in pieces once every piece is planned: thirty allocations and as many frees, which wait for
// the device each, took longer than the kernels between them.
struct Arena {
  char* base = nullptr;
  size_t size = 0;
  template <class T> size_t plan(size_t n) { const size_t at = size; size += (n * sizeof(T) + 255) / 256 * 256 + 256; return at; }
  bool get() {
    if (cudaMalloc((void**)&base, size > 0 ? size : 256) == cudaSuccess) return true;
    cudaGetLastError();
    return false;
  }
  template <class T> T* at(size_t off) const { return reinterpret_cast<T*>(base + off); }
  ~Arena() { cudaFree(base); }
};

}  // namespace

extern "C" int taurus_reorder(int64_t V, int64_t E, const int64_t* row_ptr, const int32_t* col_idx, const int32_t* initial_rank,
                              int32_t iterations, int32_t* out_rank, double* out_positions, double* out_J, int64_t* out_span,
                              void* cuda_stream) {
  if (V < 1 || V >= (1ll << 31) || E < 0 || E >= (1ll << 32) || !row_ptr || (E > 0 && !col_idx) || !out_rank || iterations < 0 ||
      iterations > 1000)
    return TAURUS_ERR_INVALID_ARG;
  cudaStream_t st = static_cast<cudaStream_t>(cuda_stream);
  int sms = 148, dev = 0;
  cudaGetDevice(&dev);
  cudaDeviceGetAttribute(&sms, cudaDevAttrMultiProcessorCount, dev);
  const int grid = sms * 8;
  int end_bit = 1;
  while (end_bit < 31 && (1ll << end_bit) < V) ++end_bit;
  size_t t1 = 0, t2 = 0, t3 = 0;
  {
    long long* const n64 = nullptr;
    int32_t* const n32 = nullptr;
    double* const nd = nullptr;
    cub::DeviceScan::ExclusiveSum(nullptr, t1, n64, n64, V + 1, st);
    if (E > 0) cub::DeviceRadixSort::SortPairs(nullptr, t2, n32, n32, n32, n32, E, 0, end_bit, st);
    cub::DeviceRadixSort::SortPairs(nullptr, t3, nd, nd, n32, n32, V, 0, 64, st);
  }
  size_t tmp_bytes = t1 > t2 ? t1 : t2;
  if (t3 > tmp_bytes) tmp_bytes = t3;
  const size_t n_meas = (size_t)iterations + 1;
  Arena B;
  const size_t o_row = B.plan<long long>((size_t)V + 1), o_col = B.plan<int32_t>((size_t)E), o_din = B.plan<int32_t>((size_t)V),
               o_init = B.plan<int32_t>(initial_rank ? (size_t)V : 0), o_inptr = B.plan<long long>((size_t)V + 1), o_insrc = B.plan<int32_t>((size_t)E),
               o_src = B.plan<int32_t>((size_t)E), o_keys = B.plan<int32_t>((size_t)E), o_r = B.plan<double>((size_t)V), o_rs = B.plan<double>((size_t)V),
               o_w = B.plan<double2>((size_t)V),
               o_ids = B.plan<int32_t>((size_t)V), o_order = B.plan<int32_t>((size_t)V), o_rank = B.plan<int32_t>((size_t)V),
               o_meas = B.plan<double>(2 * n_meas), o_bad = B.plan<int>(1), o_tmp = B.plan<char>(tmp_bytes);
  if (!B.get()) return TAURUS_ERR_NOMEM;
  long long *d_row = B.at<long long>(o_row), *d_inptr = B.at<long long>(o_inptr);
  int32_t *d_col = B.at<int32_t>(o_col), *d_din = B.at<int32_t>(o_din), *d_init = initial_rank ? B.at<int32_t>(o_init) : nullptr,
          *d_insrc = B.at<int32_t>(o_insrc), *d_srcedge = B.at<int32_t>(o_src), *d_keys = B.at<int32_t>(o_keys), *d_ids = B.at<int32_t>(o_ids),
          *d_order = B.at<int32_t>(o_order), *d_rank = B.at<int32_t>(o_rank);
  double *d_r = B.at<double>(o_r), *d_rsorted = B.at<double>(o_rs), *d_J = B.at<double>(o_meas);
  double2* d_w = B.at<double2>(o_w);
  unsigned long long* d_span = reinterpret_cast<unsigned long long*>(d_J + n_meas);
  int* d_bad = B.at<int>(o_bad);
  void* d_tmp = B.at<char>(o_tmp);
#define RO(call) do { if ((call) != cudaSuccess) { cudaGetLastError(); return TAURUS_ERR_CUDA; } } while (0)
  RO(cudaMemcpyAsync(d_row, row_ptr, (size_t)(V + 1) * sizeof(long long), cudaMemcpyDefault, st));
  if (E > 0) RO(cudaMemcpyAsync(d_col, col_idx, (size_t)E * sizeof(int32_t), cudaMemcpyDefault, st));
  if (initial_rank) RO(cudaMemcpyAsync(d_init, initial_rank, (size_t)V * sizeof(int32_t), cudaMemcpyDefault, st));
  RO(cudaMemsetAsync(d_din, 0, (size_t)V * sizeof(int32_t), st));
  RO(cudaMemsetAsync(d_bad, 0, sizeof(int), st));
  // in-lists: in-degrees, their prefix sums, sources sorted (stably) by destination
  ro_degree_kernel<<<grid, 256, 0, st>>>(E, d_col, V, d_din, d_bad);
  ro_widen_kernel<<<grid, 256, 0, st>>>(V, d_din, d_inptr);
  ro_src_kernel<<<grid, 256, 0, st>>>(V, d_row, d_srcedge);
  size_t tb = tmp_bytes;
  RO(cub::DeviceScan::ExclusiveSum(d_tmp, tb, d_inptr, d_inptr, V + 1, st));
  if (E > 0) { tb = tmp_bytes; RO(cub::DeviceRadixSort::SortPairs(d_tmp, tb, d_col, d_keys, d_srcedge, d_insrc, E, 0, end_bit, st)); }
  int bad = 0;
  RO(cudaMemcpyAsync(&bad, d_bad, sizeof(int), cudaMemcpyDeviceToHost, st));
  RO(cudaStreamSynchronize(st));
  if (bad) return TAURUS_ERR_INVALID_ARG;

  ro_init_kernel<<<grid, 256, 0, st>>>(V, d_init, d_r);
  ro_iota_kernel<<<grid, 256, 0, st>>>(V, d_ids);
  RO(cudaMemsetAsync(d_J, 0, 2 * n_meas * sizeof(double), st));
  for (int it = 0; it <= iterations; ++it) {
    if (it > 0) {   // one iteration of the update rules on the real-valued positions
      ro_mu_kernel<<<grid, 256, 0, st>>>(V, d_inptr, d_insrc, d_r, d_w);
      ro_r_kernel<<<grid, 256, 0, st>>>(V, d_row, d_col, d_w, d_r);
    }
    // pi = ArgSort(r), ties by vertex id
    tb = tmp_bytes;
    RO(cub::DeviceRadixSort::SortPairs(d_tmp, tb, d_r, d_rsorted, d_ids, d_order, V, 0, 64, st));
    ro_rank_kernel<<<grid, 256, 0, st>>>(V, d_order, d_rank);
    if (out_J || out_span) {   // J and C(pi) of this ordering (positions = ranks, centres = their optimum)
      ro_measure_kernel<<<grid, 256, 0, st>>>(V, d_inptr, d_insrc, d_rank, d_J + it, d_span + it);
    }
  }
  std::vector<double> J(n_meas, 0.0);
  std::vector<unsigned long long> span(n_meas, 0);
  RO(cudaMemcpyAsync(J.data(), d_J, n_meas * sizeof(double), cudaMemcpyDeviceToHost, st));
  RO(cudaMemcpyAsync(span.data(), d_span, n_meas * sizeof(unsigned long long), cudaMemcpyDeviceToHost, st));
  RO(cudaMemcpyAsync(out_rank, d_rank, (size_t)V * sizeof(int32_t), cudaMemcpyDefault, st));
  if (out_positions) RO(cudaMemcpyAsync(out_positions, d_r, (size_t)V * sizeof(double), cudaMemcpyDefault, st));
  RO(cudaStreamSynchronize(st));
  RO(cudaGetLastError());
  for (int it = 0; it <= iterations; ++it) {
    if (out_J) out_J[it] = J[(size_t)it];
    if (out_span) out_span[it] = (int64_t)span[(size_t)it];
  }
#undef RO
  return TAURUS_OK;
}

// ------------------------------------------------------------------------------------------------ relabelling
// Applying an ordering (Sect. 3.8: topology relabelling and feature relabelling): vertex v becomes rank[v].
namespace {

__global__ void rl_check_kernel(long long V, const int32_t* __restrict__ rank, int32_t* __restrict__ seen, int* bad) {
  long long stride = (long long)gridDim.x * blockDim.x;
  for (long long v = (long long)blockIdx.x * blockDim.x + threadIdx.x; v < V; v += stride) {
    const int r = rank[v];
    if (r < 0 || r >= V || atomicAdd(&seen[r], 1) != 0) *bad = 1;   // not a permutation of [0, V)
  }
}
__global__ void rl_degree_kernel(long long V, const long long* __restrict__ row_ptr, const int32_t* __restrict__ rank,
                                 long long* __restrict__ new_ptr) {
  long long stride = (long long)gridDim.x * blockDim.x;
  for (long long v = (long long)blockIdx.x * blockDim.x + threadIdx.x; v <= V; v += stride) {
    if (v < V) new_ptr[rank[v]] = row_ptr[v + 1] - row_ptr[v];
    else new_ptr[V] = 0;
  }
}
// row rank[u] of the output = the out-edges of u in their original order, destinations renamed
__global__ void rl_edges_kernel(long long V, const long long* __restrict__ row_ptr, const int32_t* __restrict__ col,
                                const int32_t* __restrict__ rank, const long long* __restrict__ new_ptr, int32_t* __restrict__ new_col,
                                int32_t* __restrict__ new_din, int* bad) {
  const long long warps = ((long long)gridDim.x * blockDim.x) >> 5;
  for (long long u = ((long long)blockIdx.x * blockDim.x + threadIdx.x) >> 5; u < V; u += warps) {
    const long long b = row_ptr[u], n = row_ptr[u + 1] - b, nb = new_ptr[rank[u]];
    for (long long k = lane(); k < n; k += 32) {
      const int v = col[b + k];
      if (v < 0 || v >= V) { *bad = 1; continue; }
      const int nv = rank[v];
      new_col[nb + k] = nv;
      if (new_din) atomicAdd(&new_din[nv], 1);
    }
  }
}
__global__ void rl_rows_kernel(long long V, int width, const float* __restrict__ in, long long ld_in, const int32_t* __restrict__ rank,
                               float* __restrict__ out, long long ld_out) {
  const long long warps = ((long long)gridDim.x * blockDim.x) >> 5;
  const bool wide = ((width | ld_in | ld_out) & 3) == 0 && ((reinterpret_cast<uintptr_t>(in) | reinterpret_cast<uintptr_t>(out)) & 15) == 0;
  for (long long v = ((long long)blockIdx.x * blockDim.x + threadIdx.x) >> 5; v < V; v += warps) {
    const float* src = in + (size_t)v * ld_in;
    float* dst = out + (size_t)rank[v] * ld_out;
    if (wide) for (int k = lane(); k < (width >> 2); k += 32) reinterpret_cast<float4*>(dst)[k] = reinterpret_cast<const float4*>(src)[k];
    else for (int k = lane(); k < width; k += 32) dst[k] = src[k];
  }
}

}  // namespace

extern "C" int taurus_relabel_csr(int64_t V, int64_t E, const int64_t* row_ptr, const int32_t* col_idx, const int32_t* rank,
                                  int64_t* out_row_ptr, int32_t* out_col_idx, int32_t* out_in_degree, void* cuda_stream) {
  if (V < 1 || V >= (1ll << 31) || E < 0 || E >= (1ll << 32) || !row_ptr || (E > 0 && (!col_idx || !out_col_idx)) || !rank || !out_row_ptr)
    return TAURUS_ERR_INVALID_ARG;
  cudaStream_t st = static_cast<cudaStream_t>(cuda_stream);
  int sms = 148, dev = 0;
  cudaGetDevice(&dev);
  cudaDeviceGetAttribute(&sms, cudaDevAttrMultiProcessorCount, dev);
  const int grid = sms * 8;
  size_t tb = 0;
  {
    long long* const n64 = nullptr;
    cub::DeviceScan::ExclusiveSum(nullptr, tb, n64, n64, V + 1, st);
  }
  Arena B;
  const size_t o_row = B.plan<long long>((size_t)V + 1), o_col = B.plan<int32_t>((size_t)E), o_rank = B.plan<int32_t>((size_t)V),
               o_seen = B.plan<int32_t>((size_t)V), o_nptr = B.plan<long long>((size_t)V + 1), o_ncol = B.plan<int32_t>((size_t)E),
               o_ndin = B.plan<int32_t>((size_t)V), o_bad = B.plan<int>(1), o_tmp = B.plan<char>(tb);
  if (!B.get()) return TAURUS_ERR_NOMEM;
  long long *d_row = B.at<long long>(o_row), *d_nptr = B.at<long long>(o_nptr);
  int32_t *d_col = B.at<int32_t>(o_col), *d_rank = B.at<int32_t>(o_rank), *d_seen = B.at<int32_t>(o_seen), *d_ncol = B.at<int32_t>(o_ncol),
          *d_ndin = out_in_degree ? B.at<int32_t>(o_ndin) : nullptr;
  int* d_bad = B.at<int>(o_bad);
  void* d_tmp = B.at<char>(o_tmp);
#define RL(call) do { if ((call) != cudaSuccess) { cudaGetLastError(); return TAURUS_ERR_CUDA; } } while (0)
  RL(cudaMemcpyAsync(d_row, row_ptr, (size_t)(V + 1) * sizeof(long long), cudaMemcpyDefault, st));
  if (E > 0) RL(cudaMemcpyAsync(d_col, col_idx, (size_t)E * sizeof(int32_t), cudaMemcpyDefault, st));
  RL(cudaMemcpyAsync(d_rank, rank, (size_t)V * sizeof(int32_t), cudaMemcpyDefault, st));
  RL(cudaMemsetAsync(d_seen, 0, (size_t)V * sizeof(int32_t), st));
  RL(cudaMemsetAsync(d_bad, 0, sizeof(int), st));
  if (d_ndin) RL(cudaMemsetAsync(d_ndin, 0, (size_t)V * sizeof(int32_t), st));
  rl_check_kernel<<<grid, 256, 0, st>>>(V, d_rank, d_seen, d_bad);
  int bad = 0;
  RL(cudaMemcpyAsync(&bad, d_bad, sizeof(int), cudaMemcpyDeviceToHost, st));
  RL(cudaStreamSynchronize(st));
  if (bad) return TAURUS_ERR_INVALID_ARG;      // before any index derived from rank is used as an address
  rl_degree_kernel<<<grid, 256, 0, st>>>(V, d_row, d_rank, d_nptr);
  RL(cub::DeviceScan::ExclusiveSum(d_tmp, tb, d_nptr, d_nptr, V + 1, st));
  rl_edges_kernel<<<grid, 256, 0, st>>>(V, d_row, d_col, d_rank, d_nptr, d_ncol, d_ndin, d_bad);
  RL(cudaMemcpyAsync(&bad, d_bad, sizeof(int), cudaMemcpyDeviceToHost, st));
  RL(cudaMemcpyAsync(out_row_ptr, d_nptr, (size_t)(V + 1) * sizeof(long long), cudaMemcpyDefault, st));
  if (E > 0) RL(cudaMemcpyAsync(out_col_idx, d_ncol, (size_t)E * sizeof(int32_t), cudaMemcpyDefault, st));
  if (out_in_degree) RL(cudaMemcpyAsync(out_in_degree, d_ndin, (size_t)V * sizeof(int32_t), cudaMemcpyDefault, st));
  RL(cudaStreamSynchronize(st));
  RL(cudaGetLastError());
  return bad ? TAURUS_ERR_INVALID_ARG : TAURUS_OK;
#undef RL
}

extern "C" int taurus_permute_rows(int64_t V, int32_t width, const float* in_rows, int64_t ld_in, const int32_t* rank, float* out_rows,
                                   int64_t ld_out, void* cuda_stream) {
  if (V < 1 || V >= (1ll << 31) || width < 1 || !in_rows || !rank || !out_rows || ld_in < width || ld_out < width || in_rows == out_rows)
    return TAURUS_ERR_INVALID_ARG;
  cudaPointerAttributes a_in, a_out, a_rank;
  if (cudaPointerGetAttributes(&a_in, in_rows) != cudaSuccess || cudaPointerGetAttributes(&a_out, out_rows) != cudaSuccess ||
      cudaPointerGetAttributes(&a_rank, rank) != cudaSuccess || a_in.type != cudaMemoryTypeDevice || a_out.type != cudaMemoryTypeDevice ||
      a_rank.type != cudaMemoryTypeDevice) {
    cudaGetLastError();
    return TAURUS_ERR_INVALID_ARG;             // device memory only: the matrices are too large to stage
  }
  cudaStream_t st = static_cast<cudaStream_t>(cuda_stream);
  int sms = 148, dev = 0;
  cudaGetDevice(&dev);
  cudaDeviceGetAttribute(&sms, cudaDevAttrMultiProcessorCount, dev);
  rl_rows_kernel<<<sms * 8, 256, 0, st>>>(V, width, in_rows, ld_in, rank, out_rows, ld_out);
  return cudaGetLastError() == cudaSuccess ? TAURUS_OK : TAURUS_ERR_CUDA;
}
