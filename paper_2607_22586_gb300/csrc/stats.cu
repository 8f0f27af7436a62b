// Proxy statistics over the whole prefill (Section 3.2.1: mean and standard
// deviation of the prompt's features across all prompt tokens; read in query
// space, per (query head, dimension) over the T prompt queries of a request,
// with the unbiased T - 1 estimator).
//
// A streaming reduction over Q [L][total_T][Hq][d]: every byte of Q is read
// once, in coalesced 16-byte vectors, so the pass is bounded by HBM.
//  - stats_partial_kernel: a chunk of kStatsChunk prompt queries of one request
//    and layer, one thread per 16 bytes of columns (q-head, dimension), 64
//    threads per CTA so that a few hundred chunks fill the SMs evenly; a thread
//    keeps, per column, the sums of (x - x0) and (x - x0)^2 in fp32, x0 being
//    the chunk's first query (the shift keeps the second sum free of
//    cancellation). Rows arrive 32 ahead through asynchronous copies into the
//    thread's own places of shared memory; with eight rows loaded to registers
//    and one CTA of 448 threads per chunk the compiler and the uneven waves left
//    fewer in flight: 940 MB of hidden states 179 -> 163 us (both kernels), 6.6
//    GB of prompt queries 1,065 -> 952 us, 6.9 TB/s. 128 threads: 180 us.
//    Float32 threads take four columns: with eight, as two copies of 16 bytes, a
//    warp's accesses leave every other 16 bytes out and each sector is fetched
//    twice (1.07 GB of hidden states 228 us before the copies, 347 with eight
//    columns, 178 with four).
//  - stats_merge_kernel: one thread per column merges the chunks in order with
//    the pairwise update of Chan, Golub and LeVeque (count, mean, sum of
//    squared deviations), then writes mean and std.
#include <algorithm>

#include "common.cuh"

namespace mmshift {
namespace {

constexpr int kStatsGroup = 4;     // rows per asynchronous copy group
constexpr int kStatsRing = 8;      // groups in flight per thread
constexpr int kStatsThreads = 64;  // column groups (of 16 bytes a row) per CTA
constexpr int kMergeAhead = 8;     // chunks of partial sums loaded ahead in the merge

// The 16 / sizeof(T) elements of a 16-byte word as float32.
__device__ __forceinline__ void unpack(const uint4& v, float (&x)[8]) {
  const uint32_t w[4] = {v.x, v.y, v.z, v.w};
#pragma unroll
  for (int i = 0; i < 4; ++i) {
    x[2 * i] = __uint_as_float(w[i] << 16);
    x[2 * i + 1] = __uint_as_float(w[i] & 0xffff0000u);
  }
}
__device__ __forceinline__ void unpack(const uint4& v, float (&x)[4]) {
  x[0] = __uint_as_float(v.x);
  x[1] = __uint_as_float(v.y);
  x[2] = __uint_as_float(v.z);
  x[3] = __uint_as_float(v.w);
}

__device__ __forceinline__ void copy16(void* smem, const void* gmem) {
  asm volatile("cp.async.cg.shared.global [%0], [%1], 16;" ::"r"(
                   (uint32_t)__cvta_generic_to_shared(smem)),
               "l"(gmem)
               : "memory");
}

// part: [L][B][nchunk][3][ncol] (x0, sum of x - x0, sum of (x - x0)^2)
// ncp CTAs share a chunk, each taking every ncp-th run of blockDim.x column
// groups.
template <typename T>
__global__ void __launch_bounds__(kStatsThreads) stats_partial_kernel(const __grid_constant__ StatsJob J,
                                                                     const T* Q, float* part, int ncp) {
  constexpr int C = 16 / (int)sizeof(T), G = kStatsGroup, NG = kStatsRing;   // C: columns per thread
  extern __shared__ uint4 ring[];    // [NG][G][blockDim.x]
  const int c = blockIdx.x / ncp, cp = blockIdx.x % ncp, b = blockIdx.y, l = blockIdx.z;
  const int t_len = J.t_len[b];
  const int t0 = c * kStatsChunk;
  if (t0 >= t_len) return;
  const int n = min(t_len, t0 + kStatsChunk) - t0;
  const T* q = Q + (size_t)l * J.ls + ((size_t)J.tok_off[b] + t0) * J.ncol;
  float* out = part + (((size_t)l * J.B + b) * J.nchunk + c) * 3 * J.ncol;
  const int nt = blockDim.x;
  for (int cg = cp * nt + threadIdx.x; cg < J.ncol / C; cg += ncp * nt) {
    const T* col = q + (size_t)cg * C;
    // rows 1 .. n - 1 in groups of G, NG groups on their way to this thread's
    // own places of the ring (no other thread reads them, so no barrier)
    auto slot = [&](int g, int u) { return ring + (size_t)(g * G + u) * nt + threadIdx.x; };
    auto fetch = [&](int g) {
#pragma unroll
      for (int u = 0; u < G; ++u) {
        const int t = 1 + g * G + u;
        if (t < n) copy16(slot(g % NG, u), col + (size_t)t * J.ncol);
      }
      asm volatile("cp.async.commit_group;" ::: "memory");
    };
#pragma unroll 1
    for (int g = 0; g < NG; ++g) fetch(g);
    float x0[C], s1[C], s2[C];
    unpack(__ldg(reinterpret_cast<const uint4*>(col)), x0);
#pragma unroll
    for (int k = 0; k < C; ++k) { s1[k] = 0.f; s2[k] = 0.f; }
    auto add = [&](int g, int u) {
      float x[C];
      unpack(*slot(g, u), x);
#pragma unroll
      for (int k = 0; k < C; ++k) {
        const float dv = x[k] - x0[k];
        s1[k] += dv;
        s2[k] = fmaf(dv, dv, s2[k]);
      }
    };
    const int ng = (n - 1 + G - 1) / G;
#pragma unroll 1
    for (int g = 0; g < ng; ++g) {
      asm volatile("cp.async.wait_group %0;" ::"n"(NG - 1) : "memory");
      const int rows = n - 1 - g * G;
#pragma unroll
      for (int u = 0; u < G; ++u)
        if (u < rows) add(g % NG, u);
      fetch(g + NG);                 // into the group just read
    }
    asm volatile("cp.async.wait_group 0;" ::: "memory");
#pragma unroll
    for (int k = 0; k < C; ++k) {
      out[cg * C + k] = x0[k];
      out[J.ncol + cg * C + k] = s1[k];
      out[2 * J.ncol + cg * C + k] = s2[k];
    }
  }
}

// stats: [L][B][2][ncol] (mean, std)
__global__ void __launch_bounds__(256) stats_merge_kernel(StatsJob J, const float* part,
                                                          float* stats) {
  const int col = blockIdx.x * blockDim.x + threadIdx.x;
  const int b = blockIdx.y, l = blockIdx.z;
  if (col >= J.ncol) return;
  const int t_len = J.t_len[b];
  const float* in = part + ((size_t)l * J.B + b) * J.nchunk * 3 * J.ncol + col;
  float n = 0.f, mean = 0.f, m2 = 0.f;
  const int nch = (t_len + kStatsChunk - 1) / kStatsChunk;
  for (int c0 = 0; c0 < nch; c0 += kMergeAhead) {
    // the loads of kMergeAhead chunks first, then the merges in chunk order
    float v[kMergeAhead][3];
#pragma unroll
    for (int u = 0; u < kMergeAhead; ++u)
      if (c0 + u < nch)
#pragma unroll
        for (int q = 0; q < 3; ++q) v[u][q] = in[((size_t)(c0 + u) * 3 + q) * J.ncol];
#pragma unroll
    for (int u = 0; u < kMergeAhead; ++u) {
      const int c = c0 + u;
      if (c >= nch) break;
      const float nb = (float)(min(t_len, (c + 1) * kStatsChunk) - c * kStatsChunk);
      const float x0 = v[u][0], s1 = v[u][1], s2 = v[u][2];
      const float mb = x0 + s1 / nb;
      const float m2b = fmaxf(s2 - s1 * (s1 / nb), 0.f);
      const float nab = n + nb;
      const float delta = mb - mean;
      mean += delta * (nb / nab);
      m2 += m2b + delta * delta * (n * nb / nab);
      n = nab;
    }
  }
  float* out = stats + ((size_t)l * J.B + b) * 2 * J.ncol;
  out[col] = mean;
  out[J.ncol + col] = t_len > 1 ? sqrtf(m2 / (float)(t_len - 1)) : 0.f;
}

}  // namespace

cudaError_t launch_prefill_stats(const StatsJob& J, const void* Q, float* part, float* stats,
                                 cudaStream_t st, bool bf16) {
  const int groups = J.ncol / (bf16 ? 8 : 4);
  const int threads = std::min(kStatsThreads, (groups + 31) / 32 * 32);
  const int ncp = (groups + threads - 1) / threads;
  dim3 g1(J.nchunk * ncp, J.B, J.L);
  const size_t smem = (size_t)kStatsRing * kStatsGroup * threads * 16;
  cudaError_t e;
#define MMSHIFT_STATS(T)                                                                          \
  {                                                                                              \
    if ((e = cudaFuncSetAttribute(stats_partial_kernel<T>,                                       \
                                  cudaFuncAttributeMaxDynamicSharedMemorySize, (int)smem)) !=     \
        cudaSuccess)                                                                             \
      return e;                                                                                  \
    stats_partial_kernel<T><<<g1, threads, smem, st>>>(J, (const T*)Q, part, ncp);               \
  }
  if (bf16) MMSHIFT_STATS(__nv_bfloat16) else MMSHIFT_STATS(float)
#undef MMSHIFT_STATS
  e = cudaGetLastError();
  if (e != cudaSuccess) return e;
  dim3 g2((J.ncol + 255) / 256, J.B, J.L);
  stats_merge_kernel<<<g2, 256, 0, st>>>(J, part, stats);
  return cudaGetLastError();
}

}  // namespace mmshift
