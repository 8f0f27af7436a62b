// Quality metric: attention-mass coverage of a kept set (Section 1, Fig. 1b:
// the share of decode-time attention probability that falls on the prompt
// entries kept after prefill).
//
// A decode query's coverage under one query head is the ratio of two sums of
// exponentials, over the kept keys and over all T_b keys. Both come from the
// softmax pass, which only ever needs sums: once over the prompt and once over
// the kept rows, which kept_rows_kernel copies together first; ratio_kernel
// merges the two sets of (max, sum) partials and averages over the r query
// heads. No mass of a single key is formed, so a key costs one tensor-core pass
// instead of two, and the decode queries of all r heads fill the stationary
// rows without padding each query's r rows to 16. 32 decode queries on the
// 28-layer 32K stack with 2,048 kept rows: kernels of a call 1,564 -> 278 us.
//
// Where the copied rows would not fit in the workspace of the group-mass form (few
// decode queries or large budgets) the decode queries run through steps 2-4 as
// n_dec groups of one proxy each, so the group masses hold, per (layer, KV
// head, decode query, key), the attention probability summed over the r query
// heads; coverage_kernel divides the masses of the kept keys by the masses of
// all T_b keys (r up to rounding).
#include "common.cuh"

namespace mmshift {
namespace {

constexpr int kCovThreads = 256;

__device__ __forceinline__ float block_sum(float v, float* red) {
#pragma unroll
  for (int o = 16; o > 0; o >>= 1) v += __shfl_xor_sync(0xffffffffu, v, o);
  const int warp = threadIdx.x / 32, lane = threadIdx.x % 32;
  if (lane == 0) red[warp] = v;
  __syncthreads();
  float s = 0.f;
  if (warp == 0) {
    s = lane < kCovThreads / 32 ? red[lane] : 0.f;
#pragma unroll
    for (int o = 16; o > 0; o >>= 1) s += __shfl_xor_sync(0xffffffffu, s, o);
  }
  __syncthreads();
  return s;   // valid in thread 0
}

// One CTA per (decode query g, KV head h, layer x request); fixed-order sums.
__global__ void __launch_bounds__(kCovThreads) coverage_kernel(Problem P, const float* gmass,
                                                               const int32_t* idx, float* cov,
                                                               int* status) {
  __shared__ float red[kCovThreads / 32];
  const int g = blockIdx.x, h = blockIdx.y;
  const int l = blockIdx.z / P.B, b = blockIdx.z % P.B;
  const ReqInfo R = P.req[b];
  const float* row = gmass + (((size_t)l * P.Hkv + h) * P.G + g) * P.total_T + R.tok_off;
  const int32_t* id = idx + ((size_t)l * P.R + R.out_off) * P.Hkv + h;
  float kept = 0.f, tot = 0.f;
  bool bad = false;
  for (int c = threadIdx.x; c < R.keep; c += kCovThreads) {
    const int t = id[(size_t)c * P.Hkv];
    if ((unsigned)t < (unsigned)R.t_len) kept += row[t];
    else if (t != -1) bad = true;   // -1: padding row of a head with a smaller budget
  }
  for (int t = threadIdx.x; t < R.t_len; t += kCovThreads) tot += row[t];
  if (bad) set_status(status, kStatusBadIndex);
  kept = block_sum(kept, red);
  tot = block_sum(tot, red);
  if (threadIdx.x == 0)
    cov[(((size_t)l * P.B + b) * P.Hkv + h) * P.G + g] = tot > 0.f ? kept / tot : 0.f;
}

// CTA = 256 consecutive kept-set entries (a chunk) of one (layer, request, KV
// head). The valid entries before them, which say where its rows go, come from
// the chunks' counts (kept_count_kernel) or, up to kCountAgain entries, are counted
// again by every CTA, which spares a launch of 2 to 4 us but grows with the square
// of the budget. One layer of 128K keys, 28 / 4 heads, counts against counting
// again: 8,192 kept rows 98 and 94 us a call, 16,384 104 and 102, 65,536 133 and 148.
constexpr int KRT = 256;
constexpr int kCountAgain = 16384;

// Chunk counts [L][Hkv][R / KRT + B], request b's from R.out_off / KRT + b on.
__device__ __forceinline__ size_t chunk_at(const Problem& P, int l, int h, int b) {
  return ((size_t)l * P.Hkv + h) * (P.R / KRT + P.B) + P.req[b].out_off / KRT + b;
}

__global__ void __launch_bounds__(KRT) kept_count_kernel(const __grid_constant__ Problem P,
                                                         const int32_t* idx, int32_t* counts) {
  const int h = blockIdx.y, l = blockIdx.z / P.B, b = blockIdx.z % P.B;
  const ReqInfo R = P.req[b];
  const int c = blockIdx.x * KRT + threadIdx.x;
  if (blockIdx.x * KRT >= R.keep) return;
  const int t = c < R.keep ? idx[((size_t)l * P.R + R.out_off + c) * P.Hkv + h] : -1;
  const int n = __syncthreads_count((unsigned)t < (unsigned)R.t_len);
  if (threadIdx.x == 0) counts[chunk_at(P, l, h, b) + blockIdx.x] = n;
}

template <int ROWB>
__global__ void __launch_bounds__(KRT) kept_rows_kernel(const __grid_constant__ Problem P,
                                                        const uint8_t* K, const int32_t* idx,
                                                        const int32_t* counts, uint8_t* kept,
                                                        int32_t* kept_len, int* status, bool vec) {
  constexpr int LPR = ROWB / 16;   // lanes per row
  const int h = blockIdx.y, l = blockIdx.z / P.B, b = blockIdx.z % P.B;
  const ReqInfo R = P.req[b];
  const int start = blockIdx.x * KRT, tid = threadIdx.x, lane = tid % 32, w = tid / 32;
  if (start >= R.keep) return;
  const int32_t* id = idx + ((size_t)l * P.R + R.out_off) * P.Hkv + h;
  __shared__ int wsum[KRT / 32], wcnt[KRT / 32], list[KRT];
  int before = 0;
  if (counts) {
    const int32_t* cnt = counts + chunk_at(P, l, h, b);
    for (int c = tid; c < (int)blockIdx.x; c += KRT) before += cnt[c];
  } else {
    for (int c = tid; c < start; c += KRT) before += (unsigned)id[(size_t)c * P.Hkv] < (unsigned)R.t_len;
  }
  before = __reduce_add_sync(0xffffffffu, before);
  const int c = start + tid;
  const int t = c < R.keep ? id[(size_t)c * P.Hkv] : -1;
  const bool valid = (unsigned)t < (unsigned)R.t_len;
  if (!valid && t != -1) set_status(status, kStatusBadIndex);
  const unsigned bal = __ballot_sync(0xffffffffu, valid);
  if (lane == 0) { wsum[w] = before; wcnt[w] = __popc(bal); }
  __syncthreads();
  int first = 0, pos = 0, n = 0;
  for (int i = 0; i < KRT / 32; ++i) {
    first += wsum[i];
    if (i < w) pos += wcnt[i];
    n += wcnt[i];
  }
  if (valid) list[pos + __popc(bal & ((1u << lane) - 1u))] = t;
  if (tid == 0 && start + KRT >= R.keep)
    kept_len[((size_t)l * P.B + b) * P.Hkv + h] = first + n;
  __syncthreads();
  const size_t esz = ROWB / P.d, rstride = (size_t)P.Hkv * ROWB;
  const uint8_t* src = K + (size_t)l * P.ls_kv * esz + (size_t)R.tok_off * rstride + (size_t)h * ROWB;
  uint8_t* dst = kept + ((size_t)l * P.R + R.out_off + first) * rstride + (size_t)h * ROWB;
  const int part = tid % LPR;
#pragma unroll 4
  for (int e = tid / LPR; e < n; e += KRT / LPR) {
    const uint8_t* p = src + (size_t)list[e] * rstride + part * 16;
    *reinterpret_cast<uint4*>(dst + (size_t)e * rstride + part * 16) = load_row16(p, vec);
  }
}

// (m, z) += the partials src[0], src[step], ..., n of them, in order, eight loads
// issued ahead.
__device__ __forceinline__ void merge_run(const float2* src, size_t step, int n, float& m, float& z) {
  constexpr int A = 8;
  for (int s0 = 0; s0 < n; s0 += A) {
    float2 v[A];
#pragma unroll
    for (int u = 0; u < A; ++u)
      v[u] = s0 + u < n ? src[(size_t)(s0 + u) * step] : make_float2(-INFINITY, 0.f);
#pragma unroll
    for (int u = 0; u < A; ++u) merge_ms(m, z, v[u].x, v[u].y);
  }
}

// Runs of kRun partials of every row merged into the run's first, a thread per
// (row, run), where a row has more than one run: as one thread's chain a prompt's
// partials (one per 256 keys) took longer than its softmax pass. 32 decode queries
// of 28 / 4 heads, one layer, half the prompt kept: 128K keys 383 -> 148 us, 1M keys
// 4,315 -> 1,491 (the group-mass form took 2,813); 28 layers of 32K keys, 2,048
// kept rows, 128 partials a row: 327 -> 278.
constexpr int kRun = 64;

__global__ void __launch_bounds__(128) ratio_runs_kernel(const __grid_constant__ Problem Q, float2* part) {
  const int row = (blockIdx.x % (Q.Prows_pad / 128)) * 128 + threadIdx.x;
  const int s0 = blockIdx.x / (Q.Prows_pad / 128) * kRun, h = blockIdx.y;
  const int l = blockIdx.z / Q.B, b = blockIdx.z % Q.B;
  const int n = min(kRun, Q.req[b].nsplit * Q.part_slots - s0);
  if (n <= 0 || row >= Q.Prows) return;
  float2* src = part + ((((size_t)l * Q.Hkv + h) * Q.total_splits + Q.req[b].split_off) * Q.part_slots + s0) *
                           Q.Prows_pad + row;
  float m = -INFINITY, z = 0.f;
  merge_run(src, Q.Prows_pad, n, m, z);
  *src = make_float2(m, z);
}

// CTA = NQ decode queries of one (layer, request, KV head): thread (i, jj) merges
// the partials of query i under query heads jj, jj + nj, ..., nj = blockDim.x / NQ;
// run, run_k: partials already merged into each place that holds one.
template <int NQ>
__global__ void __launch_bounds__(1024) ratio_kernel(const __grid_constant__ Problem P,
                                                    const __grid_constant__ Problem Pk,
                                                    const float2* all, const float2* kept,
                                                    int run, int run_k, float* cov) {
  __shared__ float red[1024 / NQ][NQ + 1];
  const int li = threadIdx.x % NQ, jj = threadIdx.x / NQ, nj = blockDim.x / NQ;
  const int i = blockIdx.x * NQ + li, h = blockIdx.y;
  const int l = blockIdx.z / P.B, b = blockIdx.z % P.B;
  float share = 0.f;
  if (i < P.Np) {
    auto merged = [&](const Problem& Q, const float2* part, int step, int row, float& m, float& z) {
      const float2* src = part + (((size_t)l * Q.Hkv + h) * Q.total_splits + Q.req[b].split_off) *
                                     Q.part_slots * Q.Prows_pad + row;
      const int ns = Q.req[b].nsplit * Q.part_slots;
      merge_run(src, (size_t)step * Q.Prows_pad, (ns + step - 1) / step, m, z);
    };
    for (int j = jj; j < P.r; j += nj) {
      float m = -INFINITY, z = 0.f, mk = -INFINITY, zk = 0.f;
      merged(P, all, run, j * P.gs + i, m, z);
      merged(Pk, kept, run_k, j * P.gs + i, mk, zk);
      // zk 2^(mk - m) <= z, so neither factor's product overflows; a query head
      // without a positive sum (NaN or +inf logits, or all -inf) leaves its KV
      // head no coverage, kept key or not, as the group-mass form has it
      share += z > 0.f ? zk * exp2f(mk - m) / z : NAN;
    }
  }
  red[jj][li] = share;
  __syncthreads();
  if (jj == 0 && i < P.Np) {
    float s = 0.f;
    for (int k = 0; k < nj; ++k) s += red[k][li];
    cov[(((size_t)l * P.B + b) * P.Hkv + h) * P.Np + i] = s >= 0.f ? s / (float)P.r : 0.f;
  }
}

}  // namespace

cudaError_t launch_kept_rows(const Problem& P, const void* K, const int32_t* idx, void* kept,
                             int32_t* kept_len, int32_t* scratch, int* status, cudaStream_t st) {
  int maxk = 0;
  for (int b = 0; b < P.B; ++b) maxk = max(maxk, P.req[b].keep);
  const dim3 grid((maxk + KRT - 1) / KRT, P.Hkv, P.L * P.B);
  const int esz = P.dtype == MMSHIFT_BF16 ? 2 : 4;
  const bool vec = ((reinterpret_cast<uintptr_t>(K) | (uintptr_t)(P.ls_kv * esz)) & 15) == 0;
  const uint8_t* k = static_cast<const uint8_t*>(K);
  uint8_t* o = static_cast<uint8_t*>(kept);
  int32_t* counts = maxk > kCountAgain ? scratch : nullptr;
  if (counts) {
    kept_count_kernel<<<grid, KRT, 0, st>>>(P, idx, counts);
    const cudaError_t e = cudaGetLastError();
    if (e != cudaSuccess) return e;
  }
  switch (P.d * esz) {
    case 128: kept_rows_kernel<128><<<grid, KRT, 0, st>>>(P, k, idx, counts, o, kept_len, status, vec); break;
    case 256: kept_rows_kernel<256><<<grid, KRT, 0, st>>>(P, k, idx, counts, o, kept_len, status, vec); break;
    case 512: kept_rows_kernel<512><<<grid, KRT, 0, st>>>(P, k, idx, counts, o, kept_len, status, vec); break;
    default: return cudaErrorInvalidValue;
  }
  return cudaGetLastError();
}

cudaError_t launch_coverage_ratio(const Problem& P, const Problem& Pk, float2* all, float2* kept,
                                  float* cov, cudaStream_t st) {
  int run[2] = {1, 1};
  for (int k = 0; k < 2; ++k) {
    const Problem& Q = k ? Pk : P;
    int ns = 0;
    for (int b = 0; b < Q.B; ++b) ns = max(ns, Q.req[b].nsplit * Q.part_slots);
    if (ns <= kRun) continue;
    run[k] = kRun;
    ratio_runs_kernel<<<dim3(Q.Prows_pad / 128 * ((ns + kRun - 1) / kRun), Q.Hkv, Q.L * Q.B), 128, 0, st>>>(
        Q, k ? kept : all);
    const cudaError_t e = cudaGetLastError();
    if (e != cudaSuccess) return e;
  }
  // all query heads of a KV head side by side, up to 128 (32 queries, 128 heads over
  // one KV head, 4096 keys: 125 us a call with eight at a time, 65 with 32, 51 so)
  const int heads = (P.r + 7) / 8 * 8;
  if (heads <= 32)
    ratio_kernel<32><<<dim3((P.Np + 31) / 32, P.Hkv, P.L * P.B), 32 * heads, 0, st>>>(
        P, Pk, all, kept, run[0], run[1], cov);
  else
    ratio_kernel<8><<<dim3((P.Np + 7) / 8, P.Hkv, P.L * P.B), 8 * min(128, heads), 0, st>>>(
        P, Pk, all, kept, run[0], run[1], cov);
  return cudaGetLastError();
}

cudaError_t launch_coverage(const Problem& P, const Buffers& bf, const int32_t* idx, float* cov,
                            cudaStream_t st) {
  if (P.G == 0 || P.R == 0) return cudaSuccess;
  dim3 grid(P.G, P.Hkv, P.L * P.B);
  coverage_kernel<<<grid, kCovThreads, 0, st>>>(P, bf.gmass, idx, cov, bf.status);
  return cudaGetLastError();
}

}  // namespace mmshift
