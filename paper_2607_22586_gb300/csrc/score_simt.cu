// Steps 2-4 on CUDA cores (fp32 FMA): proxy logits, row softmax over the whole
// prompt and group-mass aggregation (Section 3.2.2; Appendix B).
//
// This path serves float32 inputs, for which the tensor cores would round the
// operands (TF32), and head dims or shapes the tcgen05 path does not cover.
//
// Both passes form logits in 64 x 128 tiles (proxy rows x keys) of 128 threads,
// 8 x 8 per thread, from operands stored transposed in shared memory, so a
// step of the contraction costs four 16-byte loads per 64 FMAs. Every logit is
// one chain of FMAs over ascending dimensions.
// Pass 1: a cluster of up to eight CTAs takes one key split of 64 proxy rows,
//   each CTA a range of its 128-key tiles; per row and 64 keys a (max, sum of
//   exp2) pair of the log2-scaled logits x = s * alpha, alpha = softmax_scale
//   * log2(e), all merged in key order by the cluster's first CTA. Cluster
//   sizes change who computes a tile, not the result.
// Merge: combines the partials of each row (one per key split, four on the
//   tensor-core path) in a fixed order into c = m + log2(Z) (the log2
//   normaliser), +inf for padding rows so they weigh nothing.
// Pass 2: CTA = (layer, KV head, 128 keys, a range of groups). It streams the
//   groups' proxy rows, recomputes the logits and adds exp2(x - c), 16 rows at
//   a time in ascending order, into the group masses and the anchor (mean over
//   the r anchor rows).
#include <algorithm>

#include "common.cuh"
#include "group_ranges.h"
#include "umma.cuh"

namespace mmshift {
namespace {

constexpr int TR = 64;      // proxy rows per tile
constexpr int TK = 128;     // keys per tile: two runs of 64
constexpr int TNT = 128;    // threads: 8 row groups (8 rows) x 16 key groups (4 + 4 keys)
constexpr int TRUN = 64;    // keys per (max, sum) pair

__device__ __forceinline__ void find_split(const Problem& P, int s, int& b, int& sl) {
  b = 0;
  while (b + 1 < P.B && P.req[b + 1].split_off <= s) ++b;
  sl = s - P.req[b].split_off;
}

// A value the call's input keeps for the whole call (INPUT: by the non-coherent
// path), or one an earlier kernel of the call wrote.
template <bool INPUT, typename V>
__device__ __forceinline__ V load(const V* p) {
  if constexpr (INPUT) return __ldg(p);
  else return *p;
}

// Four consecutive elements as float32 (`vec`: the pointer allows one load).
template <bool INPUT>
__device__ __forceinline__ float4 load4(const float* p, bool vec) {
  if (vec) return load<INPUT>(reinterpret_cast<const float4*>(p));
  return make_float4(load<INPUT>(p), load<INPUT>(p + 1), load<INPUT>(p + 2), load<INPUT>(p + 3));
}
template <bool INPUT>
__device__ __forceinline__ float4 load4(const __nv_bfloat16* p, bool vec) {
  if (vec) {
    const uint2 u = load<INPUT>(reinterpret_cast<const uint2*>(p));
    return make_float4(__uint_as_float(u.x << 16), __uint_as_float(u.x & 0xffff0000u),
                       __uint_as_float(u.y << 16), __uint_as_float(u.y & 0xffff0000u));
  }
  return make_float4(to_f32(p[0]), to_f32(p[1]), to_f32(p[2]), to_f32(p[3]));
}

// Shared-memory place of element (row, k) of a transposed tile of R rows
// (R = 64 or 128). The rows of dimensions 4q..4q+3 are permuted in blocks of
// eight by q mod 4, which spreads a warp's stores (8 rows x 4 quads) over all
// banks; a thread still finds its four or eight rows side by side.
template <int R>
__device__ __forceinline__ int tile_at(int row, int k) { return k * R + (row ^ (((k >> 2) & 3) << 3)); }

// R rows x KD dimensions of src (INPUT as above; rows `stride` elements apart, zeros from row n
// on), read into registers and stored to a tile in two steps, so that the
// reads of the next piece are in flight during the FMAs of the current one.
template <typename T, int R, int KD, bool INPUT>
struct Piece {
  static constexpr int NB = (R / 8) * (KD / 16) / (TNT / 32);   // 8-row x 16-dimension blocks per warp
  float4 v[NB];
  __device__ __forceinline__ static void at(int i, int& row, int& k) {
    const int e = i * (TNT / 32) + threadIdx.x / 32, lane = threadIdx.x % 32;
    row = (e / (KD / 16)) * 8 + (lane & 7);
    k = (e % (KD / 16)) * 16 + (lane >> 3) * 4;
  }
  __device__ __forceinline__ void load(const T* src, size_t stride, int n, bool vec) {
#pragma unroll
    for (int i = 0; i < NB; ++i) {
      int row, k;
      at(i, row, k);
      v[i] = row < n ? load4<INPUT>(src + (size_t)row * stride + k, vec) : make_float4(0.f, 0.f, 0.f, 0.f);
    }
  }
  __device__ __forceinline__ void store(float* dst) const {
#pragma unroll
    for (int i = 0; i < NB; ++i) {
      int row, k;
      at(i, row, k);
      float* d = dst + tile_at<R>(row, k);
      d[0] = v[i].x;
      d[R] = v[i].y;
      d[2 * R] = v[i].z;
      d[3 * R] = v[i].w;
    }
  }
};

constexpr int KC = 32;      // dimensions per streamed piece

// acc[i][j / 2] += row (ty * 8 + i) . keys (j, j + 1) of the thread over KC
// dimensions: keys 4 tx .. 4 tx + 3 (j < 4) and 64 + 4 tx .. (j >= 4), in pairs
// (a packed FMA rounds each half like a scalar one). Bound by FMA issue: 42
// TFLOP/s on one layer of 4096 keys, d = 128, paper hyper-parameters. With 4 x 4
// per thread and row-major tiles (two shared-memory loads per four FMAs) that
// selection took 1398 us, now 803; one layer of 4001 keys with 1,024 packed
// rows per KV head 398 -> 290 us, one layer of 1024 keys, d = 64, 294 -> 101 us
// (36 and 16 CTAs before, 264 and 272 now). Scalar FMAs take 331 us on the second.
__device__ __forceinline__ void tile_dot(const float* As, const float* Bs, int ty, int tx,
                                         uint64_t (&acc)[8][4]) {
#pragma unroll 1
  for (int k0 = 0; k0 < KC; k0 += 16) {
#pragma unroll
    for (int kk = 0; kk < 16; ++kk) {
      const int x = (kk >> 2) << 3;            // tile_at's permutation of dimension k0 + kk
      const float* ap = As + (k0 + kk) * TR + ((ty * 8) ^ x);
      const float* bp = Bs + (k0 + kk) * TK + ((tx * 4) ^ x);
      const float4 a0 = *reinterpret_cast<const float4*>(ap);
      const float4 a1 = *reinterpret_cast<const float4*>(ap + 4);
      const ulonglong2 b0 = *reinterpret_cast<const ulonglong2*>(bp);
      const ulonglong2 b1 = *reinterpret_cast<const ulonglong2*>(bp + TRUN);
      const float a[8] = {a0.x, a0.y, a0.z, a0.w, a1.x, a1.y, a1.z, a1.w};
      const uint64_t b[4] = {b0.x, b0.y, b1.x, b1.y};
#pragma unroll
      for (int i = 0; i < 8; ++i) {
        const uint64_t aa = umma::pk2(a[i], a[i]);
#pragma unroll
        for (int j = 0; j < 4; ++j) acc[i][j] = umma::ffma2(aa, b[j], acc[i][j]);
      }
    }
  }
}
__device__ __forceinline__ void clear(uint64_t (&acc)[8][4]) {
#pragma unroll
  for (int i = 0; i < 8; ++i)
#pragma unroll
    for (int j = 0; j < 4; ++j) acc[i][j] = 0;     // (+0, +0)
}
// Logit j (0-7) of row i.
__device__ __forceinline__ float logit(const uint64_t (&acc)[8][4], int i, int j) {
  float lo, hi;
  umma::upk2(acc[i][j >> 1], lo, hi);
  return (j & 1) ? hi : lo;
}

// RATIO: the sums feed a ratio (coverage), over at most bf.kept_len keys where
// given; a NaN logit then makes its row's sum NaN, also where all logits of its
// 16 keys are NaN, which the selection's maxima pass over.
template <typename T, int D, bool RATIO>
__global__ void __launch_bounds__(TNT, 3) pass1_simt(const __grid_constant__ Problem P, Buffers bf,
                                                  const T* K, int nrank, bool vec) {
  dependent_start();
  extern __shared__ float sm[];
  float* As = sm;                    // [D][64] proxy rows
  float* Bs = As + TR * D;           // [2][KC][128] keys, a piece and the next one
  float2* pairs = reinterpret_cast<float2*>(Bs + 2 * KC * TK);   // [runs of this CTA][64] (max, sum)
  const int n_rt = (P.Prows + TR - 1) / TR;
  int u = blockIdx.x;
  const int rank = u % nrank; u /= nrank;
  const int rt = u % n_rt; u /= n_rt;
  const int s = u % P.total_splits; u /= P.total_splits;
  const int h = u, l = blockIdx.y;
  int b, sl;
  find_split(P, s, b, sl);
  const int t_len = P.req[b].t_len, tok_off = P.req[b].tok_off;
  const int t0 = sl * P.split_len;
  int t1 = min(t_len, t0 + P.split_len);
  if (RATIO && bf.kept_len) t1 = min(t1, bf.kept_len[((size_t)l * P.B + b) * P.Hkv + h]);
  const int tid = threadIdx.x, ty = tid / 16, tx = tid % 16;
  // this CTA's tiles of the split: rank r takes tiles [r, r + 1) * ntiles / nrank
  const int ntiles = max(0, t1 - t0 + TK - 1) / TK;
  const int k0 = rank * ntiles / nrank, k1 = (rank + 1) * ntiles / nrank;

  const T* pk = (const T*)bf.packed +
                ((((size_t)l * P.B + b) * P.Hkv + h) * P.Prows_pad + (size_t)rt * TR) * D;
  const size_t kstride = (size_t)P.Hkv * D;
  const T* kb = K + (size_t)l * P.ls_kv + (size_t)tok_off * kstride + (size_t)h * D;
  // pieces of KC dimensions of the CTA's tiles, one after the other
  constexpr int NP = D / KC;
  const int np = (k1 - k0) * NP;
  Piece<T, TK, KC, true> next;
  auto fetch = [&](int p) {
    const int tk = t0 + (k0 + p / NP) * TK;
    next.load(kb + (size_t)tk * kstride + (p % NP) * KC, kstride, t1 - tk, vec);
  };
  if (np) {
    fetch(0);
#pragma unroll 1
    for (int c = 0; c < NP; ++c) {              // Prows_pad is a multiple of TR
      Piece<T, TR, KC, false> a;
      a.load(pk + c * KC, D, TR, true);
      a.store(As + c * KC * TR);
    }
    next.store(Bs);
  }
  __syncthreads();
  uint64_t acc[8][4];
#pragma unroll 1
  for (int p = 0; p < np; ++p) {
    const int c = p % NP, kt = k0 + p / NP, tk = t0 + kt * TK;
    if (p + 1 < np) fetch(p + 1);
    if (c == 0) clear(acc);
    tile_dot(As + c * KC * TR, Bs + (p & 1) * KC * TK, ty, tx, acc);
    if (p + 1 < np) next.store(Bs + ((p + 1) & 1) * KC * TK);
    __syncthreads();
    if (c != NP - 1) continue;
#pragma unroll
    for (int half = 0; half < 2; ++half) {
#pragma unroll
      for (int i = 0; i < 8; ++i) {
        // 16 keys are the four keys of four lanes in a row: their max, then
        // their sum as one chain over ascending keys
        float x[4], m = -INFINITY;
#pragma unroll
        for (int j = 0; j < 4; ++j) {
          x[j] = tk + half * TRUN + tx * 4 + j < t1 ? logit(acc, i, half * 4 + j) * P.alpha : -INFINITY;
          m = fmaxf(m, RATIO && x[j] != x[j] ? INFINITY : x[j]);
        }
        m = fmaxf(m, __shfl_xor_sync(0xffffffffu, m, 1));
        m = fmaxf(m, __shfl_xor_sync(0xffffffffu, m, 2));
        float z = 0.f;
        if (m != -INFINITY) {
#pragma unroll
          for (int j = 0; j < 4; ++j) x[j] = fast_exp2(x[j] - m);
        } else {
#pragma unroll
          for (int j = 0; j < 4; ++j) x[j] = 0.f;
        }
#pragma unroll
        for (int step = 0; step < 4; ++step) {
          const float zin = __shfl_up_sync(0xffffffffu, z, 1);
          if ((tx & 3) == step) {
            z = step ? zin : 0.f;
#pragma unroll
            for (int j = 0; j < 4; ++j) z += x[j];
          }
        }
        z = __shfl_sync(0xffffffffu, z, (tid & 28) | 3);
        // the run's four 16-key pairs, two by two
#pragma unroll
        for (int off = 4; off < 16; off <<= 1) {
          const float m2 = __shfl_xor_sync(0xffffffffu, m, off);
          const float z2 = __shfl_xor_sync(0xffffffffu, z, off);
          merge_ms(m, z, m2, z2);
        }
        if (tx == 0) pairs[(size_t)((kt - k0) * 2 + half) * TR + ty * 8 + i] = make_float2(m, z);
      }
    }
  }
  if (nrank > 1) umma::cluster_sync(); else __syncthreads();
  if (rank == 0 && tid < TR && rt * TR + tid < P.Prows_pad) {
    float run_m = -INFINITY, run_z = 0.f;
    for (int r = 0; r < nrank; ++r) {
      const int n = 2 * ((r + 1) * ntiles / nrank - r * ntiles / nrank);
      for (int i = 0; i < n; ++i) {
        const float2* p = pairs + (size_t)i * TR + tid;
        const float2 v = r == 0 ? *p : umma::ld_cluster_f2(umma::mapa(umma::smem_u32(p), (uint32_t)r));
        merge_ms(run_m, run_z, v.x, v.y);
      }
    }
    bf.part[(((size_t)l * P.Hkv + h) * P.total_splits + s) * P.part_slots * P.Prows_pad +
            rt * TR + tid] = make_float2(run_m, run_z);
  }
  if (nrank > 1) umma::cluster_sync();   // no CTA leaves while the first may still read its pairs
}

// SUB threads per row (four when a row has at least 128 partials, else one):
// thread q of a row merges the row's partials q, q + SUB, q + 2 SUB, ... in
// order (eight loads issued ahead), then the SUB results are merged by xor
// shuffles; for a given SUB the order is fixed, and SUB depends only on the
// call's shape.
template <int kMergeSub>
__global__ void merge_kernel(const __grid_constant__ Problem P, const __grid_constant__ Buffers bf) {
  dependent_start();
  const int q = threadIdx.x % kMergeSub;
  const int p = blockIdx.x * (blockDim.x / kMergeSub) + threadIdx.x / kMergeSub;
  const int bh = blockIdx.y, l = blockIdx.z;
  const int b = bh / P.Hkv, h = bh - b * P.Hkv;
  // with anchor_split the softmax pass has no partials for the anchor rows
  const int rows = P.anchor_split ? P.n_group_rows : P.Prows_pad;
  const bool live = p < rows;
  const ReqInfo R = P.req[b];
  float m = -INFINITY, z = 0.f;
  const float2* src = bf.part +
                      (((size_t)l * P.Hkv + h) * P.total_splits + R.split_off) * P.part_slots * P.Prows_pad +
                      (live ? p : 0);
  const int ns = live ? R.nsplit * P.part_slots : 0;
  constexpr int A = 8;
  for (int s0 = q; s0 < ns; s0 += A * kMergeSub) {
    float2 v[A];
#pragma unroll
    for (int u = 0; u < A; ++u) {
      const int si = s0 + u * kMergeSub;
      v[u] = si < ns ? src[(size_t)si * P.Prows_pad] : make_float2(-INFINITY, 0.f);
    }
#pragma unroll
    for (int u = 0; u < A; ++u)
      if (s0 + u * kMergeSub < ns) merge_ms(m, z, v[u].x, v[u].y);
  }
#pragma unroll
  for (int off = 1; off < kMergeSub; off <<= 1) {
    const float m2 = __shfl_xor_sync(0xffffffffu, m, off);
    const float z2 = __shfl_xor_sync(0xffffffffu, z, off);
    merge_ms(m, z, m2, z2);
  }
  if (!live || q) return;
  const bool valid = row_kind(P, p).group >= 0;
  bf.cvals[(((size_t)l * P.B + b) * P.Hkv + h) * P.Prows_pad + p] =
      valid ? m + __log2f(z) : INFINITY;
}

template <typename T, int D>
__global__ void __launch_bounds__(TNT, 2) pass2_simt(const __grid_constant__ Problem P, Buffers bf,
                                                  const T* K, GroupRanges gr, bool vec) {
  dependent_start();
  extern __shared__ float sm[];
  float* Bs = sm;                    // [D][128] keys (stationary)
  float* As = Bs + TK * D;           // [2][KC][64] proxy rows, a piece and the next one
  float* sums = As + 2 * KC * TR;    // [4][128] sums over 16 rows
  // the longest ranges start first
  const int l = blockIdx.y, per = gridDim.x / gr.ngr;
  const int range = gr.own ? (int)blockIdx.x / per : gr.ngr - 1 - (int)blockIdx.x / per;
  int u = blockIdx.x % per;
  int g0, g1;
  range_groups(gr, P.G, range, g0, g1);
  const int h = u % P.Hkv;
  u /= P.Hkv;
  int b = 0;
  for (; b < P.B; ++b) {
    const int nt = (P.req[b].t_len + TK - 1) / TK;
    if (u < nt) break;
    u -= nt;
  }
  const int t_len = P.req[b].t_len, tok_off = P.req[b].tok_off;
  const int kt = u * TK;
  const int tid = threadIdx.x, ty = tid / 16, tx = tid % 16, lane = tid % 32, w = tid / 32;
  const size_t kstride = (size_t)P.Hkv * D;
  const T* kb = K + (size_t)l * P.ls_kv + ((size_t)tok_off + kt) * kstride + (size_t)h * D;
  const T* pk = (const T*)bf.packed + ((((size_t)l * P.B + b) * P.Hkv + h) * P.Prows_pad) * D;
  const float* cv = bf.cvals + (((size_t)l * P.B + b) * P.Hkv + h) * P.Prows_pad;
  // 16-row chunks of the groups g0 .. g1 - 1
  const int c_lo = g0 * (P.RG / kChunk);
  const int c_hi = g1 <= P.G ? g1 * (P.RG / kChunk) : P.Prows / kChunk;
  const int t = kt + tid;            // the key whose masses this thread adds up
  int cur = g0;
  float gsum = 0.f;
  auto flush = [&] {
    if (t < t_len) {
      const size_t col = (size_t)tok_off + t;
      if (cur < P.G) bf.gmass[(((size_t)l * P.Hkv + h) * P.G + cur) * P.total_T + col] = gsum;
      else bf.anchor[((size_t)l * P.Hkv + h) * P.total_T + col] = gsum / (float)P.r;
    }
    gsum = 0.f;
  };
  // pieces of KC dimensions of the 64-row tiles, one after the other
  constexpr int NP = D / KC, CPT = TR / kChunk;
  const int np = (c_hi - c_lo + CPT - 1) / CPT * NP;
  Piece<T, TR, KC, false> next;
  auto fetch = [&](int p) {
    const int row0 = (c_lo + p / NP * CPT) * kChunk;
    next.load(pk + (size_t)row0 * D + (p % NP) * KC, D, P.Prows_pad - row0, true);
  };
  fetch(0);
#pragma unroll 1
  for (int c = 0; c < NP; ++c) {
    Piece<T, TK, KC, true> k;
    k.load(kb + c * KC, kstride, t_len - kt, vec);
    k.store(Bs + c * KC * TK);
  }
  next.store(As);
  __syncthreads();
  uint64_t acc[8][4];
  float cn[8];            // cn: normalisers of the thread's eight rows
#pragma unroll 1
  for (int p = 0; p < np; ++p) {
    const int pc = p % NP, c0 = c_lo + p / NP * CPT;
    if (p + 1 < np) fetch(p + 1);
    if (pc == 0) {
      clear(acc);
      const int row = c0 * kChunk + ty * 8;     // rows in eights: all or none inside
#pragma unroll
      for (int i = 0; i < 8; ++i) cn[i] = row < P.Prows_pad ? cv[row + i] : INFINITY;
    }
    tile_dot(As + (p & 1) * KC * TR, Bs + pc * KC * TK, ty, tx, acc);
    if (p + 1 < np) next.store(As + ((p + 1) & 1) * KC * TR);
    if (pc != NP - 1) {
      __syncthreads();
      continue;
    }
    // per key, the 16 rows of a chunk (two threads: lanes i and i + 16) as one
    // chain over ascending rows
#pragma unroll
    for (int j = 0; j < 8; ++j) {
      float e[8], z = 0.f;
#pragma unroll
      for (int i = 0; i < 8; ++i) e[i] = fast_exp2(fmaf(logit(acc, i, j), P.alpha, -cn[i]));
      if (lane < 16) {
#pragma unroll
        for (int i = 0; i < 8; ++i) z += e[i];
      }
      z = __shfl_sync(0xffffffffu, z, lane & 15);
      if (lane >= 16) {
#pragma unroll
        for (int i = 0; i < 8; ++i) z += e[i];
        sums[w * TK + (j < 4 ? 0 : TRUN) + tx * 4 + (j & 3)] = z;
      }
    }
    __syncthreads();
    for (int c = 0; c < CPT && c0 + c < c_hi; ++c) {
      const int g = chunk_group(P, c0 + c);
      if (g != cur) { flush(); cur = g; }
      gsum += sums[c * TK + tid];
    }
    __syncthreads();   // the sums are read before the next tile's are written
  }
  flush();
}

cudaError_t device_sms(int* nsm) {
  int dev = 0;
  const cudaError_t e = cudaGetDevice(&dev);
  return e != cudaSuccess ? e : cudaDeviceGetAttribute(nsm, cudaDevAttrMultiProcessorCount, dev);
}

// Four elements of a row in one load: K's base, rows and layers allow it.
template <typename T>
bool quad_loads(const Problem& P, const void* K) {
  const size_t quad = 4 * sizeof(T);
  return reinterpret_cast<uintptr_t>(K) % quad == 0 && (P.ls_kv * sizeof(T)) % quad == 0;
}

template <typename T, int D, bool RATIO>
cudaError_t launch_pass1(const Problem& P, const Buffers& bf, cudaStream_t st, const void* K) {
  int nsm = 0;
  cudaError_t e = device_sms(&nsm);
  if (e != cudaSuccess) return e;
  const bool vec = quad_loads<T>(P, K);
  // pass 1: more CTAs per split (a cluster), up to one per 128-key tile, until
  // each SM has its three CTAs: more of them read the proxy rows once more
  // each (4 rounds: 344 us against 331 on 4001 keys, 930 against 899 at 4096 keys
  // with paper hyper-parameters), fewer leave SMs idle on short calls
  const int n_rt = (P.Prows + TR - 1) / TR;
  int max_len = 1;
  for (int b = 0; b < P.B; ++b) max_len = std::max(max_len, std::min(P.req[b].t_len, P.split_len));
  const int max_tiles = (max_len + TK - 1) / TK;
  const long long units = (long long)P.Hkv * P.total_splits * n_rt * P.L;
  int nrank = 1;
  while (nrank < 8 && nrank < max_tiles && units * nrank < 3LL * nsm) nrank *= 2;
  const int runs = 2 * ((max_tiles + nrank - 1) / nrank);
  const size_t sm1 = (size_t)(TR * D + 2 * KC * TK) * sizeof(float) + (size_t)runs * TR * sizeof(float2);
  if ((e = cudaFuncSetAttribute(pass1_simt<T, D, RATIO>, cudaFuncAttributeMaxDynamicSharedMemorySize,
                                (int)sm1)) != cudaSuccess) return e;
  return launch_kernel(pass1_simt<T, D, RATIO>, dim3((unsigned)(P.Hkv * P.total_splits * n_rt * nrank), P.L), TNT,
                       sm1, st, P.overlap, nrank, P, bf, (const T*)K, nrank, vec);
}

template <typename T, int D>
cudaError_t launch_t(const Problem& P, const Buffers& bf, cudaStream_t st, const void* K,
                     cudaEvent_t* ev) {
  int nsm = 0;
  cudaError_t e = device_sms(&nsm);
  if (e != cudaSuccess) return e;
  const bool vec = quad_loads<T>(P, K);
  if (ev && (e = cudaEventRecord(ev[1], st)) != cudaSuccess) return e;
  if ((e = launch_pass1<T, D, false>(P, bf, st, K)) != cudaSuccess) return e;
  if (ev && (e = cudaEventRecord(ev[2], st)) != cudaSuccess) return e;
  if ((e = launch_merge(P, bf, st)) != cudaSuccess) return e;
  if (ev && (e = cudaEventRecord(ev[3], st)) != cudaSuccess) return e;
  long long tiles = 0;
  for (int b = 0; b < P.B; ++b) tiles += (P.req[b].t_len + TK - 1) / TK;
  const long long keyu = tiles * P.Hkv * P.L;
  const GroupRanges gr = choose_ranges(P.G, P.RG, P.anchor_rows, TR, keyu, nsm);
  const size_t sm2 = (size_t)(TK * D + 2 * KC * TR + 4 * TK) * sizeof(float);
  if ((e = cudaFuncSetAttribute(pass2_simt<T, D>, cudaFuncAttributeMaxDynamicSharedMemorySize,
                                (int)sm2)) != cudaSuccess) return e;
  return launch_kernel(pass2_simt<T, D>, dim3((unsigned)(tiles * P.Hkv * gr.ngr), P.L), TNT, sm2, st,
                       P.overlap, 0, P, bf, (const T*)K, gr, vec);
}

}  // namespace

cudaError_t launch_merge(const Problem& P, const Buffers& bf, cudaStream_t st) {
  int max_ns = 0;
  for (int b = 0; b < P.B; ++b) max_ns = max(max_ns, P.req[b].nsplit * P.part_slots);
  const int rows = P.anchor_split ? P.n_group_rows : P.Prows_pad;
  if (max_ns >= 128) {
    constexpr int threads = 256, rows_per_block = threads / 4;
    dim3 grid((rows + rows_per_block - 1) / rows_per_block, P.B * P.Hkv, P.L);
    return launch_kernel(merge_kernel<4>, grid, threads, 0, st, P.overlap, 0, P, bf);
  } else {
    constexpr int threads = 128;
    dim3 grid((rows + threads - 1) / threads, P.B * P.Hkv, P.L);
    return launch_kernel(merge_kernel<1>, grid, threads, 0, st, P.overlap, 0, P, bf);
  }
}

cudaError_t launch_softmax_simt(const Problem& P, const Buffers& bf, cudaStream_t st,
                                const void* K) {
  if (P.dtype == MMSHIFT_BF16)
    return P.d == 128 ? launch_pass1<__nv_bfloat16, 128, true>(P, bf, st, K)
                      : launch_pass1<__nv_bfloat16, 64, true>(P, bf, st, K);
  return P.d == 128 ? launch_pass1<float, 128, true>(P, bf, st, K)
                    : launch_pass1<float, 64, true>(P, bf, st, K);
}

cudaError_t launch_score_simt(const Problem& P, const Buffers& bf, cudaStream_t st,
                              const void* K, cudaEvent_t* ev) {
  if (P.dtype == MMSHIFT_BF16)
    return P.d == 128 ? launch_t<__nv_bfloat16, 128>(P, bf, st, K, ev)
                      : launch_t<__nv_bfloat16, 64>(P, bf, st, K, ev);
  return P.d == 128 ? launch_t<float, 128>(P, bf, st, K, ev)
                    : launch_t<float, 64>(P, bf, st, K, ev);
}

}  // namespace mmshift
