// Routing, shuffle and unshuffle kernels of the expert-choice layer (Section 3.2, Eq. 2-4)
// and the element-wise parts of its backward pass.  Everything here is bandwidth- or
// latency-bound integer / fp32 work; the dense contractions live in gemm_*.cu.
#include "internal.h"
#include "tc_ptx.cuh"

#include <string.h>

namespace ecmoe {

// ------------------------------------------------------------------------------------------
// small helpers
// ------------------------------------------------------------------------------------------
__device__ __forceinline__ float ld_f(const float* p, int64_t i) { return p[i]; }
__device__ __forceinline__ float ld_f(const bf16* p, int64_t i) { return __bfloat162float(p[i]); }

template <typename T> struct Vec;            // one 16-byte vector of T
template <> struct Vec<float> {
  static constexpr int N = 4;
  __device__ static void unpack(const uint4& v, float* f) {
    f[0] = __uint_as_float(v.x); f[1] = __uint_as_float(v.y);
    f[2] = __uint_as_float(v.z); f[3] = __uint_as_float(v.w);
  }
  __device__ static uint4 pack(const float* f) {
    return make_uint4(__float_as_uint(f[0]), __float_as_uint(f[1]), __float_as_uint(f[2]),
                      __float_as_uint(f[3]));
  }
};
template <> struct Vec<bf16> {
  static constexpr int N = 8;
  __device__ static void unpack(const uint4& v, float* f) {
    const unsigned w[4] = {v.x, v.y, v.z, v.w};
#pragma unroll
    for (int i = 0; i < 4; ++i) {            // bf16 -> fp32 is a 16-bit shift
      f[2 * i] = __uint_as_float(w[i] << 16);
      f[2 * i + 1] = __uint_as_float(w[i] & 0xFFFF0000u);
    }
  }
  __device__ static uint4 pack(const float* f) {
    unsigned w[4];
#pragma unroll
    for (int i = 0; i < 4; ++i) {
      __nv_bfloat162 p = __floats2bfloat162_rn(f[2 * i], f[2 * i + 1]);
      w[i] = *reinterpret_cast<unsigned*>(&p);
    }
    return make_uint4(w[0], w[1], w[2], w[3]);
  }
};

__device__ __forceinline__ void cluster_barrier() {
  asm volatile("barrier.cluster.arrive.release.aligned;\n barrier.cluster.wait.acquire.aligned;" ::: "memory");
}
// this CTA's shared-memory address as CTA `rank` of the cluster has it
__device__ __forceinline__ unsigned cluster_address(const void* p, int rank) {
  unsigned r; asm volatile("mapa.shared::cluster.u32 %0, %1, %2;" : "=r"(r) : "r"((unsigned)__cvta_generic_to_shared(p)), "r"(rank)); return r;
}

static inline unsigned grid_for(int64_t work, int threads, int64_t cap = 148 * 16) {
  int64_t b = (work + threads - 1) / threads;
  if (b < 1) b = 1;
  if (b > cap) b = cap;
  return (unsigned)b;
}

// ------------------------------------------------------------------------------------------
// Gate, Eq. 2: S = Softmax(X . Wg) over the experts of each token.  FMA version (fp32 path and
// shapes the tensor-core kernel does not take).
//
// A CTA computes the logits of 32 tokens.  Its eight warps are NG column groups of 32 experts times KS = 8 / NG slices of
// the contraction: with few experts the work is a long sum per logit, and the slices keep all warps busy.  A chunk is 16
// depths per slice; the next one travels to registers while the current one is multiplied (packed pairs, four tokens
// times eight experts per thread).  The slices' sums join in ascending order, then a warp turns rows into their softmax.
// Bound by the latency of a chunk (a CTA is alone on its SM at the layer's sizes).  2048 x 512 fp32, 16 experts: 65 us with a
// thread per logit walking the whole row, 18 us now; 6080 x 1000 bf16, 10 experts: 100 and 30 us.
// ------------------------------------------------------------------------------------------
constexpr int kGateTT = 32, kGateThreads = 256, kGateSlice = 16;

__device__ __forceinline__ void gate_ld4(const float* p, float* f) {
  const float4 v = *reinterpret_cast<const float4*>(p); f[0] = v.x; f[1] = v.y; f[2] = v.z; f[3] = v.w;
}
__device__ __forceinline__ void gate_ld4(const bf16* p, float* f) {
  const uint2 v = *reinterpret_cast<const uint2*>(p);
  f[0] = __uint_as_float(v.x << 16); f[1] = __uint_as_float(v.x & 0xFFFF0000u);
  f[2] = __uint_as_float(v.y << 16); f[3] = __uint_as_float(v.y & 0xFFFF0000u);
}
__host__ __device__ constexpr int gate_smem_bytes(int NG) { return 2 * (8 / NG) * kGateSlice * (kGateTT + 32 * NG) * 4; }

// WVEC: rows of Wg are whole 16-byte (fp32) or 8-byte (bf16) groups of four
template <typename T, int NG, bool WVEC>
__global__ void __launch_bounds__(kGateThreads)
gate_softmax_simt_kernel(const T* __restrict__ X, const T* __restrict__ Wg, float* __restrict__ S, int64_t n, int d, int E,
                         const SlotMarks marks, int* status) {
  chain_enter();
  if (blockIdx.x == 0) for (int i = threadIdx.x; i < kStatusWords; i += kGateThreads) status[i] = 0;     // the first kernel of a call
  X = after_enter(X); Wg = after_enter(Wg);
  constexpr int KS = 8 / NG, DK = KS * kGateSlice, C = 32 * NG;         // chunk: DK depths of 32 tokens and of C experts
  constexpr int kX = DK * kGateTT, kW = DK * C, XQ = (kX / 4 + kGateThreads - 1) / kGateThreads, WQ = kW / 4 / kGateThreads;
  extern __shared__ __align__(16) float gate_smem[];                    // [2][X chunk [DK][32] | W chunk [DK][C]]
  const int tid = threadIdx.x, warp = tid >> 5, lane = tid & 31;
  const int64_t t0 = (int64_t)blockIdx.x * kGateTT;
  float xv[XQ][4], wv[WQ][4];
  // X quad q of this thread: four depths of one token; a warp covers 8 tokens x 64 bytes (fp32), and the XOR by 8 spreads
  // the transposed stores over the banks.  W quad: four experts at one depth.
  auto x_at = [&](int q, int& tok, int& k) {
    const int w = warp + 8 * q;
    tok = (w & 3) * 8 + (lane >> 2); k = ((w >> 2) * 4 + (lane & 3)) * 4;
  };
  auto fetch = [&](int d0) {
#pragma unroll
    for (int q = 0; q < XQ; ++q) {
      int tok, k; x_at(q, tok, k);
      const int64_t t = min(t0 + tok, n - 1);
      gate_ld4(X + t * d + (d0 + k < d ? d0 + k : 0), xv[q]);
    }
#pragma unroll
    for (int q = 0; q < WQ; ++q) {
      const int idx = tid + q * kGateThreads, k = d0 + idx / (C / 4), c = (idx % (C / 4)) * 4;
      const T* row = Wg + (int64_t)(k < d ? k : 0) * E;
      if constexpr (WVEC) gate_ld4(row + (c < E ? c : 0), wv[q]);
      else {
#pragma unroll
        for (int j = 0; j < 4; ++j) wv[q][j] = ld_f(row, c + j < E ? c + j : 0);
      }
    }
  };
  auto put = [&](float* buf, int d0) {                // what lies beyond d or E becomes zero here, after the loads have landed
#pragma unroll
    for (int q = 0; q < XQ; ++q) {
      int tok, k; x_at(q, tok, k);
      if (k < DK) {
        const bool ok = d0 + k < d;
#pragma unroll
        for (int j = 0; j < 4; ++j) buf[(k + j) * kGateTT + (tok ^ (((k >> 2) & 3) * 8))] = ok ? xv[q][j] : 0.f;
      }
    }
#pragma unroll
    for (int q = 0; q < WQ; ++q) {
      const int idx = tid + q * kGateThreads, kk = idx / (C / 4), c = (idx % (C / 4)) * 4;
      const bool ok = d0 + kk < d;
      float4 v;
      v.x = ok && c < E ? wv[q][0] : 0.f; v.y = ok && c + 1 < E ? wv[q][1] : 0.f;
      v.z = ok && c + 2 < E ? wv[q][2] : 0.f; v.w = ok && c + 3 < E ? wv[q][3] : 0.f;
      *reinterpret_cast<float4*>(buf + kX + kk * C + c) = v;
    }
  };
  const int cg = warp % NG, ks = warp / NG, tg = lane >> 2, cl = cg * 32 + (lane & 3) * 4;
  unsigned long long acc[4][4];                       // token tg * 4 + i, experts cl, cl + 1 | cl + 2, cl + 3 | cl + 16 .. cl + 19
#pragma unroll
  for (int i = 0; i < 4; ++i)
#pragma unroll
    for (int j = 0; j < 4; ++j) acc[i][j] = 0ull;
  fetch(0);
  put(gate_smem, 0);
  __syncthreads();
  int cur = 0;
  for (int d0 = 0; d0 < d; d0 += DK, cur ^= 1) {
    const float* xs = gate_smem + cur * (kX + kW) + ks * kGateSlice * kGateTT;
    const float* ws = gate_smem + cur * (kX + kW) + kX + ks * kGateSlice * C;
    if (d0 + DK < d) fetch(d0 + DK);
#pragma unroll
    for (int kk = 0; kk < kGateSlice; ++kk) {
      const float4 a = *reinterpret_cast<const float4*>(xs + kk * kGateTT + ((tg * 4) ^ (((kk >> 2) & 3) * 8)));
      const ulonglong2 b0 = *reinterpret_cast<const ulonglong2*>(ws + kk * C + cl), b1 = *reinterpret_cast<const ulonglong2*>(ws + kk * C + cl + 16);
      const float av[4] = {a.x, a.y, a.z, a.w};
#pragma unroll
      for (int i = 0; i < 4; ++i) {
        const unsigned long long aa = (unsigned long long)__float_as_uint(av[i]) | ((unsigned long long)__float_as_uint(av[i]) << 32);
        const unsigned long long bb[4] = {b0.x, b0.y, b1.x, b1.y};
#pragma unroll
        for (int j = 0; j < 4; ++j) asm("fma.rn.f32x2 %0, %1, %2, %0;" : "+l"(acc[i][j]) : "l"(aa), "l"(bb[j]));
      }
    }
    if (d0 + DK < d) {                                // the other buffer was last read before the previous barrier
      put(gate_smem + (cur ^ 1) * (kX + kW), d0 + DK);
      __syncthreads();
    }
  }
  __syncthreads();
  float* part = gate_smem;                            // [KS][32 tokens][C]: 32 KiB, no more than the buffers
  static_assert(KS * kGateTT * C <= 2 * (kX + kW), "the partial sums fit the buffers");
#pragma unroll
  for (int i = 0; i < 4; ++i) {
    float* row = part + (ks * kGateTT + tg * 4 + i) * C + cl;
    *reinterpret_cast<ulonglong2*>(row) = make_ulonglong2(acc[i][0], acc[i][1]);
    *reinterpret_cast<ulonglong2*>(row + 16) = make_ulonglong2(acc[i][2], acc[i][3]);
  }
  __syncthreads();
#pragma unroll 1
  for (int tok = warp; tok < kGateTT; tok += 8) {     // a warp per token
    const int64_t t = t0 + tok;
    if (t >= n) break;
    const int words = max(1, marks.per_token);
    if (lane < words) marks.words[t * words + lane] = 0u;
    float v[NG], mx = -INFINITY, sum = 0.f;
#pragma unroll
    for (int j = 0; j < NG; ++j) {
      v[j] = 0.f;
#pragma unroll
      for (int q = 0; q < KS; ++q) v[j] += part[(q * kGateTT + tok) * C + j * 32 + lane];
      if (j * 32 + lane < E) mx = fmaxf(mx, v[j]);
    }
    for (int o = 16; o; o >>= 1) mx = fmaxf(mx, __shfl_xor_sync(0xffffffffu, mx, o));
#pragma unroll
    for (int j = 0; j < NG; ++j) { v[j] = j * 32 + lane < E ? expf(v[j] - mx) : 0.f; sum += v[j]; }
    for (int o = 16; o; o >>= 1) sum += __shfl_xor_sync(0xffffffffu, sum, o);
    const float inv = 1.f / sum;
#pragma unroll
    for (int j = 0; j < NG; ++j) if (j * 32 + lane < E) S[t * E + j * 32 + lane] = v[j] * inv;
  }
}

template <typename T, int NG>
cudaError_t launch_gate_ng(const T* X, const T* Wg, float* S, int64_t n, int d, int E, const SlotMarks& marks, int* status, cudaStream_t st) {
  const unsigned grid = (unsigned)((n + kGateTT - 1) / kGateTT);
  const bool wvec = E % 4 == 0;                       // Wg itself is 16-byte aligned
  auto kern = wvec ? gate_softmax_simt_kernel<T, NG, true> : gate_softmax_simt_kernel<T, NG, false>;
  constexpr int smem = gate_smem_bytes(NG);
  const cudaError_t e = cudaFuncSetAttribute(kern, cudaFuncAttributeMaxDynamicSharedMemorySize, smem);
  if (e != cudaSuccess) return e;
  return launch_chained(kern, dim3(grid), dim3(kGateThreads), smem, st, X, Wg, S, n, d, E, marks, status);
}
template <typename T>
cudaError_t launch_gate_t(const T* X, const T* Wg, float* S, int64_t n, int d, int E, const SlotMarks& marks, int* status, cudaStream_t st) {
  if (E <= 32) return launch_gate_ng<T, 1>(X, Wg, S, n, d, E, marks, status, st);
  if (E <= 64) return launch_gate_ng<T, 2>(X, Wg, S, n, d, E, marks, status, st);
  if (E <= 128) return launch_gate_ng<T, 4>(X, Wg, S, n, d, E, marks, status, st);
  return launch_gate_ng<T, 8>(X, Wg, S, n, d, E, marks, status, st);
}

cudaError_t launch_gate_softmax_simt(int dtype, const void* X, const void* Wg, float* S, int64_t n,
                                     int d, int E, const SlotMarks& marks, int* status, cudaStream_t st) {
  if (E > 256) return cudaErrorInvalidValue;
  return dtype == 0 ? launch_gate_t((const float*)X, (const float*)Wg, S, n, d, E, marks, status, st)
                    : launch_gate_t((const bf16*)X, (const bf16*)Wg, S, n, d, E, marks, status, st);
}

// ------------------------------------------------------------------------------------------
// Column top-k, Eq. 2: G, I = TopK(S^T, k).
//
// Every (token t, expert i) entry gets the 64-bit key  (~bits(S[t,i]) << 32) | t.  0 <= S <= 1, so its
// bit pattern is below 2^30 and monotone in its value: a smaller key is a larger score, and among
// equal scores a lower token.  Keys of one expert are distinct, so "the k smallest keys, ascending"
// is the unique answer with ties broken toward the lower token and slots listed by descending score.
// What is not a score (NaN rows of a model that has diverged) counts as larger than any: the selection goes by
// sel_bits(), which has both top bits set whatever the value, so every column has exactly k winners.
//
// Routing groups (several independent groups of n tokens) multiply the columns: every (group, expert) pair is
// selected on its own and lands in its expert's row of I and G at the group's offset.
//
// Groups of up to kSmallN tokens with k up to one sort tile take one launch (topk_small_kernel, further down:
// one CTA per column does everything in shared memory).  Larger ones take the path described next.
//
// Selection is a most-significant-digit radix select over the 30 significant score bits, 10 bits a
// pass, run for all experts at once: a pass histograms its digit of the keys that still match the
// expert's prefix (in shared memory, merged into one global histogram per expert), and the last
// CTA of a column chunk to finish picks the bucket in which the k-th key lies.  An expert leaves
// the passes as soon as that bucket is small: either it holds exactly the keys still wanted, or at
// most kCandCap keys, the candidates, from which the final sort picks the best.  With distinct
// scores that is after two passes over S.  Experts still undecided after the three score passes
// have more than kCandCap exactly equal scores at the threshold: there the lowest tokens win, and
// one CTA per such expert walks the column in token order and takes the first ones.  One more pass
// over S then copies the winners (and candidates) out, and a bitonic network sorts each expert's keys.
//
// scratch, with C = groups * E columns: [SelState C][hist C*1024 u32][counters passes*groups*chunks u32]
//          [cursors 2C u32] (zeroed per call) [candidates C*kCandCap u64][keys C*kpad u64]
// ------------------------------------------------------------------------------------------
constexpr int kHistThreads = 1024;
constexpr int kBins = 1 << kRadixBits;
constexpr int kHistSmemBytes = (kBins + kBins / 32) * kTopkChunk * 4;   // [bin][column of the chunk]; the selection step re-uses it padded
constexpr unsigned long long kKeyTop = 3ull << 62;              // the two always-set top bits of a key

constexpr unsigned kScoreTop = 0xC0000000u;                     // the same two bits of ~bits(S)
// What the selection orders by: ~bits(S) of a score, the largest one's place for anything else.  (The key of a winner keeps
// the value's own bits.)
__device__ __forceinline__ unsigned sel_bits(unsigned inverted) { return max(inverted, kScoreTop); }
__device__ __forceinline__ unsigned sel_bits(float s) { return sel_bits(~__float_as_uint(s)); }

__device__ __forceinline__ unsigned long long make_key(float s, int64_t t) {
  return ((unsigned long long)(~__float_as_uint(s)) << 32) | (unsigned long long)(unsigned)t;
}

struct TopkLayout {
  size_t off_state, off_hist, off_counters, off_cursor, off_cand, off_keys, zero_bytes, total;
  int chunks; int64_t kpad;
};
// E experts of each of `groups` routing groups: groups * E independent columns ("virtual experts", group-major)
static TopkLayout topk_layout(int64_t n, int E, int64_t k, int groups) {
  TopkLayout L;
  L.chunks = (E + kTopkChunk - 1) / kTopkChunk;
  const size_t VE = (size_t)groups * E;
  L.kpad = 1; while (L.kpad < k) L.kpad <<= 1;
  size_t o = 0;
  auto take = [&](size_t b) { size_t r = o; o += (b + 255) & ~(size_t)255; return r; };
  L.off_state = take(sizeof(SelState) * VE);
  L.off_hist = take(VE * kBins * 4);
  L.off_counters = take((size_t)kRadixPasses * groups * L.chunks * 4);
  L.off_cursor = take(2 * VE * 4);
  L.zero_bytes = o;                       // everything up to here starts at zero
  L.off_cand = take(VE * kCandCap * 8);
  L.off_keys = take(VE * L.kpad * 8);
  L.total = o;
  return L;
}
size_t topk_scratch_bytes(int64_t n, int E, int64_t k, int groups) { return topk_layout(n, E, k, groups).total; }

__device__ __forceinline__ int pow2_at_least(int v) { int p = 1; while (p < v) p <<= 1; return p; }

// Walks the [t0, t1) x [c0, c0 + cw) slab of S with every thread of the CTA.  A thread always sees the same
// columns (four consecutive ones with VEC, one without): slab_first_col() tells it which, or -1 for none,
// and f(score, token, j) gets the j-th of them, j a compile-time 0..3, so per-column state can sit in
// registers.  VEC: 16-byte loads (E a multiple of 4), else scalar.  Four independent loads per thread
// are in flight.
template <bool VEC>
__device__ __forceinline__ int slab_first_col(int cw) {
  const int lane = threadIdx.x & 31;
  if constexpr (VEC) { const int lpr = pow2_at_least((cw + 3) >> 2); const int g = (lane % lpr) * 4; return g < cw ? g : -1; }
  else { const int cwp = pow2_at_least(cw); const int cc = lane % cwp; return cc < cw ? cc : -1; }
}
template <bool VEC, typename F>
__device__ __forceinline__ void for_slab(const float* __restrict__ S, int E, int c0, int cw, int64_t t0, int64_t t1, F&& f) {
  const int warp = threadIdx.x >> 5, lane = threadIdx.x & 31, nwarps = blockDim.x >> 5;
  constexpr int U = 4;
  if constexpr (VEC) {
    const int lpr = pow2_at_least((cw + 3) >> 2), rpw = 32 / lpr;      // lanes per row, rows per warp
    const int r = lane / lpr, g = (lane % lpr) * 4;
    if (g >= cw) return;
    const int64_t step = (int64_t)nwarps * rpw;
    for (int64_t t = t0 + warp * rpw + r; t < t1; t += step * U) {
      float4 v[U];
#pragma unroll
      for (int u = 0; u < U; ++u)
        if (t + u * step < t1) v[u] = *reinterpret_cast<const float4*>(S + (t + u * step) * E + c0 + g);
#pragma unroll
      for (int u = 0; u < U; ++u)
        if (t + u * step < t1) {
          const int64_t tt = t + u * step;
          f(v[u].x, tt, 0); f(v[u].y, tt, 1); f(v[u].z, tt, 2); f(v[u].w, tt, 3);
        }
    }
  } else {
    const int cwp = pow2_at_least(cw), rpw = 32 / cwp;
    const int r = lane / cwp, cc = lane % cwp;
    if (cc >= cw) return;
    const int64_t step = (int64_t)nwarps * rpw;
    for (int64_t t = t0 + warp * rpw + r; t < t1; t += step * U) {
      float v[U];
#pragma unroll
      for (int u = 0; u < U; ++u)
        if (t + u * step < t1) v[u] = S[(t + u * step) * E + c0 + cc];
#pragma unroll
      for (int u = 0; u < U; ++u)
        if (t + u * step < t1) f(v[u], t + u * step, 0);
    }
  }
}

template <bool VEC>
__global__ void __launch_bounds__(kHistThreads, 1)
topk_hist_kernel(const float* __restrict__ S, int64_t n, int E, unsigned k, int pass, int rows_per_cta,
                 SelState* state, unsigned* hist, unsigned* counters) {
  chain_enter();
  S = after_enter(S);
  extern __shared__ unsigned sh[];                     // [bin][column]
  __shared__ unsigned long long s_prefix[kTopkChunk];
  __shared__ int s_active[kTopkChunk];
  __shared__ int s_any, s_last;
  const int tid = threadIdx.x, chunk = blockIdx.y, nchunks = gridDim.y, grp = blockIdx.z;
  const int c0 = chunk * kTopkChunk, cw = min(kTopkChunk, E - c0);
  S += (size_t)grp * n * E;                            // this group's n rows; its experts' state, histograms
  state += (size_t)grp * E; hist += (size_t)grp * E * kBins; counters += (size_t)grp * kRadixPasses * nchunks;
  if (tid == 0) s_any = 0;
  __syncthreads();
  if (tid < kTopkChunk) {
    int act = 0; unsigned long long pre = 0;
    if (tid < cw) {
      if (pass == 0) act = 1;
      else { act = state[c0 + tid].mode == 0 ? 1 : 0; pre = state[c0 + tid].prefix; }
    }
    s_active[tid] = act; s_prefix[tid] = pre;
    if (act) s_any = 1;
  }
  for (int i = tid; i < kBins * kTopkChunk; i += kHistThreads) sh[i] = 0;
  __syncthreads();
  if (!s_any) return;                                  // uniform: every expert of the chunk is decided
  const int shift = 52 - kRadixBits * pass;            // score bits 29..20, 19..10, 9..0
  const int64_t t0 = (int64_t)blockIdx.x * rows_per_cta;
  const int64_t t1 = min(n, t0 + rows_per_cta);
  {
    // only the score half of the key matters here: v = sel_bits(S), digit (v >> sh32) & 1023, and from the
    // second pass on the bits above the digit have to equal the expert's prefix
    constexpr int NC = VEC ? 4 : 1;
    const int col0 = slab_first_col<VEC>(cw), sh32 = shift - 32;
    bool act[NC]; unsigned want[NC];
#pragma unroll
    for (int j = 0; j < NC; ++j) {
      act[j] = col0 >= 0 && col0 + j < cw && s_active[col0 + j];
      want[j] = act[j] ? (unsigned)(s_prefix[col0 + j] >> 32) >> (sh32 + kRadixBits) : 0u;
    }
    for_slab<VEC>(S, E, c0, cw, t0, t1, [&](float s, int64_t, int j) {
      const unsigned v = sel_bits(s);
      if (act[j] && (pass == 0 || (v >> (sh32 + kRadixBits)) == want[j]))
        atomicAdd(&sh[((v >> sh32) & (kBins - 1)) * kTopkChunk + col0 + j], 1u);
    });
  }
  __syncthreads();
  for (int i = tid; i < kBins * kTopkChunk; i += kHistThreads) {
    const unsigned v = sh[i];
    if (v) atomicAdd(&hist[(size_t)(c0 + i % kTopkChunk) * kBins + i / kTopkChunk], v);
  }
  __threadfence();
  __syncthreads();
  if (tid == 0) s_last = atomicAdd(&counters[pass * nchunks + chunk], 1u) == gridDim.x - 1;
  __syncthreads();
  if (!s_last) return;
  __threadfence();
  // The last CTA of this chunk sees the full histograms: one warp per expert finds the bucket of the
  // k-th key, records the decision and leaves the histogram zeroed for the next pass.
  const int warp = tid >> 5, lane = tid & 31;
  if (warp >= cw || !s_active[warp]) return;
  // The expert's kBins counts come in with coalesced, independent loads (lane holds bins lane, 32 + lane, ...),
  // are laid out in the CTA's shared histogram (free by now; one padding word per 32 keeps the banks
  // apart) and are read back as 32 consecutive bins per lane.
  unsigned* h = hist + (size_t)(c0 + warp) * kBins;
  constexpr int PER = kBins / 32;
  unsigned* col = sh + warp * (kBins + PER);
  {
    unsigned tmp[PER];
#pragma unroll
    for (int j = 0; j < PER; ++j) tmp[j] = __ldcg(h + j * 32 + lane);
#pragma unroll
    for (int j = 0; j < PER; ++j) { h[j * 32 + lane] = 0; col[j * 33 + lane] = tmp[j]; }
  }
  __syncwarp();
  unsigned lsum = 0;
#pragma unroll
  for (int j = 0; j < PER; ++j) lsum += col[lane * 33 + j];
  unsigned incl = lsum;
  for (int o = 1; o < 32; o <<= 1) { const unsigned v = __shfl_up_sync(0xffffffffu, incl, o); if (lane >= o) incl += v; }
  const unsigned excl = incl - lsum;
  const unsigned k_rem = pass == 0 ? k : state[c0 + warp].k_rem;
  if (excl < k_rem && k_rem <= incl) {                 // exactly one lane
    unsigned before = excl, in_bucket = 0; int D = 0;
    for (int j = 0; j < PER; ++j) {
      const unsigned c = col[lane * 33 + j];
      if (k_rem <= before + c) { D = j; in_bucket = c; break; }
      before += c;
    }
    const unsigned new_rem = k_rem - before;
    SelState ns;
    ns.prefix = (pass == 0 ? kKeyTop : s_prefix[warp]) | ((unsigned long long)(lane * PER + D) << shift);
    ns.shift = (unsigned)shift; ns.k_rem = new_rem; ns.cand = 0;
    if (in_bucket == new_rem) ns.mode = 1;                             // the whole bucket is taken
    else if (in_bucket <= (unsigned)kCandCap) { ns.mode = 2; ns.cand = in_bucket; }   // the sort picks new_rem of these
    else ns.mode = 0;                                                  // descend one more digit
    state[c0 + warp] = ns;
  }
}

// Experts undecided after the score passes: more than kCandCap keys share the threshold score exactly,
// and the k_rem lowest tokens among them win.  One CTA per expert walks the column in token order.
__global__ void __launch_bounds__(1024)
topk_ties_kernel(const float* __restrict__ S, int64_t n, int E, unsigned k, int64_t kpad, SelState* state,
                 unsigned long long* keys) {
  chain_enter();
  S = after_enter(S);
  __shared__ unsigned s_warp[32];
  __shared__ unsigned s_total;
  const int e = blockIdx.x, grp = blockIdx.y, tid = threadIdx.x, warp = tid >> 5, lane = tid & 31;
  S += (size_t)grp * n * E; state += (size_t)grp * E; keys += (size_t)grp * E * kpad;
  if (state[e].mode != 0) return;
  const unsigned thr = (unsigned)(state[e].prefix >> 32), k_rem = state[e].k_rem, k_def = k - k_rem;
  unsigned running = 0;
  for (int64_t base = 0; base < n && running < k_rem; base += 1024) {
    const int64_t t = base + tid;
    float s = 0.f; bool m = false;
    if (t < n) { s = S[t * E + e]; m = sel_bits(s) == thr; }
    const unsigned bal = __ballot_sync(0xffffffffu, m);
    if (lane == 0) s_warp[warp] = __popc(bal);
    __syncthreads();
    if (warp == 0) {
      const unsigned v = s_warp[lane];
      unsigned inc = v;
      for (int o = 1; o < 32; o <<= 1) { const unsigned u = __shfl_up_sync(0xffffffffu, inc, o); if (lane >= o) inc += u; }
      s_warp[lane] = inc - v;
      if (lane == 31) s_total = inc;
    }
    __syncthreads();
    const unsigned idx = running + s_warp[warp] + __popc(bal & ((1u << lane) - 1u));
    if (m && idx < k_rem) keys[(size_t)e * kpad + k_def + idx] = make_key(s, t);
    running += s_total;
    __syncthreads();
  }
  if (tid == 0) state[e].mode = 3;
}

// Copies each expert's winners to keys[i][0 ..) and its candidates to cand[i][0 ..), in no particular
// order, with one read of S: a CTA parks what it finds in shared memory, reserves one range per
// (expert, kind) with a single global atomic each and writes the keys out.  What does not fit in the
// buffer (only with very uneven inputs) takes its place with a global atomic of its own.
constexpr int kCompactCap = 4096;
template <bool VEC>
__global__ void __launch_bounds__(kHistThreads)
topk_compact_kernel(const float* __restrict__ S, int64_t n, int E, unsigned k, int64_t kpad, int rows_per_cta,
                    const SelState* __restrict__ state, unsigned* cursor, unsigned long long* keys,
                    unsigned long long* cand) {
  chain_enter();
  S = after_enter(S); state = after_enter(state);
  __shared__ unsigned long long s_key[kCompactCap];
  __shared__ unsigned char s_tag[kCompactCap];         // column within the chunk, bit 7: candidate
  __shared__ unsigned s_cnt[2][kTopkChunk], s_base[2][kTopkChunk], s_n;
  __shared__ unsigned long long s_thr[kTopkChunk];
  __shared__ unsigned s_shift[kTopkChunk], s_mode[kTopkChunk];
  const int tid = threadIdx.x, chunk = blockIdx.y, grp = blockIdx.z, groups = gridDim.z;
  const int c0 = chunk * kTopkChunk, cw = min(kTopkChunk, E - c0);
  S += (size_t)grp * n * E; state += (size_t)grp * E;
  keys += (size_t)grp * E * kpad; cand += (size_t)grp * E * kCandCap;
  unsigned* cursor_w = cursor + (size_t)grp * E;                       // winners; candidates follow all groups' winners
  unsigned* cursor_c = cursor + (size_t)groups * E + (size_t)grp * E;
  if (tid == 0) s_n = 0;
  if (tid < kTopkChunk) {
    s_cnt[0][tid] = s_cnt[1][tid] = 0;
    if (tid < cw) {
      const SelState st = state[c0 + tid];
      s_shift[tid] = st.shift; s_thr[tid] = st.prefix >> st.shift; s_mode[tid] = st.mode;
    }
  }
  __syncthreads();
  const int64_t t0 = (int64_t)blockIdx.x * rows_per_cta;
  const int64_t t1 = min(n, t0 + rows_per_cta);
  auto put = [&](int kind, int col, unsigned pos, unsigned long long key) {      // kind 0: winner, 1: candidate
    if (kind == 0) { if (pos < k) keys[(size_t)(c0 + col) * kpad + pos] = key; }
    else if (pos < (unsigned)kCandCap) cand[(size_t)(c0 + col) * kCandCap + pos] = key;
  };
  // per column of this thread: the decided score bits (thr, after dropping the low bits of sel_bits(S) that
  // are still open) and what happens to a key exactly at the threshold: 0 winner, 1 candidate, 2 nothing
  // (the tie walk has placed it)
  constexpr int NC = VEC ? 4 : 1;
  const int col0 = slab_first_col<VEC>(cw);
  unsigned thr[NC], drop[NC]; int at_thr[NC];
#pragma unroll
  for (int j = 0; j < NC; ++j) {
    const bool ok = col0 >= 0 && col0 + j < cw;
    drop[j] = ok ? s_shift[col0 + j] - 32 : 0; thr[j] = ok ? (unsigned)s_thr[col0 + j] : 0u;
    at_thr[j] = !ok ? 2 : (s_mode[col0 + j] == 1 ? 0 : (s_mode[col0 + j] == 2 ? 1 : 2));
  }
  for_slab<VEC>(S, E, c0, cw, t0, t1, [&](float s, int64_t t, int j) {
    const unsigned hi = sel_bits(s) >> drop[j];
    if (hi > thr[j]) return;
    const int kind = hi < thr[j] ? 0 : at_thr[j];
    if (kind == 2) return;
    const int col = col0 + j;
    const unsigned long long key = make_key(s, t);
    const unsigned idx = atomicAdd(&s_n, 1u);
    if (idx < (unsigned)kCompactCap) { s_key[idx] = key; s_tag[idx] = (unsigned char)(col | (kind << 7)); }
    else put(kind, col, atomicAdd(&(kind ? cursor_c : cursor_w)[c0 + col], 1u), key);
  });
  __syncthreads();
  const int held = (int)min(s_n, (unsigned)kCompactCap);
  for (int i = tid; i < held; i += kHistThreads) atomicAdd(&s_cnt[s_tag[i] >> 7][s_tag[i] & 127], 1u);
  __syncthreads();
  if (tid < 2 * kTopkChunk) {
    const int w = tid / kTopkChunk, col = tid % kTopkChunk;
    if (col < cw) { const unsigned c = s_cnt[w][col]; s_base[w][col] = c ? atomicAdd(&(w ? cursor_c : cursor_w)[c0 + col], c) : 0u; }
  }
  __syncthreads();
  if (tid < kTopkChunk) s_cnt[0][tid] = s_cnt[1][tid] = 0;
  __syncthreads();
  for (int i = tid; i < held; i += kHistThreads) {
    const int kind = s_tag[i] >> 7, col = s_tag[i] & 127;
    put(kind, col, s_base[kind][col] + atomicAdd(&s_cnt[kind][col], 1u), s_key[i]);
  }
}

// Slot j of virtual expert ve = group * E + expert lands in row `expert` of I and G (each groups * k long) at
// position group * k + j, and the token index becomes global (group * n + token within the group).
struct SlotMap { int E, groups; int64_t k, n; SlotMarks marks; };
__device__ __forceinline__ void mark_slot(const SlotMarks& m, int64_t token, int e) {
  if (m.per_token > 0) atomicOr(m.words + token * m.per_token + (e >> 5), 1u << (e & 31));
  else atomicAdd(m.words + token, 1u);
}
__device__ __forceinline__ void emit_slot(unsigned long long key, int32_t* I, float* G, const SlotMap& m, int64_t ve, int64_t j) {
  const int64_t grp = ve / m.E, e = ve % m.E;
  const int64_t o = (e * m.groups + grp) * m.k + j;
  const unsigned t = (unsigned)(key & 0xFFFFFFFFull) + (unsigned)(grp * m.n);
  I[o] = (int32_t)t;
  G[o] = __uint_as_float(~(unsigned)(key >> 32));
  mark_slot(m.marks, t, (int)e);
}

// Bitonic sorting of keys in shared memory by the whole CTA.  The steps whose stride spans a warp's keys work on shared memory
// with a barrier each; all shorter ones run in registers, a thread holding PER consecutive keys, over shuffles: 14 barriers
// instead of 45 for 512 keys (10.8 k -> 6.1 k cycles), 20 instead of 78 for 4096 (70 k -> 36 k).  `base` is the
// position of a[0] in the sequence that is sorted: a pair's direction is a bit of its position.
template <int PER>
__device__ __forceinline__ void sort_in_regs(unsigned long long (&v)[PER], unsigned pos, unsigned size, unsigned stride) {
#pragma unroll 1
  for (; stride >= PER; stride >>= 1) {               // partner in another lane
#pragma unroll
    for (int r = 0; r < PER; ++r) {
      const unsigned long long o = __shfl_xor_sync(0xffffffffu, v[r], stride / PER);
      const bool low = (pos & stride) == 0, asc = ((pos + r) & size) == 0;      // stride >= PER: the same for all r; so is asc unless size is PER
      v[r] = (v[r] < o) == (low == asc) ? v[r] : o;
    }
  }
#pragma unroll
  for (int st = PER / 2; st >= 1; st >>= 1) {         // partner in this thread
    if ((unsigned)st <= stride) {
#pragma unroll
      for (int r = 0; r < PER; ++r) {
        if ((r & st) == 0) {
          const bool asc = ((pos + r) & size) == 0;
          const unsigned long long x = v[r], y = v[r + st];
          if ((x > y) == asc) { v[r] = y; v[r + st] = x; }
        }
      }
    }
  }
}
// The steps of one network size on len keys (len a power of two, at least 32 * PER, at most PER * blockDim.x): strides
// min(size, len) / 2 down to 1.
template <int PER>
__device__ __forceinline__ void sort_one_size(unsigned long long* a, int len, unsigned base, unsigned size) {
  const unsigned tid = threadIdx.x;
  unsigned stride = min(size, (unsigned)len) >> 1;
  for (; stride >= 32 * PER; stride >>= 1) {
    for (unsigned p = tid; p < (unsigned)len >> 1; p += blockDim.x) {
      const unsigned i = ((p & ~(stride - 1)) << 1) | (p & (stride - 1)), j = i + stride;       // stride is a power of two
      const bool asc = ((base + i) & size) == 0;
      const unsigned long long x = a[i], y = a[j];
      if ((x > y) == asc) { a[i] = y; a[j] = x; }
    }
    __syncthreads();
  }
  if (tid * PER < (unsigned)len) {                    // whole warps
    unsigned long long v[PER];
#pragma unroll
    for (int r = 0; r < PER; ++r) v[r] = a[tid * PER + r];
    sort_in_regs<PER>(v, base + tid * PER, size, stride);
#pragma unroll
    for (int r = 0; r < PER; ++r) a[tid * PER + r] = v[r];
  }
  __syncthreads();
}
// All sizes up to size_hi (at least 2).  The caller's writes to a[] are behind a barrier; so are this function's.
template <int PER>
__device__ __forceinline__ void sort_keys_per(unsigned long long* a, int len, unsigned base, unsigned size_hi) {
  const unsigned tid = threadIdx.x;
  if (tid * PER < (unsigned)len) {
    unsigned long long v[PER];
#pragma unroll
    for (int r = 0; r < PER; ++r) v[r] = a[tid * PER + r];
#pragma unroll 1
    for (unsigned size = 2; size <= min(size_hi, 32u * PER); size <<= 1) sort_in_regs<PER>(v, base + tid * PER, size, size >> 1);
#pragma unroll
    for (int r = 0; r < PER; ++r) a[tid * PER + r] = v[r];
  }
  __syncthreads();
  for (unsigned size = 64 * PER; size <= size_hi; size <<= 1) sort_one_size<PER>(a, len, base, size);
}
// len: a power of two from 32 to 4 * blockDim.x, blockDim.x a power of two
__device__ __forceinline__ void sort_keys(unsigned long long* a, int len, unsigned base, unsigned size_hi) {
  if (len <= (int)blockDim.x) sort_keys_per<1>(a, len, base, size_hi);
  else if (len <= 2 * (int)blockDim.x) sort_keys_per<2>(a, len, base, size_hi);
  else sort_keys_per<4>(a, len, base, size_hi);
}

// Sorts an expert's candidates and returns (in shared memory) them in ascending order; sc holds kCandCap keys.
__device__ __forceinline__ void load_sorted_candidates(const unsigned long long* cand, int e, unsigned ncand,
                                                       unsigned long long* sc) {
  const int len = max(32, pow2_at_least((int)ncand));
  for (int i = threadIdx.x; i < len; i += blockDim.x) sc[i] = i < (int)ncand ? cand[(size_t)e * kCandCap + i] : ~0ull;
  __syncthreads();
  sort_keys(sc, len, 0, len);
}

// k up to one tile: one CTA per expert merges the candidates in, sorts the k keys and writes I and G.
constexpr int kSortThreads = 1024;
__global__ void __launch_bounds__(kSortThreads)
topk_finish_tile_kernel(const unsigned long long* __restrict__ keys, const unsigned long long* __restrict__ cand,
                        const SelState* __restrict__ state, int64_t kpad, int64_t k, SlotMap map, int32_t* I, float* G) {
  chain_enter();
  keys = after_enter(keys); cand = after_enter(cand); state = after_enter(state);
  __shared__ unsigned long long sk[kSortTile];
  __shared__ unsigned long long sc[kCandCap];
  const int e = blockIdx.x;
  const SelState st = state[e];
  const int len = max(32, (int)kpad);
  for (int i = threadIdx.x; i < len; i += kSortThreads) sk[i] = i < k ? keys[(size_t)e * kpad + i] : ~0ull;      // padding sorts last
  __syncthreads();
  if (st.mode == 2) {
    load_sorted_candidates(cand, e, st.cand, sc);
    const unsigned k_def = (unsigned)k - st.k_rem;
    for (int i = threadIdx.x; i < (int)st.k_rem; i += kSortThreads) sk[k_def + i] = sc[i];
    __syncthreads();
  }
  sort_keys(sk, len, 0, len);
  for (int i = threadIdx.x; i < k; i += kSortThreads) emit_slot(sk[i], I, G, map, e, i);
}

// k beyond one tile: the candidates are merged into the global key list first.
__global__ void __launch_bounds__(kSortThreads)
topk_resolve_kernel(unsigned long long* keys, const unsigned long long* __restrict__ cand,
                    const SelState* __restrict__ state, int64_t kpad, int64_t k) {
  chain_enter();
  cand = after_enter(cand); state = after_enter(state);
  __shared__ unsigned long long sc[kCandCap];
  const int e = blockIdx.x;
  const SelState st = state[e];
  if (st.mode != 2) return;
  load_sorted_candidates(cand, e, st.cand, sc);
  const unsigned k_def = (unsigned)k - st.k_rem;
  for (int i = threadIdx.x; i < (int)st.k_rem; i += kSortThreads) keys[(size_t)e * kpad + k_def + i] = sc[i];
}

// Bitonic steps on one tile of kSortTile keys held in shared memory: the network sizes 2 .. size_hi (size_lo = 2), or
// of the one size size_lo = size_hi beyond the tile the strides that fit.
__global__ void __launch_bounds__(kSortThreads)
topk_sort_tile_kernel(unsigned long long* keys, int64_t kpad, int64_t k, int64_t size_lo, int64_t size_hi,
                      int emit, SlotMap map, int32_t* I, float* G) {
  chain_enter();
  __shared__ unsigned long long sk[kSortTile];
  const int64_t tiles_per_expert = (kpad + kSortTile - 1) / kSortTile;
  const int64_t expert = blockIdx.x / tiles_per_expert;
  const int64_t base = (blockIdx.x % tiles_per_expert) * kSortTile;   // index inside the expert
  const int len = (int)min((int64_t)kSortTile, kpad - base);          // power of two
  unsigned long long* src = keys + expert * kpad + base;
  for (int i = threadIdx.x; i < len; i += kSortThreads) sk[i] = size_lo > 2 || base + i < k ? src[i] : ~0ull;    // padding sorts last
  __syncthreads();
  if (size_lo == 2) sort_keys(sk, len, (unsigned)base, (unsigned)size_hi);
  else sort_one_size<kSortTile / kSortThreads>(sk, len, (unsigned)base, (unsigned)size_lo);
  if (emit) {
    for (int i = threadIdx.x; i < len; i += kSortThreads)
      if (base + i < k) emit_slot(sk[i], I, G, map, expert, base + i);
  } else {
    for (int i = threadIdx.x; i < len; i += kSortThreads) src[i] = sk[i];
  }
}

// One compare-exchange step at a stride that spans tiles.
__global__ void topk_sort_global_kernel(unsigned long long* keys, int64_t kpad, int64_t total_pairs,
                                        int64_t size, int64_t stride) {
  chain_enter();
  for (int64_t p = (int64_t)blockIdx.x * blockDim.x + threadIdx.x; p < total_pairs;
       p += (int64_t)gridDim.x * blockDim.x) {
    const int64_t expert = p / (kpad >> 1), q = p % (kpad >> 1);
    const int64_t i = ((q & ~(stride - 1)) << 1) | (q & (stride - 1)), j = i + stride;       // stride is a power of two
    unsigned long long* kk = keys + expert * kpad;
    const bool asc = (i & size) == 0;
    const unsigned long long a = kk[i], b = kk[j];
    if ((a > b) == asc) { kk[i] = b; kk[j] = a; }
  }
}

// Exclusive scan of the CTA's per-thread values (any thread count that is a multiple of 32, at most 1024);
// returns the thread's offset and, in `total`, the sum over the CTA.
__device__ __forceinline__ int block_exclusive_scan(int v, int* s_warp, int& total) {
  const int lane = threadIdx.x & 31, warp = threadIdx.x >> 5, nwarps = blockDim.x >> 5;
  int inc = v;
  for (int o = 1; o < 32; o <<= 1) { const int u = __shfl_up_sync(0xffffffffu, inc, o); if (lane >= o) inc += u; }
  if (lane == 31) s_warp[warp] = inc;
  __syncthreads();
  if (warp == 0) {
    const int w = lane < nwarps ? s_warp[lane] : 0;
    int winc = w;
    for (int o = 1; o < 32; o <<= 1) { const int u = __shfl_up_sync(0xffffffffu, winc, o); if (lane >= o) winc += u; }
    s_warp[lane] = winc - w;
    if (lane == 31) s_warp[32] = winc;
  }
  __syncthreads();
  total = s_warp[32];
  return s_warp[warp] + inc - v;
}

// The token -> slot index by one CTA, from the marks: the lists' lengths are numbers of bits, a scan gives their starts, and a
// slot's place in its token's list is the number of experts below its own that took the token.  No atomics, no sorting.  Marks,
// starts and lists lie in shared memory (index_smem_bytes): what goes to a token's place in global memory costs an SM a cycle
// per word, and one CTA has all of it to do.  A thread has eight slots in flight.  What other CTAs wrote is read past L1.
__host__ __device__ __forceinline__ int64_t index_smem_words(int64_t N, int64_t total, int W) { return N * W + N + total; }
__device__ __forceinline__ void build_index(const int32_t* I, int N, int total, int k_row, const SlotMarks& m, int32_t* row_ptr,
                                            int32_t* slots, int* smem, int* s_warp, int* status) {
  const int tid = threadIdx.x, nt = blockDim.x, W = m.per_token;
  unsigned* marks = reinterpret_cast<unsigned*>(smem);                 // [N][W]
  int *start = smem + N * W, *list = start + N;                        // [N], [total]
  for (int i0 = tid; i0 < N * W; i0 += 8 * nt) {
    unsigned v[8];
#pragma unroll
    for (int u = 0; u < 8; ++u) v[u] = i0 + u * nt < N * W ? __ldcg(m.words + i0 + u * nt) : 0u;
#pragma unroll
    for (int u = 0; u < 8; ++u) if (i0 + u * nt < N * W) marks[i0 + u * nt] = v[u];
  }
  __syncthreads();
  const int per = (N + nt - 1) / nt, a = min(N, tid * per), b = min(N, a + per);
  int sum = 0;
  for (int i = a * W; i < b * W; ++i) sum += __popc(marks[i]);
  int filled;
  int run = block_exclusive_scan(sum, s_warp, filled);
  for (int t = a; t < b; ++t) {
    start[t] = run;
    for (int w = 0; w < W; ++w) run += __popc(marks[t * W + w]);
  }
  __syncthreads();
  for (int t = tid; t < N; t += nt) row_ptr[t] = start[t];
  if (tid == 0) row_ptr[N] = filled;
  for (int s0 = tid; s0 < total; s0 += 8 * nt) {
    int t[8];
#pragma unroll
    for (int u = 0; u < 8; ++u) t[u] = s0 + u * nt < total ? __ldcg(I + s0 + u * nt) : -1;     // -1: an empty slot (token-choice routing only), or none
#pragma unroll
    for (int u = 0; u < 8; ++u) {
      if (t[u] < 0 || !idx_ok(t[u], 0, N, status)) continue;
      const int e = (s0 + u * nt) / k_row;
      int at = start[t[u]] + __popc(marks[t[u] * W + (e >> 5)] & ((1u << (e & 31)) - 1u));
      for (int w = 0; w < e >> 5; ++w) at += __popc(marks[t[u] * W + w]);
      list[at] = s0 + u * nt;
    }
  }
  __syncthreads();
  for (int s = tid; s < filled; s += nt) slots[s] = list[s];
}

// Small groups (n <= kSmallN tokens, k <= kSortTile): the whole selection of one expert in one CTA.  The
// column is brought into shared memory once (as v = ~bits(S)), three 10-bit histogram passes over it find
// the value of the k-th key exactly, keys below it are winners, keys equal to it win in token order, and the
// k keys are sorted and written out: one launch instead of eight, for the sizes where launches are what costs.
// A CTA per expert leaves most SMs idle, so a CTA's own latency is what counts: about four keys per thread, eight loads of
// a thread in flight, every thread takes part in a pass's scan, and the walk in token order is taken only when
// not all keys at the threshold are wanted.  2048 tokens, k = 512: 33.5 k cycles before that, 17 k now.
// With row_ptr, the last CTA to finish also builds the token -> slot index (build_index; `done` counts the CTAs).
// CLUSTER: a column alone costs a CTA a request per token, of which it uses 4 of 32 bytes (8192 tokens: 10.5 k cycles, 16384:
// 33 k; with the third pass, which is hardly ever needed, 24.5 us at 8192 tokens and 32 experts, 22.5 now).  The CTAs of eight experts form a cluster: each reads an eighth of the tokens, all eight scores of a token together, and sends every
// score to its expert's CTA.
constexpr int kSmallN = 16384;
// INDEX: with row_ptr.  build_index wants 54 registers, the selection alone gets by with 32, so that an SM holds two CTAs of 1024
// threads (PER_SM) and up to 296 columns need no second round.  Clusters share SMs only where they are many: forward passes, one and
// two per SM, of 8192 tokens: 32 experts 57.3 and 60.2 us, 64 161.0 and 166.2, 128 63.3 and 60.0; of 16384: 64 87.7 and 101, 128 108
// and 104, 256 132 and 136; of 6000: 256 88.0 and 83.1.
template <bool CLUSTER, bool INDEX, int PER_SM>
__global__ void __launch_bounds__(1024, PER_SM)
topk_small_kernel(const float* __restrict__ S, int n, int E, int k, int kpad, const SlotMap map, int32_t* I, float* G, int32_t* row_ptr,
                  int32_t* slots, int* done, int* status) {
  if constexpr (CLUSTER) cluster_barrier();            // every CTA of the cluster has started: its shared memory may be written
  chain_enter();
  S = after_enter(S);
  extern __shared__ unsigned long long sm_keys[];      // [kpad] keys (kpad >= 32), then [n] values, then [kBins] histogram
  unsigned* val = reinterpret_cast<unsigned*>(sm_keys + kpad);
  unsigned* hist = val + n;
  __shared__ unsigned s_prefix, s_rem, s_eq, s_less, s_warp[33];
  const int e = blockIdx.x, grp = blockIdx.y, tid = threadIdx.x, lane = tid & 31, warp = tid >> 5;
  const int nt = blockDim.x, nwarps = nt >> 5;         // 128 .. 1024 threads (a power of two), by the size of the group
  if constexpr (CLUSTER) {
    const int rank = e & 7, e0 = e - rank, ne = min(8, E - e0);
    const int per = (n + 7) / 8, t1 = min(n, (rank + 1) * per);
    unsigned dst[8];
#pragma unroll
    for (int j = 0; j < 8; ++j) dst[j] = cluster_address(val, j);
    const bool vec = E % 4 == 0;                       // rows of S are whole 16-byte groups, and so is e0
    for (int t = rank * per + tid; t < t1; t += nt) {
      const float* p = S + ((size_t)grp * n + t) * E + e0;
      float x[8];
      if (vec) {
        const float4 a = *reinterpret_cast<const float4*>(p);
        x[0] = a.x; x[1] = a.y; x[2] = a.z; x[3] = a.w;
        if (ne > 4) { const float4 b = *reinterpret_cast<const float4*>(p + 4); x[4] = b.x; x[5] = b.y; x[6] = b.z; x[7] = b.w; }
      } else {
#pragma unroll
        for (int j = 0; j < 8; ++j) x[j] = j < ne ? p[j] : 0.f;
      }
#pragma unroll
      for (int j = 0; j < 8; ++j)
        if (j < ne) asm volatile("st.shared::cluster.u32 [%0], %1;" ::"r"(dst[j] + 4u * (unsigned)t), "r"(~__float_as_uint(x[j])) : "memory");
    }
    cluster_barrier();
    if (e >= E) return;
  } else {
    const float* col = S + (size_t)grp * n * E + e;
    for (int t0 = tid; t0 < n; t0 += 8 * nt) {
      float x[8];
#pragma unroll
      for (int u = 0; u < 8; ++u) x[u] = col[(size_t)min(t0 + u * nt, n - 1) * E];
#pragma unroll
      for (int u = 0; u < 8; ++u) if (t0 + u * nt < n) val[t0 + u * nt] = ~__float_as_uint(x[u]);
    }
  }
  for (int i = tid; i < kpad; i += nt) sm_keys[i] = ~0ull;
  for (int i = tid; i < kBins; i += nt) hist[i] = 0;
  if (tid == 0) { s_prefix = 0; s_rem = (unsigned)k; s_less = 0; }
  __syncthreads();
  // sel_bits() has its two top bits set; digits of 10 bits from bit 29 down
  const int per = kBins / nt;                          // consecutive bins of a thread in the scan: 1 .. 8
  int sh = 20;
  for (int pass = 0; pass < 3; ++pass) {
    sh = 20 - 10 * pass;
    const unsigned pre = s_prefix, rem = s_rem;
    for (int t = tid; t < n; t += nt) {
      const unsigned v = sel_bits(val[t]);
      if (pass == 0 || (v >> (sh + 10)) == (pre >> (sh + 10))) atomicAdd(&hist[(v >> sh) & (kBins - 1)], 1u);
    }
    __syncthreads();
    // bucket of the rem-th smallest v among the matching ones; the histogram is left zeroed
    unsigned c[8], lsum = 0;
#pragma unroll
    for (int j = 0; j < 8; ++j) {
      c[j] = 0;
      if (j < per) { c[j] = hist[tid * per + j]; hist[tid * per + j] = 0; lsum += c[j]; }
    }
    unsigned incl = lsum;
#pragma unroll
    for (int o = 1; o < 32; o <<= 1) { const unsigned u = __shfl_up_sync(0xffffffffu, incl, o); if (lane >= o) incl += u; }
    if (lane == 31) s_warp[warp] = incl;
    __syncthreads();
    unsigned before = lane < warp ? s_warp[lane] : 0u; // warps in front of this one: at most 31
#pragma unroll
    for (int o = 16; o; o >>= 1) before += __shfl_xor_sync(0xffffffffu, before, o);
    before += incl - lsum;
    if (before < rem && rem <= before + lsum) {        // exactly one thread
      int D = 0; unsigned in = 0; bool found = false;
#pragma unroll
      for (int j = 0; j < 8; ++j) {
        if (!found && j < per) {
          if (rem <= before + c[j]) { D = j; in = c[j]; found = true; } else before += c[j];
        }
      }
      s_prefix = (pass == 0 ? kScoreTop : pre) | ((unsigned)(tid * per + D) << sh);
      s_rem = rem - before;
      s_eq = in;
    }
    __syncthreads();
    if (s_eq == s_rem) break;                          // the whole bucket is wanted: nearly always after 20 of the 30 bits
  }
  const unsigned thr = s_prefix >> sh, k_rem = s_rem, k_less = (unsigned)k - k_rem;      // k_rem keys equal to thr are wanted
  // winners in any order: the keys below the threshold, and those at it when all of them are wanted
  const bool all_eq = s_eq == k_rem;
  for (int t0 = tid - lane; t0 < n; t0 += 4 * nt) {    // uniform across the warp
    unsigned v[4], bal[4], sum = 0;
#pragma unroll
    for (int u = 0; u < 4; ++u) {
      const int t = t0 + u * nt + lane;
      v[u] = t < n ? val[t] : 0xFFFFFFFFu;
      const unsigned sv = sel_bits(v[u]) >> sh;
      bal[u] = __ballot_sync(0xffffffffu, t < n && (sv < thr || (all_eq && sv == thr)));
      sum += __popc(bal[u]);
    }
    if (sum == 0) continue;
    unsigned at = 0;
    if (lane == 0) at = atomicAdd(&s_less, sum);
    at = __shfl_sync(0xffffffffu, at, 0);
#pragma unroll
    for (int u = 0; u < 4; ++u) {
      if (bal[u] >> lane & 1u) sm_keys[at + __popc(bal[u] & ((1u << lane) - 1u))] = ((unsigned long long)v[u] << 32) | (unsigned)(t0 + u * nt + lane);
      at += __popc(bal[u]);
    }
  }
  // else (all 30 bits are decided) the first k_rem keys at the threshold in token order
  unsigned running = 0;
  for (int base = 0; !all_eq && base < n && running < k_rem; base += nt) {
    const int t = base + tid;
    const bool m = t < n && sel_bits(val[t]) == thr;
    const unsigned bal = __ballot_sync(0xffffffffu, m);
    if (lane == 0) s_warp[warp] = __popc(bal);
    __syncthreads();
    if (warp == 0) {
      const unsigned v = lane < nwarps ? s_warp[lane] : 0u;
      unsigned inc = v;
      for (int o = 1; o < 32; o <<= 1) { const unsigned u = __shfl_up_sync(0xffffffffu, inc, o); if (lane >= o) inc += u; }
      s_warp[lane] = inc - v;
      if (lane == 31) s_warp[32] = inc;
    }
    __syncthreads();
    const unsigned idx = running + s_warp[warp] + __popc(bal & ((1u << lane) - 1u));
    if (m && idx < k_rem) sm_keys[k_less + idx] = ((unsigned long long)val[t] << 32) | (unsigned)t;
    running += s_warp[32];
    __syncthreads();
  }
  __syncthreads();
  sort_keys(sm_keys, kpad, 0, (unsigned)kpad);
  for (int i = tid; i < k; i += nt) emit_slot(sm_keys[i], I, G, map, (int64_t)grp * E + e, i);
  if constexpr (INDEX) {
    __threadfence();
    __syncthreads();
    if (tid == 0) s_less = atomicAdd(done, 1) == E * map.groups - 1 ? 1u : 0u;
    __syncthreads();
    if (!s_less) return;
    __threadfence();
    build_index(I, n * map.groups, E * k * map.groups, k * map.groups, map.marks, row_ptr, slots, reinterpret_cast<int*>(sm_keys),
                reinterpret_cast<int*>(s_warp), status);
  }
}

// Dynamic shared memory of a launch: the attribute is one per device, whatever threads launch, so it is always set to the most
// that any call needs, never less than another's
constexpr int kMostSelectSmem = kSortTile * 8 + kSmallN * 4 + kBins * 4;
constexpr int kIndexClusterTokens = 16384, kIndexClusterSlots = 1 << 17;
IndexPlan plan_index(int64_t ng, int E, int64_t k, int groups, bool selects, void* topk_scratch, void* inverse_scratch) {
  const int64_t N = ng * groups, total = (int64_t)E * k * groups;
  const int words = (E + 31) / 32;
  IndexPlan p;
  // The selection's last CTA builds the index where everything fits its shared memory (2048 tokens, 8 experts: 24.5 us with two
  // launches that counted, filled and sorted, 20.5 so), the columns are one round of CTAs (1024 threads each, as the index wants them:
  // sixteen groups of 256 tokens, 64 experts 55.8 us so, 25.6 by a cluster) and a token's marks are two words (2048 tokens, 128
  // experts: 27.2 so, 24.4 by a cluster; 64 experts, two groups: 26.2 either way); else a cluster of eight CTAs, up to 16384 tokens (8192 tokens, 32 experts: 18.4 us with
  // atomics and sorting, 14.4 from the marks; one CTA alone takes 22).  Their marks may take the place of the large selection's
  // scratch, which such a call does not use.
  const bool one_launch = selects && ng <= kSmallN && k <= kSortTile;
  p.fused = one_launch && N <= 4096 && (int64_t)E * groups <= 148 && words <= 2 && index_smem_words(N, total, words) * 4 <= kMostSelectSmem;
  p.small = p.fused || (N <= kIndexClusterTokens && total <= kIndexClusterSlots && (one_launch || !selects));
  p.marks.per_token = p.small || words == 1 ? words : 0;
  p.marks.words = (unsigned*)(p.marks.per_token > 1 ? topk_scratch : inverse_scratch);
  return p;
}

cudaError_t launch_topk(const float* S, int64_t n, int E, int64_t k, int groups, int32_t* I, float* G,
                        const IndexPlan& plan, int32_t* row_ptr, int32_t* slots, void* scratch, int* status, cudaStream_t st) {
  const TopkLayout L = topk_layout(n, E, k, groups);
  if (n <= kSmallN && L.kpad <= kSortTile) {
    const SlotMap smap = {E, groups, k, n, plan.marks};
    const int kpad = L.kpad < 32 ? 32 : (int)L.kpad;   // the sort works on whole warps of keys
    int smem = (int)(kpad * 8 + n * 4 + kBins * 4);
    if (plan.fused) smem = max(smem, (int)index_smem_words(n * groups, (int64_t)E * k * groups, plan.marks.per_token) * 4);
    const bool cluster = n > 4096 && E >= 8;
    auto kern = cluster ? ((int64_t)E * groups > 96 ? topk_small_kernel<true, false, 2> : topk_small_kernel<true, false, 1>)
                        : plan.fused ? topk_small_kernel<false, true, 1> : topk_small_kernel<false, false, 2>;
    cudaError_t e0 = cudaFuncSetAttribute(kern, cudaFuncAttributeMaxDynamicSharedMemorySize, kMostSelectSmem);
    if (e0 != cudaSuccess) return e0;
    int threads = 128;                                 // at most four keys per thread for the sort (kpad < 2 n)
    while (threads < 1024 && threads * 4 < n) threads <<= 1;
    while (threads < 1024 && threads * 4 < kpad) threads <<= 1;
    while (plan.fused && threads < 1024 && threads * 8 < (int64_t)E * k * groups) threads <<= 1;
    return launch_chained_cluster(cluster ? 8 : 1, kern, dim3(cluster ? (E + 7) / 8 * 8 : E, groups), dim3(threads), smem, st, S, (int)n, E, (int)k, kpad, smap, I, G,
                                  row_ptr, slots, status + kSelectCounter, status);
  }
  const int64_t VE = (int64_t)groups * E;              // independent columns: E per group
  char* base = (char*)scratch;
  SelState* state = (SelState*)(base + L.off_state);
  unsigned* hist = (unsigned*)(base + L.off_hist);
  unsigned* counters = (unsigned*)(base + L.off_counters);
  unsigned* cursor = (unsigned*)(base + L.off_cursor);
  unsigned long long* cand = (unsigned long long*)(base + L.off_cand);
  unsigned long long* keys = (unsigned long long*)(base + L.off_keys);
  const SlotMap map = {E, groups, k, n, plan.marks};
  cudaError_t e;
  const bool vec = E % 4 == 0 && ((uintptr_t)S & 15) == 0;
  // the histogram kernels use 132 KiB of dynamic shared memory
  if ((e = vec ? cudaFuncSetAttribute(topk_hist_kernel<true>, cudaFuncAttributeMaxDynamicSharedMemorySize, kHistSmemBytes)
               : cudaFuncSetAttribute(topk_hist_kernel<false>, cudaFuncAttributeMaxDynamicSharedMemorySize, kHistSmemBytes)) != cudaSuccess) return e;
  if ((e = cudaMemsetAsync(base, 0, L.zero_bytes, st)) != cudaSuccess) return e;
  // rows per CTA: one CTA per SM fits (the histogram takes 132 KiB of shared memory), so one wave over all
  // chunks and groups; at least 256 rows each
  int64_t want = (int64_t)148 / ((int64_t)L.chunks * groups); if (want < 1) want = 1;
  int64_t rows = (n + want - 1) / want; if (rows < 256) rows = 256;
  const dim3 grid((unsigned)((n + rows - 1) / rows), (unsigned)L.chunks, (unsigned)groups);
  for (int pass = 0; pass < kRadixPasses; ++pass) {
    if (vec) launch_chained(topk_hist_kernel<true>, grid, dim3(kHistThreads), kHistSmemBytes, st, S, n, E, (unsigned)k, pass, (int)rows, state, hist, counters);
    else launch_chained(topk_hist_kernel<false>, grid, dim3(kHistThreads), kHistSmemBytes, st, S, n, E, (unsigned)k, pass, (int)rows, state, hist, counters);
  }
  launch_chained(topk_ties_kernel, dim3(E, groups), dim3(1024), 0, st, S, n, E, (unsigned)k, L.kpad, state, keys);
  if (vec) launch_chained(topk_compact_kernel<true>, grid, dim3(kHistThreads), 0, st, S, n, E, (unsigned)k, L.kpad, (int)rows, state, cursor, keys, cand);
  else launch_chained(topk_compact_kernel<false>, grid, dim3(kHistThreads), 0, st, S, n, E, (unsigned)k, L.kpad, (int)rows, state, cursor, keys, cand);
  if (L.kpad <= kSortTile) {
    launch_chained(topk_finish_tile_kernel, dim3((unsigned)VE), dim3(kSortThreads), 0, st, keys, cand, state, L.kpad, k, map, I, G);
  } else {
    const int64_t tiles = (L.kpad + kSortTile - 1) / kSortTile;
    const unsigned sort_grid = (unsigned)(VE * tiles);
    launch_chained(topk_resolve_kernel, dim3((unsigned)VE), dim3(kSortThreads), 0, st, keys, cand, state, L.kpad, k);
    launch_chained(topk_sort_tile_kernel, dim3(sort_grid), dim3(kSortThreads), 0, st, keys, L.kpad, k, 2, kSortTile, 0, map, I, G);
    const int64_t pairs = VE * (L.kpad >> 1);
    for (int64_t size = 2 * kSortTile; size <= L.kpad; size <<= 1) {
      for (int64_t stride = size >> 1; stride >= kSortTile; stride >>= 1) {
        launch_chained(topk_sort_global_kernel, dim3(grid_for(pairs, 256)), dim3(256), 0, st, keys, L.kpad, pairs, size, stride);
      }
      launch_chained(topk_sort_tile_kernel, dim3(sort_grid), dim3(kSortThreads), 0, st, keys, L.kpad, k, size, size, size == L.kpad, map, I, G);
    }
  }
  return cudaGetLastError();
}

// ------------------------------------------------------------------------------------------
// Token-choice contrast routing (Section 3.1): every token picks its two best experts, experts have buffers.
// ------------------------------------------------------------------------------------------
// One warp per token row of S: the two largest scores, equal scores to the lower expert.  A score in [0, 1] orders
// like its bit pattern; the key puts the inverted expert index below it so that one max decides both.
__global__ void __launch_bounds__(256) token_top2_kernel(const float* __restrict__ S, int64_t rows, int E, int32_t* __restrict__ choice) {
  chain_enter();
  S = after_enter(S);
  const int lane = threadIdx.x & 31;
  const int64_t warps = ((int64_t)gridDim.x * blockDim.x) >> 5;
  for (int64_t t = ((int64_t)blockIdx.x * blockDim.x + threadIdx.x) >> 5; t < rows; t += warps) {
    unsigned long long best = 0, second = 0;           // 0 is below every real key (the index part of a real key is > 0)
    for (int i = lane; i < E; i += 32) {
      const unsigned long long key = ((unsigned long long)__float_as_uint(S[t * E + i]) << 32) | (0xFFFFFFFFu - (unsigned)i);
      if (key > best) { second = best; best = key; } else if (key > second) second = key;
    }
    unsigned long long top = best;
    for (int o = 16; o; o >>= 1) { const unsigned long long v = __shfl_xor_sync(0xffffffffu, top, o); top = v > top ? v : top; }
    const unsigned long long mine = best == top ? second : best;          // the winner's lane offers its runner-up
    unsigned long long nxt = mine;
    for (int o = 16; o; o >>= 1) { const unsigned long long v = __shfl_xor_sync(0xffffffffu, nxt, o); nxt = v > nxt ? v : nxt; }
    if (lane == 0) {
      choice[2 * t] = (int32_t)(0xFFFFFFFFu - (unsigned)top);
      choice[2 * t + 1] = (int32_t)(0xFFFFFFFFu - (unsigned)nxt);
    }
  }
}

// One CTA per (expert, group) walks the group's tokens in order; a token that chose the expert takes the next slot
// while there is one.  A token's two choices are different experts, so the order of the requests to one expert is
// the token order.  Empty slots get -1 / 0.
__global__ void __launch_bounds__(1024)
token_admit_kernel(const float* __restrict__ S, const int32_t* __restrict__ choice, int n, int E, int k,
                   int32_t* __restrict__ I, float* __restrict__ G, int32_t* __restrict__ load, int32_t* __restrict__ requested, const SlotMarks marks) {
  chain_enter();
  S = after_enter(S); choice = after_enter(choice);
  __shared__ unsigned s_warp[33];
  const int e = blockIdx.x, grp = blockIdx.y, groups = gridDim.y, tid = threadIdx.x, warp = tid >> 5, lane = tid & 31;
  const int64_t row0 = (int64_t)grp * n;
  int32_t* Ie = I + ((int64_t)e * groups + grp) * k;
  float* Ge = G + ((int64_t)e * groups + grp) * k;
  unsigned running = 0;
  for (int base = 0; base < n; base += 1024) {
    const int t = base + tid;
    bool m = false;
    if (t < n) { const int2 c = *reinterpret_cast<const int2*>(choice + 2 * (row0 + t)); m = c.x == e || c.y == e; }
    const unsigned bal = __ballot_sync(0xffffffffu, m);
    if (lane == 0) s_warp[warp] = __popc(bal);
    __syncthreads();
    if (warp == 0) {
      const unsigned v = s_warp[lane];
      unsigned inc = v;
      for (int o = 1; o < 32; o <<= 1) { const unsigned u = __shfl_up_sync(0xffffffffu, inc, o); if (lane >= o) inc += u; }
      s_warp[lane] = inc - v;
      if (lane == 31) s_warp[32] = inc;
    }
    __syncthreads();
    const unsigned pos = running + s_warp[warp] + __popc(bal & ((1u << lane) - 1u));
    if (m && pos < (unsigned)k) { Ie[pos] = (int32_t)(row0 + t); Ge[pos] = S[(row0 + t) * E + e]; mark_slot(marks, row0 + t, e); }
    running += s_warp[32];
    __syncthreads();
  }
  const unsigned filled = running < (unsigned)k ? running : (unsigned)k;
  for (int j = (int)filled + tid; j < k; j += 1024) { Ie[j] = -1; Ge[j] = 0.f; }
  if (tid == 0) { load[grp * E + e] = (int32_t)filled; requested[grp * E + e] = (int32_t)running; }
}

cudaError_t launch_token_top2(const float* S, int64_t rows, int E, int32_t* choice, cudaStream_t st) {
  launch_chained(token_top2_kernel, dim3(grid_for(rows * 32, 256, 148 * 8)), dim3(256), 0, st, S, rows, E, choice);
  return cudaGetLastError();
}

cudaError_t launch_token_admit(const float* S, const int32_t* choice, int64_t n, int E, int64_t k, int groups,
                               int32_t* I, float* G, int32_t* load, int32_t* requested, const SlotMarks& marks, cudaStream_t st) {
  launch_chained(token_admit_kernel, dim3(E, groups), dim3(1024), 0, st, S, choice, (int)n, E, (int)k, I, G, load, requested, marks);
  return cudaGetLastError();
}

// ------------------------------------------------------------------------------------------
// Index form of P = Onehot(I) (Eq. 2) read by token: row_ptr / slots, from I and the marks the selection left (SlotMarks).
// Up to 4096 tokens the selection's last CTA does it (build_index, above), up to 16384 a cluster.  Beyond, a scan of the lists' lengths in two steps, then every slot goes to its place: with up to 32 experts its rank is read from the
// marks; with more (a word per token: the masks would outgrow the scratch) places are handed out by atomics and each token's
// list is sorted, so the result does not depend on the order in which threads ran.
// scratch: [marks n+1 words][tile sums ceil(n / kScanTile) int32]
// ------------------------------------------------------------------------------------------
constexpr int kScanTile = 4096, kScanThreads = 1024;
static size_t inv_cnt_bytes(int64_t n) { return ((size_t)(n + 1) * 4 + 255) & ~(size_t)255; }
size_t inverse_scratch_bytes(int64_t n) {
  return inv_cnt_bytes(n) + ((((size_t)(n + kScanTile - 1) / kScanTile) * 4 + 255) & ~(size_t)255);
}

// Step 1: exclusive scan inside each tile of kScanTile counts (four per thread), tile sums aside.
__global__ void __launch_bounds__(kScanThreads) inv_scan_tile_kernel(const SlotMarks m, int64_t n, int32_t* row_ptr, int32_t* tile_sum) {
  chain_enter();
  __shared__ int s_warp[33];
  const int64_t base = (int64_t)blockIdx.x * kScanTile + threadIdx.x * 4;
  int c[4];
#pragma unroll
  for (int j = 0; j < 4; ++j) { const unsigned v = base + j < n ? m.words[base + j] : 0u; c[j] = m.per_token ? __popc(v) : (int)v; }
  int total;
  int run = block_exclusive_scan(c[0] + c[1] + c[2] + c[3], s_warp, total);
#pragma unroll
  for (int j = 0; j < 4; ++j) { if (base + j < n) row_ptr[base + j] = run; run += c[j]; }
  if (threadIdx.x == 0) tile_sum[blockIdx.x] = total;
}

// Step 2: every tile adds the sum of the tiles before it; the last one also writes row_ptr[n].
__global__ void __launch_bounds__(kScanThreads) inv_scan_add_kernel(const int32_t* __restrict__ tile_sum, int64_t n,
                                                                     int32_t* row_ptr) {
  chain_enter();
  tile_sum = after_enter(tile_sum);
  __shared__ int s_warp[33];
  int part = 0;
  for (int j = threadIdx.x; j < (int)blockIdx.x; j += kScanThreads) part += tile_sum[j];
  int before;
  block_exclusive_scan(part, s_warp, before);
  const int64_t base = (int64_t)blockIdx.x * kScanTile + threadIdx.x * 4;
#pragma unroll
  for (int j = 0; j < 4; ++j) if (base + j < n) row_ptr[base + j] += before;
  if (blockIdx.x == gridDim.x - 1 && threadIdx.x == 0) row_ptr[n] = before + tile_sum[blockIdx.x];
}

// Puts each slot into its token's list: where its rank says, or at a place handed out by counting the token's word down to zero.
__global__ void inv_fill_kernel(const int32_t* __restrict__ I, int64_t total, int64_t k_row, const int32_t* __restrict__ row_ptr,
                                const SlotMarks m, int32_t* slots, int64_t n, int* status) {
  chain_enter();
  I = after_enter(I); row_ptr = after_enter(row_ptr);
  for (int64_t s = (int64_t)blockIdx.x * blockDim.x + threadIdx.x; s < total; s += (int64_t)gridDim.x * blockDim.x) {
    const int t = I[s];                                // -1: an empty slot (token-choice routing only)
    if (t < 0 || !idx_ok(t, 0, n, status)) continue;
    const int at = m.per_token ? __popc(m.words[t] & ((1u << (int)(s / k_row)) - 1u)) : (int)atomicSub(m.words + t, 1u) - 1;
    slots[row_ptr[t] + at] = (int32_t)s;
  }
}

// Sorts one token's list of slots (ascending).  Up to eight entries, which is nearly every token, are brought in together,
// sorted in registers and written back: one round trip to memory where an insertion sort in place takes one per step.
__device__ __forceinline__ void sort_list(int32_t* slots, int lo, int hi) {
  const int len = hi - lo;
  if (len <= 1) return;
  if (len <= 8) {
    int v[8];
#pragma unroll
    for (int i = 0; i < 8; ++i) v[i] = i < len ? slots[lo + i] : 0x7FFFFFFF;
    // odd-even transposition: eight rounds sort eight
#pragma unroll
    for (int r = 0; r < 8; ++r)
#pragma unroll
      for (int i = r & 1; i + 1 < 8; i += 2) {
        const int x = min(v[i], v[i + 1]), y = max(v[i], v[i + 1]);
        v[i] = x; v[i + 1] = y;
      }
#pragma unroll
    for (int i = 0; i < 8; ++i) if (i < len) slots[lo + i] = v[i];
    return;
  }
  for (int i = lo + 1; i < hi; ++i) {
    const int v = slots[i]; int j = i - 1;
    while (j >= lo && slots[j] > v) { slots[j + 1] = slots[j]; --j; }
    slots[j + 1] = v;
  }
}

__global__ void inv_sort_kernel(const int32_t* __restrict__ row_ptr, int64_t n, int32_t* slots) {
  chain_enter();
  row_ptr = after_enter(row_ptr);
  for (int64_t t = (int64_t)blockIdx.x * blockDim.x + threadIdx.x; t < n; t += (int64_t)gridDim.x * blockDim.x) {
    sort_list(slots, row_ptr[t], row_ptr[t + 1]);
  }
}

// Up to kIndexClusterTokens tokens: one cluster of eight CTAs, each an eighth of the tokens in the scan (the eight sums are read from
// the other CTAs' shared memory) and an eighth of the slots in the fill.
__global__ void __launch_bounds__(1024)
index_cluster_kernel(const int32_t* __restrict__ I, int n, int total, int k_row, const SlotMarks m, int32_t* row_ptr, int32_t* slots, int* status) {
  chain_enter();
  I = after_enter(I);
  __shared__ int s_warp[33];
  __shared__ int s_tile;                               // sum of this CTA's part of the counts
  const int tid = threadIdx.x, rank = blockIdx.x, W = m.per_token;     // the grid is the one cluster
  // exclusive scan: CTA `rank` takes tokens [lo, hi), a thread `per` consecutive ones of them (at most two)
  const int per_cta = (n + 7) / 8, lo = min(n, rank * per_cta), hi = min(n, lo + per_cta);
  const int per = (per_cta + 1023) / 1024, a = min(hi, lo + tid * per), b = min(hi, a + per);
  int len[kIndexClusterTokens / 8192], sum = 0;
#pragma unroll
  for (int j = 0; j < kIndexClusterTokens / 8192; ++j) {
    len[j] = 0;
    if (a + j < b) for (int w = 0; w < W; ++w) len[j] += __popc(m.words[(int64_t)(a + j) * W + w]);
    sum += len[j];
  }
  int tile;
  int run = block_exclusive_scan(sum, s_warp, tile);
  if (tid == 0) s_tile = tile;
  cluster_barrier();
  int before = 0;
  for (int r = 0; r < rank; ++r) {
    int v;
    asm volatile("ld.shared::cluster.s32 %0, [%1];" : "=r"(v) : "r"(cluster_address(&s_tile, r)));
    before += v;
  }
  run += before;
#pragma unroll
  for (int j = 0; j < kIndexClusterTokens / 8192; ++j) if (a + j < b) { row_ptr[a + j] = run; run += len[j]; }
  if (rank == 7 && tid == 0) row_ptr[n] = before + tile;
  cluster_barrier();                                   // row_ptr is visible to the cluster, and nobody reads s_tile any more
  for (int s0 = rank * 1024 + tid; s0 < total; s0 += 8 * 8192) {
    int t[8], at[8], e[8];
#pragma unroll
    for (int u = 0; u < 8; ++u) {
      const int s = s0 + u * 8192;
      t[u] = s < total ? I[s] : -1;                    // -1: an empty slot (token-choice routing only), or none
      e[u] = s / k_row;
    }
#pragma unroll
    for (int u = 0; u < 8; ++u) {
      if (t[u] >= 0 && !idx_ok(t[u], 0, n, status)) t[u] = -1;
      at[u] = t[u] >= 0 ? __ldcg(row_ptr + t[u]) : 0;
    }
    for (int w = 0; w < W; ++w) {
#pragma unroll
      for (int u = 0; u < 8; ++u)
        if (t[u] >= 0 && w <= e[u] >> 5) {
          const unsigned bits = m.words[(int64_t)t[u] * W + w];
          at[u] += __popc(w == e[u] >> 5 ? bits & ((1u << (e[u] & 31)) - 1u) : bits);
        }
    }
#pragma unroll
    for (int u = 0; u < 8; ++u) if (t[u] >= 0) slots[at[u]] = s0 + u * 8192;
  }
}

cudaError_t launch_inverse_index(const int32_t* I, int64_t n, int64_t total, int64_t k_row, const IndexPlan& plan, int32_t* row_ptr,
                                 int32_t* slots, void* scratch, int* status, cudaStream_t st) {
  if (plan.small)
    return launch_chained_cluster(8, index_cluster_kernel, dim3(8), dim3(1024), 0, st, I, (int)n, (int)total, (int)k_row, plan.marks, row_ptr, slots, status);
  int32_t* tile_sum = (int32_t*)((char*)scratch + inv_cnt_bytes(n));
  const unsigned tiles = (unsigned)((n + kScanTile - 1) / kScanTile);
  launch_chained(inv_scan_tile_kernel, dim3(tiles), dim3(kScanThreads), 0, st, plan.marks, n, row_ptr, tile_sum);
  launch_chained(inv_scan_add_kernel, dim3(tiles), dim3(kScanThreads), 0, st, tile_sum, n, row_ptr);
  launch_chained(inv_fill_kernel, dim3(grid_for(total, 256)), dim3(256), 0, st, I, total, k_row, row_ptr, plan.marks, slots, n, status);
  if (!plan.marks.per_token) launch_chained(inv_sort_kernel, dim3(grid_for(n, 256)), dim3(256), 0, st, row_ptr, n, slots);
  return cudaGetLastError();
}

// ------------------------------------------------------------------------------------------
// Validation of an index structure (on request, and what the debug build's checks are modelled on): every access
// below is range-checked, so any contents are safe to hand in.  Violations are counted.
// ------------------------------------------------------------------------------------------
__global__ void validate_routing_kernel(const int32_t* __restrict__ I, const int32_t* __restrict__ row_ptr,
                                        const int32_t* __restrict__ slots, int64_t n, int64_t ng, int E, int64_t k_total,
                                        int64_t kg, int groups, int allow_empty, int* violations) {
  const int64_t total = (int64_t)E * k_total;
  const int64_t stride = (int64_t)gridDim.x * blockDim.x, g0 = (int64_t)blockIdx.x * blockDim.x + threadIdx.x;
  int bad = 0;
  // slots: a token of the slot's own routing group, or -1 where empty slots exist
  for (int64_t s = g0; s < total; s += stride) {
    const int t = I[s];
    const int64_t grp = (s % k_total) / kg;
    if (t == -1) { if (!allow_empty) ++bad; }
    else if (t < 0 || t >= n || t / ng != grp) ++bad;
  }
  // the token -> slot lists
  for (int64_t t = g0; t < n; t += stride) {
    const int64_t a = row_ptr[t], b = row_ptr[t + 1];
    if (t == 0 && a != 0) ++bad;
    if (a < 0 || b < a || b > total) { ++bad; continue; }
    int prev = -1;
    for (int64_t q = a; q < b; ++q) {
      const int s = slots[q];
      if (s < 0 || s >= total) { ++bad; continue; }
      if (s <= prev) ++bad;                             // ascending slot ids, hence ascending expert
      if (I[s] != t) ++bad;
      prev = s;
    }
  }
  if (bad) atomicAdd(violations, bad);
}

// every filled slot is listed exactly once: row_ptr[n] equals the number of filled slots
__global__ void validate_count_kernel(const int32_t* __restrict__ I, const int32_t* __restrict__ row_ptr, int64_t n, int64_t total,
                                      int* filled) {
  int c = 0;
  for (int64_t s = (int64_t)blockIdx.x * blockDim.x + threadIdx.x; s < total; s += (int64_t)gridDim.x * blockDim.x) c += I[s] >= 0;
  if (c) atomicAdd(filled, c);
}
__global__ void validate_total_kernel(const int32_t* __restrict__ row_ptr, int64_t n, const int* filled, int* violations) {
  if (row_ptr[n] != *filled) atomicAdd(violations, 1);
}

cudaError_t launch_validate_routing(const int32_t* I, const int32_t* row_ptr, const int32_t* slots, int64_t n, int64_t ng,
                                    int E, int64_t k_total, int64_t kg, int groups, int allow_empty, int* violations,
                                    cudaStream_t st) {
  const int64_t total = (int64_t)E * k_total;
  cudaError_t e = cudaMemsetAsync(violations, 0, 2 * sizeof(int), st);       // [0] violations, [1] filled slots
  if (e != cudaSuccess) return e;
  count_launch(3);
  validate_routing_kernel<<<grid_for(total > n ? total : n, 256), 256, 0, st>>>(I, row_ptr, slots, n, ng, E, k_total, kg, groups,
                                                                                 allow_empty, violations);
  validate_count_kernel<<<grid_for(total, 256), 256, 0, st>>>(I, row_ptr, n, total, violations + 1);
  validate_total_kernel<<<1, 1, 0, st>>>(row_ptr, n, violations + 1, violations);
  return cudaGetLastError();
}

// ------------------------------------------------------------------------------------------
// Shuffle, Eq. 3: X_in = P . X as an indexed row copy in 16-byte vectors.
// ------------------------------------------------------------------------------------------
// Which row a piece of the output belongs to.  A 64-bit division per 16 bytes is as much work to issue as HBM has to move (the
// combine at 262144 x 1024: 516 us with it, 505 without), so the host prepares a multiplication: for g < 2^31 and
// 2^(l-1) < d <= 2^l, mul = ceil(2^(31+l) / d) < 2^32 + 1 gives g / d = g * mul >> (31 + l), because mul * d - 2^(31+l) < d <= 2^l
// so that the excess g * (mul * d - 2^(31+l)) / (d * 2^(31+l)) stays below 1 / d.  (A power-of-two group of lanes per row needs
// no division either, but takes a row of an odd width in several dependent steps: combine 50 against 19 us at 9000 x 600.)
struct RowOf { unsigned long long mul; int shift, d, wide; };
static inline RowOf row_of(int64_t total, int d) {
  RowOf r; r.d = d; r.wide = total >= ((int64_t)1 << 31) ? 1 : 0;
  int l = 0; while (((int64_t)1 << l) < d) ++l;
  r.shift = 31 + l;
  r.mul = (((unsigned long long)1 << r.shift) + (unsigned)d - 1) / (unsigned)d;
  return r;
}
__device__ __forceinline__ int64_t row_of(int64_t g, const RowOf& r) {
  return r.wide ? g / r.d : (int64_t)((unsigned long long)(unsigned)g * r.mul >> r.shift);
}

__global__ void gather_kernel(const uint4* __restrict__ X, const int32_t* __restrict__ I, uint4* __restrict__ X_in,
                              int64_t total_vec, int vec_per_row, const RowOf row, int64_t n, int* status) {
  chain_enter();
  X = after_enter(X); I = after_enter(I);
  for (int64_t g = (int64_t)blockIdx.x * blockDim.x + threadIdx.x; g < total_vec; g += (int64_t)gridDim.x * blockDim.x) {
    const int64_t s = row_of(g, row); const int v = (int)(g - s * vec_per_row);
    int t = I[s];                                      // -1: an empty slot (token-choice routing only) holds a zero row
    if (t >= 0 && !idx_ok(t, 0, n, v == 0 ? status : nullptr)) t = -1;
    X_in[g] = t >= 0 ? X[(int64_t)t * vec_per_row + v] : make_uint4(0, 0, 0, 0);
  }
}

cudaError_t launch_gather(int dtype, const void* X, const int32_t* I, void* X_in, int64_t total, int d, int64_t n, int* status,
                          cudaStream_t st) {
  const int vpr = d * (dtype == 0 ? 4 : 2) / 16;
  const int64_t tv = total * vpr;
  launch_chained(gather_kernel, dim3(grid_for(tv, 256, 148 * 32)), dim3(256), 0, st, (const uint4*)X, I, (uint4*)X_in, tv, vpr, row_of(tv, vpr), n, status);
  return cudaGetLastError();
}

// ------------------------------------------------------------------------------------------
// Unshuffle, Eq. 4: X_out[t,:] = sum over the slots of t (ascending expert) of G[s] * X_e[s,:].
// Read through the token->slot index, so no atomics and a fixed summation order.
// ------------------------------------------------------------------------------------------
// four consecutive elements of a row of T
__device__ __forceinline__ void load4(const float* p, float* f) {
  const float4 v = *reinterpret_cast<const float4*>(p); f[0] = v.x; f[1] = v.y; f[2] = v.z; f[3] = v.w;
}
__device__ __forceinline__ void load4(const bf16* p, float* f) {
  const uint2 v = *reinterpret_cast<const uint2*>(p);
  f[0] = __uint_as_float(v.x << 16); f[1] = __uint_as_float(v.x & 0xFFFF0000u);
  f[2] = __uint_as_float(v.y << 16); f[3] = __uint_as_float(v.y & 0xFFFF0000u);
}
__device__ __forceinline__ void store4(float* p, const float* f) {
  *reinterpret_cast<float4*>(p) = make_float4(f[0], f[1], f[2], f[3]);
}
__device__ __forceinline__ void store4(bf16* p, const float* f) {
  __nv_bfloat162 a = __floats2bfloat162_rn(f[0], f[1]), b = __floats2bfloat162_rn(f[2], f[3]);
  *reinterpret_cast<uint2*>(p) = make_uint2(*reinterpret_cast<unsigned*>(&a), *reinterpret_cast<unsigned*>(&b));
}

template <typename T>
__global__ void combine_kernel(const float* __restrict__ X_e, const float* __restrict__ G,
                               const int32_t* __restrict__ row_ptr, const int32_t* __restrict__ slots,
                               T* __restrict__ X_out, int64_t total_quads, int quads_per_row, const RowOf row,
                               int64_t slots_total, int* status) {
  chain_enter();
  X_e = after_enter(X_e); G = after_enter(G); row_ptr = after_enter(row_ptr); slots = after_enter(slots);
  for (int64_t g = (int64_t)blockIdx.x * blockDim.x + threadIdx.x; g < total_quads; g += (int64_t)gridDim.x * blockDim.x) {
    const int64_t t = row_of(g, row); const int v = (int)(g - t * quads_per_row);
    float acc[4] = {0.f, 0.f, 0.f, 0.f};
    int a = row_ptr[t], b = row_ptr[t + 1];
    if (!idx_ok(a, 0, slots_total + 1, v == 0 ? status : nullptr) || !idx_ok(b, a, slots_total + 1, v == 0 ? status : nullptr)) a = b = 0;
    // four slots at a time: their ids, then their weights and row pieces, are fetched together, and
    // added in slot order
    for (int q0 = a; q0 < b; q0 += 4) {
      int s[4]; float w[4]; float4 x[4];
#pragma unroll
      for (int u = 0; u < 4; ++u) {
        s[u] = q0 + u < b ? slots[q0 + u] : -1;
        if (s[u] >= 0 && !idx_ok(s[u], 0, slots_total, v == 0 ? status : nullptr)) s[u] = -1;
      }
#pragma unroll
      for (int u = 0; u < 4; ++u) {
        w[u] = s[u] >= 0 ? G[s[u]] : 0.f;
        x[u] = s[u] >= 0 ? *reinterpret_cast<const float4*>(X_e + ((int64_t)s[u] * quads_per_row + v) * 4) : make_float4(0.f, 0.f, 0.f, 0.f);
      }
#pragma unroll
      for (int u = 0; u < 4; ++u) {
        if (s[u] >= 0) {
          acc[0] = fmaf(w[u], x[u].x, acc[0]); acc[1] = fmaf(w[u], x[u].y, acc[1]);
          acc[2] = fmaf(w[u], x[u].z, acc[2]); acc[3] = fmaf(w[u], x[u].w, acc[3]);
        }
      }
    }
    store4(X_out + g * 4, acc);
  }
}

// The same for many rows: a producer warp streams the rows of X_e that a CTA's tokens need (consecutive tokens' slots are one run
// of `slots`) into a ring in shared memory with bulk copies, GROUP / 32 warps take a token's rows from it in slot order.  The
// plain kernel holds a row piece per thread behind two dependent loads of indices; here some 190 KiB per SM are on their way at
// all times.  A ring entry has a barrier for its bytes (and its weight, stored before them) and one for its readers.
// 262144 x 1024, two slots a token: 490 -> 420 us from a flushed L2, 16384 x 4096: 121 -> 119.
// Where the ring is taken, from both sides measured (us plain / ring, L2 flushed, E k d in millions of floats).
//   Rows from 768 floats on: a row costs the producer and its readers a fixed time, and below it a warp cannot ask for them fast
//   enough: bf16 results 1024 wide, 512 M: 490 / 420; 768, 384 M: 332 / 326; 640, 320 M: 281 / 294; 512, 256 M: 242 / 266; 256, 64 M: 72 / 115; 64, 32 M: 49 / 213.
//   X_e beyond L2: below it a CTA's start-up is not won back (16384 slots of 768: 18.5 / 20.5; 8192 of 1024: the routing chain 49.2 / 50.6).
//   fp32 results, whose stores weigh as much as half of the loads: up to 2048 wide and from 256 M on (1024, 512 M: 557 / 513; 1024, 256 M:
//   377 / 364; 2048, 512 M: 545 / 528); else 1024, 128 M: 138 / 139; 768, 192 M: 272 / 279; 4096, 256 M: 257 / 270; 8192, 512 M: 500 / 516.
constexpr int kRingBytes = 192 * 1024, kRingFrom = 768, kRingTo = 8192, kRingToF32 = 2048, kRingWarps = 8, kRingMost = kRingBytes / (4 * kRingFrom);
template <typename T> constexpr bool takes_ring(int64_t floats, int d) {
  return sizeof(T) == 2 ? floats >= 32 << 20 && d >= kRingFrom && d <= kRingTo : floats >= 256 << 20 && d >= kRingFrom && d <= kRingToF32;
}
struct Ring { uint64_t full[kRingMost], empty[kRingMost]; float weight[kRingMost]; int row[kRingMost]; int gave_up; };
// bounded, like every wait: false when it ran out, or when another warp's did.  The clock also runs while another process has the
// device, so this is not a fault: the warps then read what is left of their rows from global memory.
__device__ __forceinline__ bool ring_wait(uint32_t bar, uint32_t parity, volatile int* gave_up, unsigned long long wait_ns) {
  if (mbar_try(bar, parity)) return true;
  const unsigned long long t0 = globaltimer();
  for (uint32_t spin = 1;; ++spin) {
    if (mbar_try(bar, parity)) return true;
    if ((spin & 63u) == 0 && (*gave_up || globaltimer() - t0 > wait_ns)) { *gave_up = 1; return false; }
  }
}
// Waits for row number `row` of the CTA in entry `at`.  A group whose tokens have no slots runs ahead of the others and may come to an
// entry a whole round early, when the parity of its barrier says nothing yet: the entry's own row number, written before its bytes
// are asked for, has to be the wanted one first.
__device__ __forceinline__ bool ring_take(Ring& ring, uint32_t full, int at, int row, uint32_t parity, unsigned long long wait_ns) {
  volatile int* held = &ring.row[at];
  if (*held != row) {
    const unsigned long long t0 = globaltimer();
    for (uint32_t spin = 1; *held != row; ++spin)
      if ((spin & 63u) == 0 && (*(volatile int*)&ring.gave_up || globaltimer() - t0 > wait_ns)) { *(volatile int*)&ring.gave_up = 1; return false; }
  }
  return ring_wait(full, parity, &ring.gave_up, wait_ns);
}
// The first token at which `slot_weight` per slot and `token_weight` per token before it add up to `work` or more: where a CTA's share
// begins.  One warp, 32 candidates a step.
__device__ __forceinline__ int64_t share_start(const int32_t* row_ptr, int64_t n, int slot_weight, int token_weight, int64_t work) {
  int64_t lo = 0, hi = n;                              // every token before lo is short of it, hi is not (or is n)
  while (lo < hi) {
    const int64_t step = (hi - lo + 31) / 32, t = min(hi - 1, lo + ((threadIdx.x & 31) + 1) * step - 1);
    const int below = __popc(__ballot_sync(0xffffffffu, (int64_t)row_ptr[t] * slot_weight + t * token_weight < work));     // candidates ascend
    if (below < 32) hi = min(hi - 1, lo + (below + 1) * step - 1);
    lo = min(hi, lo + below * step);
  }
  return lo;
}

template <typename T, int GROUP, int NQ>
__global__ void __launch_bounds__(32 * (kRingWarps + 1), 1)
combine_ring_kernel(const float* X_e, const float* G, const int32_t* row_ptr, const int32_t* slots, T* X_out, int64_t n, int d, int depth,
                    unsigned long long wait_ns, int silent) {
  extern __shared__ __align__(128) uint8_t ring_smem[];                // [depth][d] fp32
  __shared__ Ring ring;
  const int warp = threadIdx.x >> 5, lane = threadIdx.x & 31;
  const uint32_t full0 = smem_u32(ring.full), empty0 = smem_u32(ring.empty);
  if (threadIdx.x == 0) {
    for (int i = 0; i < depth; ++i) { mbar_init(full0 + 8 * i, 1); mbar_init(empty0 + 8 * i, GROUP / 32); ring.row[i] = -1; }
    ring.gave_up = 0;
    asm volatile("fence.mbarrier_init.release.cluster;" ::: "memory");
  }
  chain_enter();
  // A CTA's tokens: shares of equal bytes, a row of fp32 read per slot and a row written per token, wherever the slots lie.  (Equal
  // numbers of tokens leave the work to a few CTAs when all experts take the same ones: 65536 x 1024, 64 experts: 4260 us, 176 so,
  // where the plain kernel takes 123: with 64 slots a token, one group at a time has the ring to itself.)
  __shared__ int64_t share[2];
  if (warp < 2) {
    const int64_t work = (int64_t)row_ptr[n] * 4 + n * (int64_t)sizeof(T);
    const int64_t t = share_start(row_ptr, n, 4, sizeof(T), work * (blockIdx.x + warp) / gridDim.x);
    if (lane == 0) share[warp] = t;
  }
  __syncthreads();
  const int64_t t0 = share[0], t1 = share[1];
  if (t0 >= t1) return;
  const int64_t qa = row_ptr[t0];
  if (warp == kRingWarps) {                            // ---- producer: entry by entry, up to 32 at a time
    const int64_t qb = row_ptr[t1];
    const int step = min(32, depth);                   // a lane never waits for another of the same step
    const uint32_t bytes = (uint32_t)d * 4u;
    int64_t q = qa + lane;
    int id = lane < step && q < qb ? slots[q] : -1;
    float w = id >= 0 ? G[id] : 0.f;
    int at = lane % depth; uint32_t phase = 1;         // lane < step <= depth
    for (; q - lane < qb; q += step) {
      const int idn = lane < step && q + step < qb ? slots[q + step] : -1;
      bool ok = true;
#ifdef EC_DEBUG
      if ((int)blockIdx.x == silent && q - lane > qa) break;           // asks for no more rows than the first few
#endif
      if (id >= 0) {
        ok = ring_wait(empty0 + 8 * at, phase, &ring.gave_up, wait_ns);
        if (ok) {
          ring.weight[at] = w;
          *(volatile int*)&ring.row[at] = (int)(q - qa);
          mbar_expect_tx(full0 + 8 * at, bytes);
          asm volatile("cp.async.bulk.shared::cluster.global.mbarrier::complete_tx::bytes [%0], [%1], %2, [%3];"
                       ::"r"(smem_u32(ring_smem) + (uint32_t)at * bytes), "l"(X_e + (int64_t)id * d), "r"(bytes), "r"(full0 + 8 * at) : "memory");
        }
      }
      if (!__all_sync(0xffffffffu, ok)) break;
      id = idn; w = id >= 0 ? G[id] : 0.f;
      at += step;
      if (at >= depth) { at -= depth; phase ^= 1; }
    }
  } else {                                             // ---- consumers: a group per token
    constexpr int kGroups = kRingWarps * 32 / GROUP;
    const int grp = threadIdx.x / GROUP, gl = threadIdx.x % GROUP;
    // the bounds of the group's next 32 lists, a lane each, and of the 32 after them: tokens without slots cost a row of zeros, no round trip
    auto bound = [&](int64_t t, int end) { return t < t1 ? row_ptr[t + end] : 0; };
    int64_t t = t0 + grp;
    int la = 0, lb = 0, la2 = bound(t + lane * kGroups, 0), lb2 = bound(t + lane * kGroups, 1);
    bool ok = true;                                    // until a wait runs out
    for (int i = 0; t < t1; t += kGroups, i = (i + 1) & 31) {
      if (i == 0) { la = la2; lb = lb2; la2 = bound(t + (32 + lane) * kGroups, 0); lb2 = bound(t + (32 + lane) * kGroups, 1); }
      const int64_t a = __shfl_sync(0xffffffffu, la, i), b = __shfl_sync(0xffffffffu, lb, i);
      float acc[NQ][4];
#pragma unroll
      for (int j = 0; j < NQ; ++j) acc[j][0] = acc[j][1] = acc[j][2] = acc[j][3] = 0.f;
      int at = (int)((a - qa) % depth); uint32_t phase = (uint32_t)((a - qa) / depth) & 1u;
      auto add = [&](int j, float w, const float4& f) {
        acc[j][0] = fmaf(w, f.x, acc[j][0]); acc[j][1] = fmaf(w, f.y, acc[j][1]);
        acc[j][2] = fmaf(w, f.z, acc[j][2]); acc[j][3] = fmaf(w, f.w, acc[j][3]);
      };
      int64_t q = a;
      for (; ok && q < b; ++q) {
        ok = __all_sync(0xffffffffu, ring_take(ring, full0 + 8 * at, at, (int)(q - qa), phase, wait_ns));
        if (!ok) break;
        const float w = ring.weight[at];
        const float4* x = reinterpret_cast<const float4*>(ring_smem) + (int64_t)at * (d / 4);
#pragma unroll
        for (int j = 0; j < NQ; ++j) if (gl + j * GROUP < d / 4) add(j, w, x[gl + j * GROUP]);
        __syncwarp();
        if (lane == 0) mbar_arrive(empty0 + 8 * at);
        if (++at == depth) { at = 0; phase ^= 1; }
      }
      for (; q < b; ++q) {                             // without the ring
        const int64_t id = slots[q];
#pragma unroll
        for (int j = 0; j < NQ; ++j) if (gl + j * GROUP < d / 4) add(j, G[id], reinterpret_cast<const float4*>(X_e + id * d)[gl + j * GROUP]);
      }
#pragma unroll
      for (int j = 0; j < NQ; ++j) if (gl + j * GROUP < d / 4) store4(X_out + t * d + 4 * (gl + j * GROUP), acc[j]);
    }
  }
  __syncthreads();
  if (ring.gave_up) {                                  // copies in flight land before the shared memory goes
    const unsigned long long s0 = globaltimer();
    while (globaltimer() - s0 < 200000ull) __nanosleep(1000);
  }
}

template <typename T, int GROUP, int NQ>
cudaError_t launch_combine_ring(const float* X_e, const float* G, const int32_t* row_ptr, const int32_t* slots, T* X_out, int64_t n, int d,
                                int sms, unsigned long long wait_ns, int silent, cudaStream_t st) {
  auto kern = combine_ring_kernel<T, GROUP, NQ>;
  const cudaError_t e = cudaFuncSetAttribute(kern, cudaFuncAttributeMaxDynamicSharedMemorySize, kRingBytes);
  if (e != cudaSuccess) return e;
  const int depth = kRingBytes / (d * 4);
  return launch_chained(kern, dim3((unsigned)(n < sms ? n : sms)), dim3(32 * (kRingWarps + 1)), (size_t)depth * d * 4, st, X_e, G, row_ptr, slots, X_out, n, d,
                        depth, wait_ns, silent);
}
template <typename T>
cudaError_t launch_combine_t(const float* X_e, const float* G, const int32_t* row_ptr, const int32_t* slots, T* X_out, int64_t n, int d,
                             int64_t slots_total, int* status, cudaStream_t st, unsigned long long wait_ns, int silent) {
#ifdef EC_DEBUG                                        // the debug build's lists may be anything: the plain kernel checks every index
  const bool ring = silent >= 0 && takes_ring<T>((int64_t)1 << 40, d);
#else
  const bool ring = takes_ring<T>(slots_total * d, d);
#endif
  if (ring) {
    int dev = 0, sms = 148;
    cudaGetDevice(&dev);
    cudaDeviceGetAttribute(&sms, cudaDevAttrMultiProcessorCount, dev);
    if (d <= 1024) return launch_combine_ring<T, 32, 8>(X_e, G, row_ptr, slots, X_out, n, d, sms, wait_ns, silent, st);
    if (d <= 2048) return launch_combine_ring<T, 64, 8>(X_e, G, row_ptr, slots, X_out, n, d, sms, wait_ns, silent, st);
    if constexpr (sizeof(T) == 2) {
      if (d <= 4096) return launch_combine_ring<T, 128, 8>(X_e, G, row_ptr, slots, X_out, n, d, sms, wait_ns, silent, st);
      return launch_combine_ring<T, 256, 8>(X_e, G, row_ptr, slots, X_out, n, d, sms, wait_ns, silent, st);
    }
  }
  const int qpr = d / 4;
  const int64_t tq = n * qpr;
  return launch_chained(combine_kernel<T>, dim3(grid_for(tq, 256, 148 * 32)), dim3(256), 0, st, X_e, G, row_ptr, slots, X_out, tq, qpr, row_of(tq, qpr),
                        slots_total, status);
}
cudaError_t launch_combine(int dtype, const float* X_e, const float* G, const int32_t* row_ptr, const int32_t* slots,
                           void* X_out, int64_t n, int d, int64_t slots_total, int* status, cudaStream_t st,
                           unsigned long long wait_ns, int silent) {
  return dtype == 0 ? launch_combine_t(X_e, G, row_ptr, slots, (float*)X_out, n, d, slots_total, status, st, wait_ns, silent)
                    : launch_combine_t(X_e, G, row_ptr, slots, (bf16*)X_out, n, d, slots_total, status, st, wait_ns, silent);
}

// ------------------------------------------------------------------------------------------
// Backward of Eq. 4 and of the softmax of Eq. 2, one warp per token t.  For every slot s of t (expert i):
//   dX_e[s,:] = G[s] * dX_out[t,:],   dG[s] = <dX_out[t,:], X_e[s,:]>,
// and with dS[t,i] = dG of that slot (0 where t has none),
//   dL[t,i] = S[t,i] * (dS[t,i] - sum_i' dS[t,i'] * S[t,i']).
// A row of dX_out is read once for two slots, and what the softmax needs is in the warp's hands.  Bound by HBM at the
// layer's sizes.  With one warp per slot and the softmax in a launch of its own (the lists of the next tokens are fetched ahead here, two
// rows of X_e travel together): 2048 x 256, 8 experts 15.7 -> 8.8 us; 8192 x 768, 32 experts 31.8 -> 24.9; 6080 x 1000, ten experts
// 22.7 -> 17.0; 16384 x 4096, 64 experts 182 -> 196, where rows in slot order are the better order for HBM.  (Four rows at a time
// leave no registers for loads in flight: 27.0 us at 8192 x 768.)
// ------------------------------------------------------------------------------------------
__device__ __forceinline__ void st_dl(float* p, int64_t i, float v) { p[i] = v; }
__device__ __forceinline__ void st_dl(bf16* p, int64_t i, float v) { p[i] = __float2bfloat16(v); }

// SLOTS of a token's slots at once: dX_e of each, and each one's dot product in every lane.  A lane takes 16 bytes of dX_out at a
// time: `vecs` such pieces a row.
template <int SLOTS, typename T>
__device__ __forceinline__ void bwd_rows(const uint4* dy_row, const float* X_e, T* dX_e, const int (&s)[2], const float (&w)[2], int vecs, float (&dot)[2]) {
  constexpr int N = Vec<T>::N;
  const int lane = threadIdx.x & 31;
#pragma unroll
  for (int u = 0; u < SLOTS; ++u) dot[u] = 0.f;
#pragma unroll 2
  for (int v = lane; v < vecs; v += 32) {
    const uint4 raw = dy_row[v];
    float4 xe[SLOTS][N / 4];
#pragma unroll
    for (int u = 0; u < SLOTS; ++u)
#pragma unroll
      for (int j = 0; j < N / 4; ++j) xe[u][j] = *reinterpret_cast<const float4*>(X_e + ((int64_t)s[u] * vecs + v) * N + 4 * j);
    float dy[N]; Vec<T>::unpack(raw, dy);
#pragma unroll
    for (int u = 0; u < SLOTS; ++u) {
      float o[N];
#pragma unroll
      for (int j = 0; j < N / 4; ++j) {
        const float x[4] = {xe[u][j].x, xe[u][j].y, xe[u][j].z, xe[u][j].w};
#pragma unroll
        for (int i = 0; i < 4; ++i) { o[4 * j + i] = w[u] * dy[4 * j + i]; dot[u] = fmaf(dy[4 * j + i], x[i], dot[u]); }
      }
      reinterpret_cast<uint4*>(dX_e)[(int64_t)s[u] * vecs + v] = Vec<T>::pack(o);
    }
  }
#pragma unroll
  for (int o = 16; o; o >>= 1)
#pragma unroll
    for (int u = 0; u < SLOTS; ++u) dot[u] += __shfl_xor_sync(0xffffffffu, dot[u], o);
}

// A token with more than kBwdLong slots is shared by a CTA's warps: where all experts take the same block of tokens, a warp per
// token leaves most of the chip idle.  (64 slots a token, 16384 tokens of 1024: 117 us with a warp per token, 55 so; of 4096: 404 and 148.)
// CTAs of four warps: with eight the common path, whose warps wait for each other at the end, takes 1 % longer.
constexpr int kBwdLong = 8, kBwdLongs = 64, kBwdThreads = 128;
// Their slots go by pairs over the warps, then a warp per token does the softmax, in the order of bwd_tokens_kernel.  Not inlined: the
// registers it would take there cost the common path 1 us of 29.
template <typename T, typename TL>
__device__ __noinline__ void bwd_long_lists(const int64_t* tokens, int count, const T* dX_out, const float* X_e, const float* G, const float* S,
                                            const int32_t* row_ptr, const int32_t* slots, T* dX_e, float* dG, TL* dL, int vecs, int E, int k, int* status) {
  const int lane = threadIdx.x & 31, warp = threadIdx.x >> 5, warps = blockDim.x >> 5, slots_total = E * k;
  auto slot = [&](int q) { const int s = slots[q]; return s >= 0 && idx_ok(s, 0, slots_total, status) ? s : -1; };
  for (int i = 0; i < count; ++i) {
    const int64_t t = tokens[i];
    const uint4* dy = reinterpret_cast<const uint4*>(dX_out) + t * vecs;
    for (int q = row_ptr[t] + 2 * warp, b = row_ptr[t + 1]; q < b; q += 2 * warps) {
      int s[2] = {slot(q), q + 1 < b ? slot(q + 1) : -1};
      if (s[0] < 0) { s[0] = s[1]; s[1] = -1; }
      if (s[0] < 0) continue;
      const float w[2] = {G[s[0]], s[1] >= 0 ? G[s[1]] : 0.f};
      float dg[2];
      if (s[1] >= 0) bwd_rows<2>(dy, X_e, dX_e, s, w, vecs, dg); else bwd_rows<1>(dy, X_e, dX_e, s, w, vecs, dg);
      if (lane == 0) { dG[s[0]] = dg[0]; if (s[1] >= 0) dG[s[1]] = dg[1]; }
    }
  }
  __syncthreads();                                     // dG is read back by other warps
  for (int i = warp; i < count; i += warps) {
    const int64_t t = tokens[i];
    const int a = row_ptr[t], b = row_ptr[t + 1];
    const float* St = S + t * E;
    float dot = 0.f;
    for (int q = a + lane; q < b; q += 32) { const int s = slot(q); if (s >= 0) dot = fmaf(dG[s], St[s / k], dot); }
    for (int o = 16; o; o >>= 1) dot += __shfl_xor_sync(0xffffffffu, dot, o);
    for (int e = lane; e < E; e += 32) st_dl(dL, t * E + e, -St[e] * dot);
    __syncwarp();
    for (int q = a + lane; q < b; q += 32) { const int s = slot(q); if (s >= 0) st_dl(dL, t * E + s / k, St[s / k] * (dG[s] - dot)); }
  }
}

// empty: not null where slots may be empty (token-choice routing): I, whose negative entries get zero rows and no gradient
template <typename T, typename TL>
__global__ void __launch_bounds__(kBwdThreads, 1024 / kBwdThreads) bwd_tokens_kernel(const T* dX_out, const float* X_e, const float* G, const float* S, const int32_t* row_ptr,
                                                            const int32_t* slots, const int32_t* empty, T* dX_e, float* dG, TL* dL, int64_t n, int vecs,
                                                            int E, int k, int clear, int* status) {
  chain_enter();
  if (clear && blockIdx.x == 0 && threadIdx.x < kStatusWords) status[threadIdx.x] = 0;       // the first kernel of a call
  const int lane = threadIdx.x & 31, slots_total = E * k;
  // neighbouring tokens lie in different CTAs, and a CTA's long lists (s_long) wait for all of its warps
  __shared__ int s_longs;
  __shared__ int64_t s_long[kBwdLongs];
  const int warp = threadIdx.x >> 5;
  const int64_t warps = ((int64_t)gridDim.x * blockDim.x) >> 5, first = (int64_t)warp * gridDim.x + blockIdx.x;
  if (threadIdx.x == 0) s_longs = 0;
  __syncthreads();
  auto list_of = [&](int64_t t, int& a, int& b) {
    a = b = 0;
    if (t >= n) return;
    a = row_ptr[t]; b = row_ptr[t + 1];
    if (!idx_ok(a, 0, slots_total + 1, lane == 0 ? status : nullptr) || !idx_ok(b, a, slots_total + 1, lane == 0 ? status : nullptr)) a = b = 0;
  };
  auto slot_at = [&](int q, int b) {                   // this lane's slot, or -1
    const int s = q + lane < b ? slots[q + lane] : -1;
    return s >= 0 && idx_ok(s, 0, slots_total, status) ? s : -1;
  };
  // a token's list is fetched while the one before it is worked on, its bounds one token earlier still
  int a, b, an, bn;
  list_of(first, a, b); list_of(first + warps, an, bn);
  int id = slot_at(a, b), longs = 0;
  for (int64_t t = first; t < n; t += warps) {
    const int idn = slot_at(an, bn);
    int a2, b2; list_of(t + 2 * warps, a2, b2);
    if (b - a > kBwdLong) {
      longs = 1;
      int at = lane == 0 ? atomicAdd(&s_longs, 1) : 0;
      at = __shfl_sync(0xffffffffu, at, 0);
      if (at < kBwdLongs) {
        if (lane == 0) s_long[at] = t;
        a = an; b = bn; id = idn; an = a2; bn = b2;
        continue;
      }
    }
    float dot = 0.f, mine = 0.f, sc = 0.f;             // of this lane's slot: dG, and its score
    for (int q = a; q < b; q += 32) {                  // nearly always once
      if (q > a) id = slot_at(q, b);
      const float wl = id >= 0 ? G[id] : 0.f;
      sc = id >= 0 ? S[t * E + id / k] : 0.f;
      unsigned left = __ballot_sync(0xffffffffu, id >= 0);
      while (left) {
        int s[2], from[2], have = 0; float w[2], dg[2];
#pragma unroll
        for (int u = 0; u < 2; ++u) {
          from[u] = left ? __ffs(left) - 1 : 0;
          have += left ? 1 : 0;
          left &= left - 1u;
          s[u] = __shfl_sync(0xffffffffu, id, from[u]); w[u] = __shfl_sync(0xffffffffu, wl, from[u]);
        }
        const uint4* dy = reinterpret_cast<const uint4*>(dX_out) + t * vecs;
        if (have == 1) bwd_rows<1>(dy, X_e, dX_e, s, w, vecs, dg);
        else bwd_rows<2>(dy, X_e, dX_e, s, w, vecs, dg);
#pragma unroll
        for (int u = 0; u < 2; ++u) if (u < have && lane == from[u]) mine = dg[u];
      }
      if (id >= 0) { dG[id] = mine; dot = fmaf(mine, sc, dot); }
    }
    for (int o = 16; o; o >>= 1) dot += __shfl_xor_sync(0xffffffffu, dot, o);
    for (int i = lane; i < E; i += 32) st_dl(dL, t * E + i, -S[t * E + i] * dot);
    __syncwarp();                                      // dG of this token may be read back, dL is written over
    if (b - a <= 32) {
      if (id >= 0) st_dl(dL, t * E + id / k, sc * (mine - dot));       // the slots of one token belong to distinct experts
    } else {
      for (int q = a + lane; q < b; q += 32) {
        const int s = slots[q];
        if (idx_ok(s, 0, slots_total, nullptr)) st_dl(dL, t * E + s / k, S[t * E + s / k] * (dG[s] - dot));
      }
    }
    a = an; b = bn; id = idn; an = a2; bn = b2;
  }
  if (__syncthreads_or(longs)) bwd_long_lists(s_long, min(s_longs, kBwdLongs), dX_out, X_e, G, S, row_ptr, slots, dX_e, dG, dL, vecs, E, k, status);
  if (empty == nullptr) return;
  for (int64_t s = first; s < slots_total; s += warps) {
    if (empty[s] >= 0) continue;
    for (int v = lane; v < vecs; v += 32) reinterpret_cast<uint4*>(dX_e)[s * vecs + v] = make_uint4(0, 0, 0, 0);
    if (lane == 0) dG[s] = 0.f;
  }
}

template <typename T, typename TL>
cudaError_t launch_bwd_tokens_t(const void* dX_out, const float* X_e, const float* G, const float* S, const int32_t* row_ptr, const int32_t* slots,
                                const int32_t* empty, void* dX_e, float* dG, void* dL, int64_t n, int d, int E, int64_t k, int clear, int* status, cudaStream_t st) {
  return launch_chained(bwd_tokens_kernel<T, TL>, dim3(grid_for(n * 32, kBwdThreads, 148 * 32)), dim3(kBwdThreads), 0, st, (const T*)dX_out, X_e, G, S, row_ptr, slots, empty,
                        (T*)dX_e, dG, (TL*)dL, n, d / Vec<T>::N, E, (int)k, clear, status);
}
cudaError_t launch_bwd_tokens(int dtype, const void* dX_out, const float* X_e, const float* G, const float* S, const int32_t* row_ptr, const int32_t* slots,
                              const int32_t* empty, void* dX_e, float* dG, void* dL, int dl_bf16, int64_t n, int d, int E, int64_t k, int clear, int* status,
                              cudaStream_t st) {
  if (dtype == 0) return launch_bwd_tokens_t<float, float>(dX_out, X_e, G, S, row_ptr, slots, empty, dX_e, dG, dL, n, d, E, k, clear, status, st);
  if (dl_bf16) return launch_bwd_tokens_t<bf16, bf16>(dX_out, X_e, G, S, row_ptr, slots, empty, dX_e, dG, dL, n, d, E, k, clear, status, st);
  return launch_bwd_tokens_t<bf16, float>(dX_out, X_e, G, S, row_ptr, slots, empty, dX_e, dG, dL, n, d, E, k, clear, status, st);
}

// ------------------------------------------------------------------------------------------
// Column sums per expert (gradients of the bias terms Eq. 3 leaves out).  A CTA owns 64 columns of one expert; its eight
// warps take every eighth row, a lane two columns, and the eight sums join in ascending order, so the result does not
// depend on scheduling.  Bound by the latency of the eight loads a warp has in flight.  Ten experts of 608 rows, 2072 and
// 1000 columns in bf16: 105 us with one thread per column, 20 us now, both launches.
// ------------------------------------------------------------------------------------------
__device__ __forceinline__ float2 ld_pair(const float* p) { return *reinterpret_cast<const float2*>(p); }
__device__ __forceinline__ float2 ld_pair(const bf16* p) {
  const unsigned v = *reinterpret_cast<const unsigned*>(p);
  return make_float2(__uint_as_float(v << 16), __uint_as_float(v & 0xFFFF0000u));
}
template <typename T>
__global__ void __launch_bounds__(256) column_sums_kernel(const T* __restrict__ A, T* __restrict__ out, int64_t rows, int cols,
                                                          const int32_t* __restrict__ batch_rows) {
  chain_enter();
  A = after_enter(A); batch_rows = after_enter(batch_rows);
  __shared__ float2 s_part[8][32];
  const int b = blockIdx.y, warp = threadIdx.x >> 5, lane = threadIdx.x & 31, c = blockIdx.x * 64 + lane * 2;      // cols is a multiple of 4
  int64_t lim = rows;
  if (batch_rows != nullptr && batch_rows[b] < lim) lim = batch_rows[b];
  const T* p = A + (int64_t)b * rows * cols + (c < cols ? c : 0);
  float2 acc = make_float2(0.f, 0.f);
  int64_t r = warp;
  for (; r + 56 < lim; r += 64) {
    float2 v[8];
#pragma unroll
    for (int u = 0; u < 8; ++u) v[u] = ld_pair(p + (r + 8 * u) * cols);
#pragma unroll
    for (int u = 0; u < 8; ++u) { acc.x += v[u].x; acc.y += v[u].y; }
  }
  for (; r < lim; r += 8) { const float2 v = ld_pair(p + r * cols); acc.x += v.x; acc.y += v.y; }
  s_part[warp][lane] = acc;
  __syncthreads();
  if (warp != 0 || c >= cols) return;
#pragma unroll
  for (int w = 1; w < 8; ++w) { acc.x += s_part[w][lane].x; acc.y += s_part[w][lane].y; }
  T* o = out + (int64_t)b * cols + c;
  if constexpr (sizeof(T) == 4) { o[0] = acc.x; o[1] = acc.y; } else { o[0] = __float2bfloat16(acc.x); o[1] = __float2bfloat16(acc.y); }
}

cudaError_t launch_column_sums(int dtype, const void* A, void* out, int batches, int64_t rows, int cols,
                               const int32_t* batch_rows, cudaStream_t st) {
  const dim3 grid((cols + 63) / 64, batches);
  if (dtype == 0) launch_chained(column_sums_kernel<float>, grid, dim3(256), 0, st, (const float*)A, (float*)out, rows, cols, batch_rows);
  else launch_chained(column_sums_kernel<bf16>, grid, dim3(256), 0, st, (const bf16*)A, (bf16*)out, rows, cols, batch_rows);
  return cudaGetLastError();
}

// ------------------------------------------------------------------------------------------
// Fixed-order sum of split partial results.
// ------------------------------------------------------------------------------------------
template <typename T>
__global__ void reduce_partials_kernel(const float* __restrict__ part, T* __restrict__ out, int P, int64_t elems) {
  chain_enter();
  part = after_enter(part);
  for (int64_t g = (int64_t)blockIdx.x * blockDim.x + threadIdx.x; g < elems; g += (int64_t)gridDim.x * blockDim.x) {
    float acc = 0.f;
    for (int p = 0; p < P; ++p) acc += part[(int64_t)p * elems + g];
    if constexpr (sizeof(T) == 4) out[g] = acc; else out[g] = __float2bfloat16(acc);
  }
}

cudaError_t launch_reduce_partials(int dtype, const float* part, void* out, int P, int64_t elems, cudaStream_t st) {
  if (dtype == 0) { launch_chained(reduce_partials_kernel<float>, dim3(grid_for(elems, 256)), dim3(256), 0, st, part, (float*)out, P, elems); }
  else { launch_chained(reduce_partials_kernel<bf16>, dim3(grid_for(elems, 256)), dim3(256), 0, st, part, (bf16*)out, P, elems); }
  return cudaGetLastError();
}

}  // namespace ecmoe
