// Expert choice with at most b experts per token (Section 3.3): the matrix A [e, n] of
//
//     max <S^T, A> + lambda H(A)   s.t.  rows sum to k,  columns sum to at most b,  0 <= A <= 1
//
// by Dykstra's algorithm with Kullback-Leibler projections onto the three sets in turn, a fixed number of
// rounds.  The projections are rescalings and a clip, so the iteration runs on L = log A, stored token-major
// ([n, e], like S) beside the log correction factors of the column set (one per token) and of the box set
// (one per entry):
//
//     rows:     L[t, i] += log k - logsumexp_t L[:, i]
//     columns:  B = L[t, :] + qc[t];  m = min(0, log b - logsumexp_i B);  L[t, :] = B + m;  qc[t] = -m
//     box:      B = L + qb;  L = min(B, 0);  qb = B - L
//
// A warp owns a token (its e values, a few per lane), so the column and box steps need only warp shuffles; the
// row step needs a sum over all tokens, which a round prepares for the next: every CTA leaves (max, sum of exp)
// of its tokens per expert, and the CTAs each combine those in a fixed order (so the result does not depend on
// scheduling) before they touch their tokens.  Three forms:
//   - resident: one cooperative launch for all rounds; a warp keeps log A and the factors of its (at most 8 /
//     experts-per-lane) tokens in registers, and only the row partials go through memory, as words that carry their
//     round's number: a CTA waits for the words it needs, there is no grid barrier (see Exchange).  Used whenever the tokens
//     fit (up to about 19 k tokens at 64 experts).  Groups that one cluster of 8 or 16 CTAs holds (up to 4096 tokens at 32
//     experts) pass the partials through the cluster's shared memory instead (see Box);
//   - resident in shared memory: the same launch with the state in the CTA's shared memory, for up to about
//     2.4 M entries per device (16384 tokens x 128 experts, 65536 x 32);
//   - one launch per round with the state (2 x 4 bytes per entry) in global memory, where it stays in L2 at
//     the layer sizes.  For everything else.
// Whichever it is, a round costs latency (one round trip for the partials or a launch, the reduction trees), not
// bandwidth.  Routing groups are independent problems (grid.y).
#include "internal.h"
#include "tc_ptx.cuh"

#include <math.h>

namespace ecmoe {

namespace {

constexpr int kCapThreads = 1024;
constexpr int kCapWarps = kCapThreads / 32;
constexpr int kCapMaxE = 256;
constexpr int kRoundLoads = 4;                       // partials a thread of the row step has in flight (one launch per round)
constexpr int kCapBatch = 4;                         // tokens of a warp whose loads are in flight together (fewer with many experts per lane)
constexpr int kCapResident = 8;                      // (tokens per warp) x (experts per lane) the resident form holds:
                                                     // log A and the box factors of that many entries in a lane's registers

// (m, s) stands for s * exp(m); the sum of two such numbers (the same bits whichever operand comes first)
__device__ __forceinline__ void lse_add(float& m, float& s, float m2, float s2) {
  if (s2 == 0.f) return;
  if (s == 0.f) { m = m2; s = s2; return; }
  if (m2 > m) { s = s * __expf(m - m2) + s2; m = m2; } else { s += s2 * __expf(m2 - m); }
}
// butterfly over `width` adjacent lanes (a power of two): every lane ends with the same sum
__device__ __forceinline__ void lse_butterfly(float& m, float& s, int width) {
  for (int o = width >> 1; o > 0; o >>= 1) {
    const float m2 = __shfl_xor_sync(0xffffffffu, m, o), s2 = __shfl_xor_sync(0xffffffffu, s, o);
    lse_add(m, s, m2, s2);
  }
}

// ---- exchange of the row partials in the resident forms ---------------------------------------------
// A word is 64 bits in global memory: a value in the low half, the number of the pass that wrote it in the high half.
// Value and number are stored and loaded together, so a reader that sees the number has the value, without a barrier.
// A round takes two hops: every CTA leaves its sums, one word per expert; the CTA an expert belongs to (expert i to CTA
// i mod the group's CTAs, a warp per expert) adds them up and leaves the expert's shift in one word for every CTA.
// Cycles of a round spent here at 16384 tokens x 64 experts on 148 CTAs: 14 k with a grid barrier and every CTA reading
// all partials after it; 7.5 k with words in one hop, every CTA reading all CTAs' words, 11 MB per sweep; 6.9 k in two hops
// with one copy of the shifts; 4.7 k like this.  Pass p uses the buffers p & 1; nobody can be two passes ahead of a
// reader, since every pass waits for all CTAs' words of the one before.  The words start with the number 2^32 - 1 (the
// launcher fills them).  All CTAs of a cooperative launch are on the device at once; a wait is nevertheless bounded:
// after kCapWaitNs the status word says so and the CTAs leave, with zeros in their part of A: what follows on the stream
// reads A before anyone has looked at the status.
__device__ __forceinline__ void word_store(unsigned long long* p, float v, unsigned pass) {
  asm volatile("st.relaxed.gpu.global.u64 [%0], %1;" ::"l"(p), "l"((unsigned long long)__float_as_uint(v) | ((unsigned long long)pass << 32)) : "memory");
}
__device__ __forceinline__ unsigned long long word_load(const unsigned long long* p) {
  unsigned long long v; asm volatile("ld.relaxed.gpu.global.u64 %0, [%1];" : "=l"(v) : "l"(p) : "memory"); return v;
}
__device__ __forceinline__ unsigned long long cap_timer() {
  unsigned long long t; asm volatile("mov.u64 %0, %%globaltimer;" : "=l"(t)); return t;
}
// Fetches the words row[q], row[q + 32], ... of up to N CTAs (below bpg), all in flight together, until each carries
// `pass`; 0 beyond the last CTA.  False when the wait ran out.
constexpr int kCapLoads = 5;
template <int N>
__device__ __forceinline__ bool words_fetch(const unsigned long long* row, int q, int bpg, unsigned pass, unsigned long long wait_ns, float (&v)[N]) {
  unsigned long long w[N];
#pragma unroll
  for (int u = 0; u < N; ++u) w[u] = q + u * 32 < bpg ? word_load(row + q + u * 32) : (unsigned long long)pass << 32;
  unsigned long long t0 = 0;
  for (unsigned spin = 0;; ++spin) {
    bool ok = true;
#pragma unroll
    for (int u = 0; u < N; ++u) ok = ok && (unsigned)(w[u] >> 32) == pass;
    if (ok) break;
    if ((spin & 255u) == 255u) {
      if (t0 == 0) t0 = cap_timer();
      else if (cap_timer() - t0 > wait_ns) return false;
    }
#pragma unroll
    for (int u = 0; u < N; ++u)
      if ((unsigned)(w[u] >> 32) != pass) w[u] = word_load(row + q + u * 32);
  }
#pragma unroll
  for (int u = 0; u < N; ++u) v[u] = __uint_as_float((unsigned)w[u]);
  return true;
}
// first_max, first_sum, even, odd: [groups * E][CTAs of a group]; shift_even, shift_odd: [groups][CTAs of a group][E], a copy
// for each reader (148 CTAs waiting for the same four lines of L2 hold up the store they wait for)
struct Exchange {
  unsigned long long *first_max, *first_sum, *even, *odd, *shift_even, *shift_odd; int* status;
  unsigned long long wait_ns;
  int silent;                                        // debug build: this CTA of a group leaves no words after the first pass (-1: none)
  static size_t words(int bpg, int groups, int E) { return (size_t)6 * bpg * groups * E; }
  static Exchange at(unsigned long long* p, int bpg, int groups, int E, int* status, unsigned long long wait_ns, int silent) {
    const size_t n = (size_t)bpg * groups * E;
    return {p, p + n, p + 2 * n, p + 3 * n, p + 4 * n, p + 5 * n, status, wait_ns, silent};
  }
};

// Shared memory of a CTA: wpart [warps][E + 1] float2 | shift [E] float
__device__ __forceinline__ float* shift_of(float2* smem, int E) { return reinterpret_cast<float*>(smem + kCapWarps * (E + 1)); }

// shift[i] = log k - log(sum over the group's tokens of exp L[:, i]) from the partials the CTAs of group g left.
// P adjacent lanes share an expert: each combines every P-th CTA's partial in ascending order, a butterfly joins them.
// Every thread of the CTA calls these.  The form of one launch per round reads (max, sum) pairs:
__device__ __forceinline__ int row_lanes(int E) { int P = 32; while (P * E > kCapThreads) P >>= 1; return P; }       // E <= 256: P >= 4
__device__ __forceinline__ void row_shifts(const float2* part_in, int g, int bpg, int E, float log_k, float* shift) {
  const int P = row_lanes(E);
  const int i = threadIdx.x / P, p0 = threadIdx.x % P;
  float m = 0.f, s = 0.f;
  if (i < E) {
    for (int q = p0; q < bpg; q += kRoundLoads * P) {
      float2 v[kRoundLoads];
#pragma unroll
      for (int u = 0; u < kRoundLoads; ++u) {
        const int qq = q + u * P;
        v[u] = qq < bpg ? __ldcg(part_in + ((int64_t)g * E + i) * bpg + qq) : make_float2(0.f, 0.f);   // adjacent lanes, adjacent CTAs
      }
#pragma unroll
      for (int u = 0; u < kRoundLoads; ++u) lse_add(m, s, v[u].x, v[u].y);
    }
  }
  lse_butterfly(m, s, P);                            // whole warps take part: P divides 32
  if (i < E && p0 == 0) shift[i] = log_k - (m + __logf(s));
  __syncthreads();
}
// The resident forms wait for words.  Pass 0 has a maximum and a sum per expert; from then on every entry is at most 1, the
// maxima are taken as 0 and the sums are added as they are.  False when a wait ran out (for all threads of the CTA).
__device__ __forceinline__ bool row_shifts(const Exchange& x, int pass, int g, int bpg, int blk, int E, float log_k, float* shift) {
  const int warp = threadIdx.x >> 5, lane = threadIdx.x & 31;
  unsigned long long* out = ((pass & 1) ? x.shift_odd : x.shift_even) + (int64_t)g * bpg * E;
  bool ok = true;
  for (int i = blk + warp * bpg; i < E; i += kCapWarps * bpg) {        // this CTA's experts: uniform across the warp
    const int64_t row = ((int64_t)g * E + i) * bpg;
    float m = 0.f, s = 0.f;
    if (pass == 0) {
      for (int q = lane; ok && q < bpg; q += 32) {
        float mv[1], v[1];
        ok = words_fetch(x.first_max + row, q, bpg, 0u, x.wait_ns, mv) && words_fetch(x.first_sum + row, q, bpg, 0u, x.wait_ns, v);
        if (ok) lse_add(m, s, mv[0], v[0]);
      }
      lse_butterfly(m, s, 32);
    } else {
      for (int q = lane; ok && q < bpg; q += kCapLoads * 32) {
        float v[kCapLoads];
        ok = words_fetch(((pass & 1) ? x.odd : x.even) + row, q, bpg, (unsigned)pass, x.wait_ns, v);
#pragma unroll
        for (int u = 0; u < kCapLoads; ++u) s += ok ? v[u] : 0.f;
      }
#pragma unroll
      for (int o = 16; o > 0; o >>= 1) s += __shfl_xor_sync(0xffffffffu, s, o);
    }
    ok = __all_sync(0xffffffffu, ok);
    if (!ok) break;
    const float v = log_k - (m + __logf(s));
    for (int q = lane; q < bpg; q += 32) word_store(out + (int64_t)q * E + i, v, (unsigned)pass);
  }
  if (ok && threadIdx.x < E) {
    float v[1];
    ok = words_fetch(out + (int64_t)blk * E + threadIdx.x, 0, 1, (unsigned)pass, x.wait_ns, v);
    if (ok) shift[threadIdx.x] = v[0];
  }
  if (__syncthreads_and(ok)) return true;
  if (threadIdx.x == 0) { atomicExch(x.status + 1, 8); atomicExch(x.status, 5 /* EC_ERR_TIMEOUT */); }
  return false;
}

// The CTA's (max, sum of exp) per expert from the lanes' running values; warp w joins experts w, w + 32, ...  A row of
// wpart has a word to spare, which spreads the 32 warps' values of one expert over the banks.
template <int EPL>
__device__ __forceinline__ void publish_partials(const float (&pm)[EPL], const float (&ps)[EPL], float2* wpart, int E,
                                                 float2* __restrict__ part_out, int g, int bpg, int blk) {
  const int warp = threadIdx.x >> 5, lane = threadIdx.x & 31;
  __syncthreads();                                   // the previous use of wpart and shift is over
#pragma unroll
  for (int j = 0; j < EPL; ++j) if (lane + 32 * j < E) wpart[warp * (E + 1) + lane + 32 * j] = make_float2(pm[j], ps[j]);
  __syncthreads();
  for (int i = warp; i < E; i += kCapWarps) {
    float2 v = wpart[lane * (E + 1) + i];
    lse_butterfly(v.x, v.y, 32);
    if (lane == 0) part_out[((int64_t)g * E + i) * bpg + blk] = v;     // expert-major: the row step reads along the CTAs
  }
}
// The same as words.  wpart was last read before the barrier of the row step in between, so one barrier is enough.
template <int EPL>
__device__ __forceinline__ void publish_words(const float (&pm)[EPL], const float (&ps)[EPL], float2* wpart, int E, const Exchange& x,
                                              int pass, int g, int bpg, int blk) {
  const int warp = threadIdx.x >> 5, lane = threadIdx.x & 31;
#ifdef EC_DEBUG
  if (pass > 0 && blk == x.silent) return;
#endif
  if (pass == 0) {
#pragma unroll
    for (int j = 0; j < EPL; ++j) if (lane + 32 * j < E) wpart[warp * (E + 1) + lane + 32 * j] = make_float2(pm[j], ps[j]);
    __syncthreads();
    for (int i = warp; i < E; i += kCapWarps) {
      float2 v = wpart[lane * (E + 1) + i];
      lse_butterfly(v.x, v.y, 32);
      if (lane == 0) {
        word_store(x.first_max + ((int64_t)g * E + i) * bpg + blk, v.x, 0u);
        word_store(x.first_sum + ((int64_t)g * E + i) * bpg + blk, v.y, 0u);
      }
    }
    return;
  }
  float* sums = reinterpret_cast<float*>(wpart);     // [warps][E + 1]; with E even the odd pitch keeps the banks apart
  const int pitch = E | 1;
#pragma unroll
  for (int j = 0; j < EPL; ++j) if (lane + 32 * j < E) sums[warp * pitch + lane + 32 * j] = ps[j];
  __syncthreads();
  constexpr int kRows = EPL >= 8 ? 4 : EPL;          // experts a warp joins side by side (it has at most EPL of them)
  for (int i0 = warp; i0 < E; i0 += kRows * kCapWarps) {
    float v[kRows];
#pragma unroll
    for (int u = 0; u < kRows; ++u) v[u] = i0 + u * kCapWarps < E ? sums[lane * pitch + i0 + u * kCapWarps] : 0.f;
#pragma unroll
    for (int o = 16; o > 0; o >>= 1)
#pragma unroll
      for (int u = 0; u < kRows; ++u) v[u] += __shfl_xor_sync(0xffffffffu, v[u], o);
    if (lane == 0) {
#pragma unroll
      for (int u = 0; u < kRows; ++u)
        if (i0 + u * kCapWarps < E) word_store(((pass & 1) ? x.odd : x.even) + ((int64_t)g * E + i0 + u * kCapWarps) * bpg + blk, v[u], (unsigned)pass);
    }
  }
}

// One token, one round after the row step: columns, then the box.  x: log A of the token's experts held by this
// lane (already shifted by the row step), qb / qc: log correction factors.  Returns nothing; updates in place.
template <int EPL>
__device__ __forceinline__ void token_round(float (&x)[EPL], float (&qb)[EPL], float& qc, int lane, int E, float log_b) {
  // After the row step every entry is at most k (its row sums to k), so exp cannot overflow and the column sum
  // needs no shift by the maximum; a column so small that the sum underflows is far below b and stays as it is.
  float sum = 0.f;
#pragma unroll
  for (int j = 0; j < EPL; ++j) if (lane + 32 * j < E) sum += __expf(x[j]);
#pragma unroll
  for (int o = 16; o > 0; o >>= 1) sum += __shfl_xor_sync(0xffffffffu, sum, o);
  const float m = fminf(0.f, log_b - (__logf(sum) + qc));             // a column above b is scaled down to b
#pragma unroll
  for (int j = 0; j < EPL; ++j) {
    if (lane + 32 * j < E) {
      const float B = x[j] + qc + m + qb[j];
      const float v = fminf(B, 0.f);                                 // entries above 1 are clipped
      qb[j] = B - v;
      x[j] = v;
    }
  }
  qc = -m;
}

// ---- one launch per round ------------------------------------------------------------------------
// phase 0: L = S / lambda and its row partials.  phase 1: one round (rows, columns, box) and the row
// partials of its result; `first` treats the correction factors as 1 without reading them, `last`
// also writes A = exp(L).
template <int EPL>
__global__ void __launch_bounds__(kCapThreads)
capped_round_kernel(const float* __restrict__ S, float* __restrict__ L, float* __restrict__ qb, float* __restrict__ qc,
                    float* __restrict__ A, const float2* __restrict__ part_in, float2* __restrict__ part_out,
                    int64_t ng, int E, float inv_lambda, float log_k, float log_b, int phase, int first, int last) {
  constexpr int kBatch = EPL >= 8 ? 1 : (EPL >= 4 ? 2 : kCapBatch);   // so that a batch fits the 64 registers of a thread
  extern __shared__ float2 cap_smem[];
  float* shift = shift_of(cap_smem, E);
  const int g = blockIdx.y, bpg = gridDim.x, blk = blockIdx.x;
  const int warp = threadIdx.x >> 5, lane = threadIdx.x & 31;
  float pm[EPL], ps[EPL];
#pragma unroll
  for (int j = 0; j < EPL; ++j) { pm[j] = 0.f; ps[j] = 0.f; }
  // A warp takes its tokens kBatch at a time: the loads of a batch are issued together (they do not depend on
  // the row sums, so the first batch's are in flight while the CTA combines the partials), the arithmetic
  // follows token by token in ascending order.
  const int64_t stride = (int64_t)bpg * kCapWarps;
  float x[kBatch][EPL], qbv[kBatch][EPL], qcv[kBatch];
  auto load_batch = [&](int64_t tb) {
#pragma unroll
    for (int u = 0; u < kBatch; ++u) {
      const int64_t t = tb + u * stride;
      const int64_t tok = (int64_t)g * ng + t, row = tok * E;
      qcv[u] = 0.f;
#pragma unroll
      for (int j = 0; j < EPL; ++j) {
        const int i = lane + 32 * j;
        const bool ok = t < ng && i < E;
        x[u][j] = !ok ? -INFINITY : (phase == 0 ? S[row + i] * inv_lambda : L[row + i]);
        qbv[u][j] = (ok && phase == 1 && !first) ? qb[row + i] : 0.f;
      }
      if (t < ng && phase == 1 && !first) qcv[u] = qc[tok];
    }
  };
  int64_t tb = (int64_t)blk * kCapWarps + warp;
  load_batch(tb);                                    // loads nothing for a warp without tokens
  if (phase == 1) row_shifts(part_in, g, bpg, E, log_k, shift);       // every thread of the CTA gets here
  while (tb < ng) {
#pragma unroll
    for (int u = 0; u < kBatch; ++u) {
      const int64_t t = tb + u * stride;
      if (t < ng) {                                                    // uniform across the warp
        const int64_t tok = (int64_t)g * ng + t, row = tok * E;
        if (phase == 1) {
#pragma unroll
          for (int j = 0; j < EPL; ++j) if (lane + 32 * j < E) x[u][j] += shift[lane + 32 * j];     // rows sum to k
          token_round<EPL>(x[u], qbv[u], qcv[u], lane, E, log_b);
          if (lane == 0) qc[tok] = qcv[u];
        }
#pragma unroll
        for (int j = 0; j < EPL; ++j) {
          const int i = lane + 32 * j;
          if (i < E) {
            L[row + i] = x[u][j];
            if (phase == 1) qb[row + i] = qbv[u][j];
            if (last) A[row + i] = __expf(x[u][j]);
            if (phase == 0) lse_add(pm[j], ps[j], x[u][j], 1.f);
            else ps[j] += __expf(x[u][j]);           // after a round: entries at most 1, row sums well above underflow
          }
        }
      }
    }
    tb += kBatch * stride;
    if (tb < ng) load_batch(tb);
  }
  publish_partials<EPL>(pm, ps, cap_smem, E, part_out, g, bpg, blk);
}

// ---- resident: all rounds in one cooperative launch ------------------------------------------------
// exp and log without the denormal ranges' extra instructions: an entry below 2^-126 counts as 0 in the sums
__device__ __forceinline__ float exp_ftz(float x) { float y; asm("ex2.approx.ftz.f32 %0, %1;" : "=f"(y) : "f"(x * 1.4426950408889634f)); return y; }
__device__ __forceinline__ float log_ftz(float x) { float y; asm("lg2.approx.ftz.f32 %0, %1;" : "=f"(y) : "f"(x)); return y * 0.6931471805599453f; }

// Sums of T values (a power of two) over the warp at once: lane l ends with the sum of value l mod T.  T - 1 + log2(32 / T)
// shuffles where T butterflies take 5 T.
template <int T>
__device__ __forceinline__ float warp_sums(float (&v)[T]) {
  const int lane = threadIdx.x & 31;
#pragma unroll
  for (int b = 1; b < T; b <<= 1) {
    const bool up = (lane & b) != 0;
#pragma unroll
    for (int i = 0; i < T / (2 * b); ++i) {
      const float give = up ? v[2 * i] : v[2 * i + 1], keep = up ? v[2 * i + 1] : v[2 * i];
      v[i] = keep + __shfl_xor_sync(0xffffffffu, give, b);
    }
  }
  float s = v[0];
#pragma unroll
  for (int o = T; o < 32; o <<= 1) s += __shfl_xor_sync(0xffffffffu, s, o);
  return s;
}

// ---- exchange inside a cluster -----------------------------------------------------------------
// The words above cost two hops through L2 a round.  Where one cluster of 8 or 16 CTAs holds a group, a round's sums stay in shared
// memory: expert i belongs to the CTA of rank i mod (cluster size); a CTA sends its sum there (st.async, which counts the bytes
// on a barrier), a warp of that CTA adds them up in order of rank and sends the shift to every CTA.  Two sets of everything, used in
// turn: nobody can be two passes ahead of a reader, since every pass waits for all CTAs' sums of the one before.  Pass 0 (maxima
// too) goes through the words.  583 tokens x 16 experts: 296 -> 197 us for 100 rounds.  Several clusters joined by one hop
// through L2 are slower than the words: 6435 x 32: 311 us with words, 395 with clusters, since the two hops inside the cluster take
// nearly as long as two through L2.
constexpr int kBoxRanks = 16, kBoxOwned = kCapMaxE / 8;
struct Box { float inbox[2][kBoxOwned][kBoxRanks]; float shift[2][kCapMaxE]; uint64_t inbox_bar[2], shift_bar[2]; };
__device__ __forceinline__ void send_async(const void* where, const void* bar, int rank, float v) {
  asm volatile("st.async.shared::cluster.mbarrier::complete_tx::bytes.b32 [%0], %1, [%2];"
               ::"r"(map_to_cta(smem_u32(where), (uint32_t)rank)), "r"(__float_as_uint(v)), "r"(map_to_cta(smem_u32(bar), (uint32_t)rank)) : "memory");
}
__device__ __forceinline__ bool box_try(uint32_t bar, uint32_t parity) {             // what came from other CTAs is visible behind it
  uint32_t ok;
  asm volatile("{\n .reg .pred p;\n mbarrier.try_wait.parity.acquire.cluster.shared::cta.b64 p, [%1], %2;\n selp.u32 %0, 1, 0, p;\n}\n"
               : "=r"(ok) : "r"(bar), "r"(parity) : "memory");
  return ok != 0;
}
__device__ __forceinline__ bool box_wait(const void* bar, uint32_t parity, unsigned long long wait_ns) {
  const uint32_t b = smem_u32(bar);
  if (box_try(b, parity)) return true;
  const unsigned long long t0 = cap_timer();
  for (unsigned spin = 1;; ++spin) {
    if (box_try(b, parity)) return true;
    if ((spin & 63u) == 0 && cap_timer() - t0 > wait_ns) return false;
  }
}
// The CTA's sums of pass `pass` (>= 1) to their owners; see publish_words
template <int EPL>
__device__ __forceinline__ void publish_box(const float (&ps)[EPL], float* sums, int E, Box& box, int pass, int rank, int ranks, const Exchange& x) {
  const int warp = threadIdx.x >> 5, lane = threadIdx.x & 31;
#ifdef EC_DEBUG
  if (rank == x.silent) return;
#endif
  const int pitch = E | 1;
#pragma unroll
  for (int j = 0; j < EPL; ++j) if (lane + 32 * j < E) sums[warp * pitch + lane + 32 * j] = ps[j];
  __syncthreads();
  constexpr int kRows = EPL >= 8 ? 4 : EPL;
  for (int i0 = warp; i0 < E; i0 += kRows * kCapWarps) {
    float v[kRows];
#pragma unroll
    for (int u = 0; u < kRows; ++u) v[u] = i0 + u * kCapWarps < E ? sums[lane * pitch + i0 + u * kCapWarps] : 0.f;
#pragma unroll
    for (int o = 16; o > 0; o >>= 1)
#pragma unroll
      for (int u = 0; u < kRows; ++u) v[u] += __shfl_xor_sync(0xffffffffu, v[u], o);
    if (lane == 0) {
#pragma unroll
      for (int u = 0; u < kRows; ++u) {
        const int i = i0 + u * kCapWarps;
        if (i < E) send_async(&box.inbox[pass & 1][i / ranks][rank], &box.inbox_bar[pass & 1], i % ranks, v[u]);
      }
    }
  }
}
// The shifts of pass `pass` (>= 1) in box.shift[pass & 1]; false for the whole CTA when a wait ran out
__device__ __forceinline__ bool shifts_box(Box& box, const Exchange& x, int pass, int rank, int ranks, int E, float log_k) {
  const int warp = threadIdx.x >> 5, lane = threadIdx.x & 31, par = pass & 1;
  const uint32_t phase = (uint32_t)((pass - 1) >> 1) & 1u;
  const int own = (E - rank + ranks - 1) / ranks;                      // experts rank, rank + ranks, ...: at most one per warp
  if (threadIdx.x == 0) {
    mbar_expect_tx(smem_u32(&box.inbox_bar[par]), (uint32_t)(own * ranks * 4));
    mbar_expect_tx(smem_u32(&box.shift_bar[par]), (uint32_t)(E * 4));
  }
  bool ok = true;
  if (warp < own) {
    ok = __all_sync(0xffffffffu, box_wait(&box.inbox_bar[par], phase, x.wait_ns));
    float s = 0.f;
    for (int r = 0; r < ranks; ++r) s += box.inbox[par][warp][r];
    if (ok && lane < ranks) send_async(&box.shift[par][warp * ranks + rank], &box.shift_bar[par], lane, log_k - __logf(s));
  }
  if (ok) ok = box_wait(&box.shift_bar[par], phase, x.wait_ns);
  if (__syncthreads_and(ok)) return true;
  if (threadIdx.x == 0) { atomicExch(x.status + 1, 8); atomicExch(x.status, 5 /* EC_ERR_TIMEOUT */); }
  return false;
}

// Needs ng <= TPW * gridDim.x * warps per CTA and all CTAs on the device at once.  A warp works on its TPW tokens side by
// side: their column sums share one set of shuffles, lane l keeps the column factor of token l mod TPW and one
// logarithm serves all of them.  exp(L) of the previous round times exp(shift) is exp(L) after the row step, so an entry costs one
// exponential a round.  Places without a token or an expert hold kNowhere, whose exponential is 0 and stays 0.
// 16384 tokens x 64 experts, cycles of a round: one token after the other with two exponentials an entry 4.1 k, this form 1.25 k.
constexpr float kNowhere = -1e30f;
template <int EPL, int TPW, bool CLUSTER>
__global__ void __launch_bounds__(kCapThreads)
capped_resident_kernel(const float* __restrict__ S, float* __restrict__ A, const Exchange ex, int64_t ng, int E,
                       float inv_lambda, float log_k, float log_b, int iters) {
  extern __shared__ float2 cap_smem[];
  float* shift = shift_of(cap_smem, E);
  __shared__ Box box[1];                             // (the compiler drops it where nothing uses it)
  const int g = blockIdx.y, bpg = gridDim.x, blk = blockIdx.x;
  if constexpr (CLUSTER) {
    if (threadIdx.x == 0) {
      for (int p = 0; p < 2; ++p) { mbar_init(smem_u32(&box[0].inbox_bar[p]), 1); mbar_init(smem_u32(&box[0].shift_bar[p]), 1); }
      asm volatile("fence.mbarrier_init.release.cluster;" ::: "memory");
    }
    __syncthreads();
    cluster_sync_all();                              // nobody sends before every barrier of the cluster is there
  }
  const int warp = threadIdx.x >> 5, lane = threadIdx.x & 31;
  const int64_t stride = (int64_t)bpg * kCapWarps, t0 = (int64_t)blk * kCapWarps + warp;
  float x[TPW][EPL], ea[TPW][EPL], qb[TPW][EPL], qc = 0.f, pm[EPL], ps[EPL];
#pragma unroll
  for (int j = 0; j < EPL; ++j) { pm[j] = 0.f; ps[j] = 0.f; }
#pragma unroll
  for (int u = 0; u < TPW; ++u) {
    const int64_t t = t0 + u * stride, row = ((int64_t)g * ng + t) * E;
#pragma unroll
    for (int j = 0; j < EPL; ++j) {
      const int i = lane + 32 * j;
      qb[u][j] = 0.f; ea[u][j] = 0.f;
      x[u][j] = (t < ng && i < E) ? S[row + i] * inv_lambda : kNowhere;
      if (t < ng && i < E) lse_add(pm[j], ps[j], x[u][j], 1.f);
    }
  }
  publish_words<EPL>(pm, ps, cap_smem, E, ex, 0, g, bpg, blk);
  bool whole = true;                                 // no wait ran out
  for (int it = 0; it < iters; ++it) {
    const float* now = shift;
    if (CLUSTER && it > 0) {
      if (!(whole = shifts_box(box[0], ex, it, blk, bpg, E, log_k))) break;
      now = box[0].shift[it & 1];
    } else if (!(whole = row_shifts(ex, it, g, bpg, blk, E, log_k, shift))) {
      break;
    }
    float sh[EPL], es[EPL], sum[TPW];
#pragma unroll
    for (int j = 0; j < EPL; ++j) { ps[j] = 0.f; sh[j] = lane + 32 * j < E ? now[lane + 32 * j] : 0.f; es[j] = exp_ftz(sh[j]); }
#pragma unroll
    for (int u = 0; u < TPW; ++u) {
      sum[u] = 0.f;
#pragma unroll
      for (int j = 0; j < EPL; ++j) {
        x[u][j] += sh[j];                            // rows sum to k
        // After the row step every entry is at most k, so nothing overflows and the column sum needs no shift by the
        // maximum; a column so small that the sum underflows is far below b and stays as it is.
        sum[u] += it == 0 ? exp_ftz(x[u][j]) : ea[u][j] * es[j];
      }
    }
    const float total = warp_sums<TPW>(sum);
    const float m = fminf(0.f, log_b - (log_ftz(total) + qc));         // a column above b is scaled down to b
    const float mq = m + qc;
    qc = -m;
#pragma unroll
    for (int u = 0; u < TPW; ++u) {
      const float c = __shfl_sync(0xffffffffu, mq, u);
#pragma unroll
      for (int j = 0; j < EPL; ++j) {
        const float Bv = x[u][j] + c + qb[u][j];
        x[u][j] = fminf(Bv, 0.f);                    // entries above 1 are clipped
        qb[u][j] = Bv - x[u][j];
        ea[u][j] = exp_ftz(x[u][j]);
        ps[j] += ea[u][j];
      }
    }
    if (it + 1 < iters) {
      if constexpr (CLUSTER) publish_box<EPL>(ps, reinterpret_cast<float*>(cap_smem), E, box[0], it + 1, blk, bpg, ex);
      else publish_words<EPL>(pm, ps, cap_smem, E, ex, it + 1, g, bpg, blk);
    }
  }
  if constexpr (CLUSTER) {                           // nothing is on its way to a CTA that has left
    if (!whole) { const unsigned long long t1 = cap_timer(); while (cap_timer() - t1 < 100000ull) __nanosleep(1000); }       // what nobody waited for lands
    __syncwarp();
    cluster_sync_all();
  }
#pragma unroll
  for (int u = 0; u < TPW; ++u) {
    const int64_t t = t0 + u * stride, row = ((int64_t)g * ng + t) * E;
#pragma unroll
    for (int j = 0; j < EPL; ++j) if (t < ng && lane + 32 * j < E) A[row + lane + 32 * j] = whole ? __expf(x[u][j]) : 0.f;
  }
}

// The same with the state in shared memory instead of registers, for groups whose tokens do not fit the registers:
// behind wpart and shift come log A and the box factors of the warp's tokens ([warp][token][2][E]) and the column
// factors ([warp][token]).  A warp touches only its own part, so no barrier guards it.
template <int EPL>
__global__ void __launch_bounds__(kCapThreads)
capped_resident_smem_kernel(const float* __restrict__ S, float* __restrict__ A, const Exchange ex, int64_t ng, int E, float inv_lambda, float log_k, float log_b,
                            int iters, int tpw) {
  extern __shared__ float2 cap_smem[];
  float* shift = shift_of(cap_smem, E);
  const int g = blockIdx.y, bpg = gridDim.x, blk = blockIdx.x;
  const int warp = threadIdx.x >> 5, lane = threadIdx.x & 31;
  const int64_t stride = (int64_t)bpg * kCapWarps, t0 = (int64_t)blk * kCapWarps + warp;
  float* mine = shift + E + (size_t)warp * tpw * 2 * E;            // this warp's tokens: [token][log A | box factor][E]
  float* my_qc = shift + E + (size_t)kCapWarps * tpw * 2 * E + warp * tpw;
  float pm[EPL], ps[EPL];
#pragma unroll
  for (int j = 0; j < EPL; ++j) { pm[j] = 0.f; ps[j] = 0.f; }
  for (int u = 0; u < tpw; ++u) {
    const int64_t t = t0 + u * stride, row = ((int64_t)g * ng + t) * E;
    if (t < ng) {                                    // uniform across the warp
#pragma unroll
      for (int j = 0; j < EPL; ++j) {
        const int i = lane + 32 * j;
        if (i < E) {
          const float v = S[row + i] * inv_lambda;
          mine[(2 * u) * E + i] = v; mine[(2 * u + 1) * E + i] = 0.f;
          lse_add(pm[j], ps[j], v, 1.f);
        }
      }
      if (lane == 0) my_qc[u] = 0.f;
    }
  }
  publish_words<EPL>(pm, ps, cap_smem, E, ex, 0, g, bpg, blk);
  bool whole = true;                                 // no wait ran out
  for (int it = 0; it < iters; ++it) {
    if (!(whole = row_shifts(ex, it, g, bpg, blk, E, log_k, shift))) break;
#pragma unroll
    for (int j = 0; j < EPL; ++j) { pm[j] = 0.f; ps[j] = 0.f; }
    for (int u = 0; u < tpw; ++u) {
      if (t0 + u * stride < ng) {                    // uniform across the warp
        float x[EPL], qb[EPL];
#pragma unroll
        for (int j = 0; j < EPL; ++j) {
          const int i = lane + 32 * j;
          x[j] = i < E ? mine[(2 * u) * E + i] + shift[i] : -INFINITY;                               // rows sum to k
          qb[j] = i < E ? mine[(2 * u + 1) * E + i] : 0.f;
        }
        float qc = my_qc[u];
        __syncwarp();                                // every lane has read the column factor before lane 0 rewrites it
        token_round<EPL>(x, qb, qc, lane, E, log_b);
        if (lane == 0) my_qc[u] = qc;
#pragma unroll
        for (int j = 0; j < EPL; ++j) {
          const int i = lane + 32 * j;
          if (i < E) { mine[(2 * u) * E + i] = x[j]; mine[(2 * u + 1) * E + i] = qb[j]; ps[j] += __expf(x[j]); }
        }
      }
    }
    if (it + 1 < iters) publish_words<EPL>(pm, ps, cap_smem, E, ex, it + 1, g, bpg, blk);
  }
  for (int u = 0; u < tpw; ++u) {
    const int64_t t = t0 + u * stride, row = ((int64_t)g * ng + t) * E;
#pragma unroll
    for (int j = 0; j < EPL; ++j) if (t < ng && lane + 32 * j < E) A[row + lane + 32 * j] = whole ? __expf(mine[(2 * u) * E + lane + 32 * j]) : 0.f;
  }
}

__global__ void gather_gate_kernel(const float* __restrict__ S, const int32_t* __restrict__ I, float* __restrict__ G,
                                   int64_t slots_total, int64_t k, int E, int64_t n, int* status) {
  chain_enter();
  S = after_enter(S); I = after_enter(I);
  for (int64_t s = (int64_t)blockIdx.x * blockDim.x + threadIdx.x; s < slots_total; s += (int64_t)gridDim.x * blockDim.x) {
    const int t = I[s];
    G[s] = idx_ok(t, 0, n, status) ? S[(int64_t)t * E + (int)(s / k)] : 0.f;
  }
}

int blocks_per_group(int64_t ng, int groups, int sms) {
  int64_t b = sms / groups;
  const int64_t most = (ng + kCapWarps - 1) / kCapWarps;            // at least one token per warp
  if (b > most) b = most;
  return (int)(b < 1 ? 1 : b);
}
// The partials are sized for the largest grid any device could ask for, so the layout does not depend on the device.
constexpr int kCapMaxBlocks = 1024;

size_t align256(size_t b) { return (b + 255) & ~(size_t)255; }
size_t cap_smem_bytes(int E) { return (size_t)kCapWarps * (E + 1) * 8 + (size_t)E * 4; }      // at most 65.3 KiB

struct ResidentArgs {
  const float* S; float* A; Exchange ex; int64_t ng; int E; float inv_lambda, log_k, log_b; int iters;
};
// no word carries a pass number: one left by an earlier call could carry a number this call waits for
cudaError_t exchange_clear(const ResidentArgs& a, dim3 grid, cudaStream_t st) {
  return cudaMemsetAsync(a.ex.first_max, 0xFF, Exchange::words(grid.x, grid.y, a.E) * sizeof(unsigned long long), st);
}
// One cluster of `ranks` CTAs per group.  *fits: the device holds them all at once
template <int EPL, int TPW>
cudaError_t launch_cluster(ResidentArgs a, int ranks, int groups, size_t room, bool* fits, cudaStream_t st) {
  *fits = false;
  auto kern = capped_resident_kernel<EPL, TPW, true>;
  const size_t smem = cap_smem_bytes(a.E), words = Exchange::words(ranks, groups, a.E);
  if (words > room) return cudaSuccess;
  if (cudaFuncSetAttribute(kern, cudaFuncAttributeMaxDynamicSharedMemorySize, 66 * 1024) != cudaSuccess ||
      cudaFuncSetAttribute(kern, cudaFuncAttributeNonPortableClusterSizeAllowed, 1) != cudaSuccess) return cudaErrorInvalidValue;
  cudaLaunchAttribute attr[2];
  attr[0].id = cudaLaunchAttributeClusterDimension;
  attr[0].val.clusterDim.x = (unsigned)ranks; attr[0].val.clusterDim.y = 1; attr[0].val.clusterDim.z = 1;
  attr[1].id = cudaLaunchAttributeCooperative;
  attr[1].val.cooperative = 1;
  cudaLaunchConfig_t cfg = {};
  cfg.gridDim = dim3((unsigned)ranks, (unsigned)groups); cfg.blockDim = dim3(kCapThreads); cfg.dynamicSmemBytes = smem; cfg.stream = st;
  cfg.attrs = attr; cfg.numAttrs = 1;
  int most = 0;
  if (cudaOccupancyMaxActiveClusters(&most, kern, &cfg) != cudaSuccess) { cudaGetLastError(); return cudaSuccess; }
  if (most < groups) return cudaSuccess;
  a.ex = Exchange::at(a.ex.first_max, ranks, groups, a.E, a.ex.status, a.ex.wait_ns, a.ex.silent);
  const cudaError_t e = cudaMemsetAsync(a.ex.first_max, 0xFF, words * sizeof(unsigned long long), st);
  if (e != cudaSuccess) return e;
  cfg.numAttrs = 2;
  *fits = true;
  count_launch();
  return cudaLaunchKernelEx(&cfg, kern, a.S, a.A, a.ex, a.ng, a.E, a.inv_lambda, a.log_k, a.log_b, a.iters);
}
// As few tokens a warp as eight CTAs allow, then sixteen
template <int EPL>
cudaError_t launch_cluster_tpw(ResidentArgs a, int groups, size_t room, bool* fits, cudaStream_t st) {
  constexpr int kMost = kCapResident / EPL;
  const int64_t at_once = (int64_t)8 * kCapWarps;
  *fits = false;
  if constexpr (kMost >= 4) if (a.ng <= at_once * (kMost / 4)) return launch_cluster<EPL, kMost / 4>(a, 8, groups, room, fits, st);
  if constexpr (kMost >= 2) if (a.ng <= at_once * (kMost / 2)) return launch_cluster<EPL, kMost / 2>(a, 8, groups, room, fits, st);
  if (a.ng <= at_once * kMost) return launch_cluster<EPL, kMost>(a, 8, groups, room, fits, st);
  if (a.ng <= at_once * kMost * 2) return launch_cluster<EPL, kMost>(a, 16, groups, room, fits, st);
  return cudaSuccess;
}
template <int EPL, int TPW>
cudaError_t launch_resident(ResidentArgs a, dim3 grid, int sms, bool* fits, cudaStream_t st) {
  auto kern = capped_resident_kernel<EPL, TPW, false>;
  const size_t smem = cap_smem_bytes(a.E);
  if (smem > 48 * 1024 && cudaFuncSetAttribute(kern, cudaFuncAttributeMaxDynamicSharedMemorySize, 66 * 1024) != cudaSuccess)
    return cudaErrorInvalidValue;
  int per_sm = 0;
  if (cudaOccupancyMaxActiveBlocksPerMultiprocessor(&per_sm, kern, kCapThreads, smem) != cudaSuccess) return cudaErrorInvalidValue;
  *fits = (int64_t)per_sm * sms >= (int64_t)grid.x * grid.y;         // the CTAs wait for one another: all on the device at once
  if (!*fits) return cudaSuccess;
  const cudaError_t e = exchange_clear(a, grid, st);
  if (e != cudaSuccess) return e;
  void* args[] = {&a.S, &a.A, &a.ex, &a.ng, &a.E, &a.inv_lambda, &a.log_k, &a.log_b, &a.iters};
  count_launch();
  return cudaLaunchCooperativeKernel((void*)kern, grid, dim3(kCapThreads), args, smem, st);
}
template <int EPL>
cudaError_t launch_resident_tpw(int tpw, ResidentArgs a, dim3 grid, int sms, bool* fits, cudaStream_t st) {
  if constexpr (EPL <= 8) if (tpw <= 1) return launch_resident<EPL, 1>(a, grid, sms, fits, st);
  if constexpr (EPL <= 4) if (tpw <= 2) return launch_resident<EPL, 2>(a, grid, sms, fits, st);
  if constexpr (EPL <= 2) if (tpw <= 4) return launch_resident<EPL, 4>(a, grid, sms, fits, st);
  if constexpr (EPL <= 1) if (tpw <= 8) return launch_resident<EPL, 8>(a, grid, sms, fits, st);
  *fits = false;
  return cudaSuccess;
}

constexpr size_t kCapSmemLimit = 200 * 1024;         // of a CTA's 227 KiB
template <int EPL>
cudaError_t launch_resident_smem(ResidentArgs a, int tpw, dim3 grid, int sms, bool* fits, cudaStream_t st) {
  auto kern = capped_resident_smem_kernel<EPL>;
  const size_t smem = cap_smem_bytes(a.E) + (size_t)kCapWarps * tpw * (2 * a.E + 1) * 4;
  *fits = false;
  if (smem > kCapSmemLimit) return cudaSuccess;
  if (cudaFuncSetAttribute(kern, cudaFuncAttributeMaxDynamicSharedMemorySize, (int)kCapSmemLimit) != cudaSuccess) return cudaErrorInvalidValue;
  int per_sm = 0;
  if (cudaOccupancyMaxActiveBlocksPerMultiprocessor(&per_sm, kern, kCapThreads, smem) != cudaSuccess) return cudaErrorInvalidValue;
  *fits = (int64_t)per_sm * sms >= (int64_t)grid.x * grid.y;
  if (!*fits) return cudaSuccess;
  const cudaError_t e = exchange_clear(a, grid, st);
  if (e != cudaSuccess) return e;
  void* args[] = {&a.S, &a.A, &a.ex, &a.ng, &a.E, &a.inv_lambda, &a.log_k, &a.log_b, &a.iters, &tpw};
  count_launch();
  return cudaLaunchCooperativeKernel((void*)kern, grid, dim3(kCapThreads), args, smem, st);
}

}  // namespace

// scratch: L [n, E] | qb [n, E] | qc [n] | two sets of row partials
size_t capped_scratch_bytes(int64_t n, int E, int groups) {
  const size_t blocks = (size_t)(groups > kCapMaxBlocks ? groups : kCapMaxBlocks);
  return 2 * align256((size_t)n * E * 4) + align256((size_t)n * 4) + 2 * align256(blocks * E * sizeof(float2));
}

cudaError_t launch_capped_assignment(const float* S, int64_t ng, int E, int64_t kg, int groups, int b, int iters,
                                     float lambda, float* A, void* scratch, int* status, cudaStream_t st, unsigned long long wait_ns,
                                     int silent_cta) {
  if (E > kCapMaxE || iters < 1 || b < 1 || !(lambda > 0.f)) return cudaErrorInvalidValue;
  const int64_t n = ng * groups;
  char* p = (char*)scratch;
  float* L = (float*)p; p += align256((size_t)n * E * 4);
  float* qb = (float*)p; p += align256((size_t)n * E * 4);
  float* qc = (float*)p; p += align256((size_t)n * 4);
  const size_t blocks = (size_t)(groups > kCapMaxBlocks ? groups : kCapMaxBlocks);
  float2* part[2] = {(float2*)p, (float2*)(p + align256(blocks * E * sizeof(float2)))};
  int dev = 0, sms = 148, coop = 0;
  cudaGetDevice(&dev);
  cudaDeviceGetAttribute(&sms, cudaDevAttrMultiProcessorCount, dev);
  cudaDeviceGetAttribute(&coop, cudaDevAttrCooperativeLaunch, dev);
  int bpg = blocks_per_group(ng, groups, sms);
  if ((int64_t)bpg * groups > (int64_t)blocks) bpg = (int)(blocks / groups);
  const dim3 grid(bpg, groups);
  // the words of the resident forms take the place of the two sets of partials
  const size_t room = 2 * align256(blocks * E * sizeof(float2)) / sizeof(unsigned long long);
  if (Exchange::words(bpg, groups, E) > room) coop = 0;
  const Exchange ex = Exchange::at(reinterpret_cast<unsigned long long*>(part[0]), bpg, groups, E, status, wait_ns, silent_cta);
  const float inv_lambda = 1.f / lambda, log_k = logf((float)kg), log_b = logf((float)b);
  const int epl = E <= 32 ? 1 : (E <= 64 ? 2 : (E <= 128 ? 4 : 8));
  const int64_t tpw = (ng + (int64_t)bpg * kCapWarps - 1) / ((int64_t)bpg * kCapWarps);
  if (coop && iters > 1) {                           // one pass alone goes through the words anyway
    ResidentArgs a{S, A, ex, ng, E, inv_lambda, log_k, log_b, iters};
    bool fits = false;
    const cudaError_t e = epl == 1 ? launch_cluster_tpw<1>(a, groups, room, &fits, st) : epl == 2 ? launch_cluster_tpw<2>(a, groups, room, &fits, st)
                        : epl == 4 ? launch_cluster_tpw<4>(a, groups, room, &fits, st) : launch_cluster_tpw<8>(a, groups, room, &fits, st);
    if (e != cudaSuccess || fits) return e;
  }
  if (coop && tpw * epl <= kCapResident) {
    ResidentArgs a{S, A, ex, ng, E, inv_lambda, log_k, log_b, iters};
    bool fits = false;
    cudaError_t e = epl == 1 ? launch_resident_tpw<1>((int)tpw, a, grid, sms, &fits, st)
                  : epl == 2 ? launch_resident_tpw<2>((int)tpw, a, grid, sms, &fits, st)
                  : epl == 4 ? launch_resident_tpw<4>((int)tpw, a, grid, sms, &fits, st)
                             : launch_resident_tpw<8>((int)tpw, a, grid, sms, &fits, st);
    if (e != cudaSuccess) return e;
    if (fits) return cudaGetLastError();
  }
  if (coop && tpw * epl > kCapResident && tpw <= 1024) {             // too many entries for registers: try shared memory
    ResidentArgs a{S, A, ex, ng, E, inv_lambda, log_k, log_b, iters};
    bool fits = false;
    cudaError_t e = epl == 1 ? launch_resident_smem<1>(a, (int)tpw, grid, sms, &fits, st)
                  : epl == 2 ? launch_resident_smem<2>(a, (int)tpw, grid, sms, &fits, st)
                  : epl == 4 ? launch_resident_smem<4>(a, (int)tpw, grid, sms, &fits, st)
                             : launch_resident_smem<8>(a, (int)tpw, grid, sms, &fits, st);
    if (e != cudaSuccess) return e;
    if (fits) return cudaGetLastError();
  }
  const size_t smem = cap_smem_bytes(E);
  if (smem > 48 * 1024 &&                            // E > 180: more than the default limit
      cudaFuncSetAttribute(capped_round_kernel<8>, cudaFuncAttributeMaxDynamicSharedMemorySize, 66 * 1024) != cudaSuccess)
    return cudaErrorInvalidValue;
  auto round = [&](int phase, int first, int last, const float2* in, float2* out) {
    count_launch();
    if (E <= 32) capped_round_kernel<1><<<grid, kCapThreads, smem, st>>>(S, L, qb, qc, A, in, out, ng, E, inv_lambda, log_k, log_b, phase, first, last);
    else if (E <= 64) capped_round_kernel<2><<<grid, kCapThreads, smem, st>>>(S, L, qb, qc, A, in, out, ng, E, inv_lambda, log_k, log_b, phase, first, last);
    else if (E <= 128) capped_round_kernel<4><<<grid, kCapThreads, smem, st>>>(S, L, qb, qc, A, in, out, ng, E, inv_lambda, log_k, log_b, phase, first, last);
    else capped_round_kernel<8><<<grid, kCapThreads, smem, st>>>(S, L, qb, qc, A, in, out, ng, E, inv_lambda, log_k, log_b, phase, first, last);
  };
  round(0, 0, 0, nullptr, part[0]);
  for (int it = 0; it < iters; ++it) round(1, it == 0, it == iters - 1, part[it & 1], part[(it + 1) & 1]);
  return cudaGetLastError();
}

cudaError_t launch_gather_gate(const float* S, const int32_t* I, float* G, int64_t slots_total, int64_t k, int E,
                               int64_t n, int* status, cudaStream_t st) {
  const int64_t blocks = (slots_total + 255) / 256;
  return launch_chained(gather_gate_kernel, dim3((unsigned)(blocks > 1184 ? 1184 : blocks)), dim3(256), 0, st, S, I, G, slots_total, k, E, n, status);
}

}  // namespace ecmoe
