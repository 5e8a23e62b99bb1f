// Plain FMA batched GEMM with arbitrary element strides and the layer's fused epilogues.
// It is the arithmetic of the fp32 path's gate gradients and of its small expert products (the others run on the tensor cores
// in three bf16 pieces, gemm_f32_tc.cu) and, with one bf16 operand, of the gate gradients whose expert count the tcgen05
// kernel does not take.  fp32 accumulation throughout: every result is one chain of fused multiply-adds in ascending k, or, where a tile's contraction is shared by two groups of threads
// (KS = 2: they take its k-tiles in turn), the sum of two such chains.
//
// A CTA computes a BM x BN tile, a thread TM x TN results of it (groups of four rows and four columns, so that every
// fragment is a 16-byte shared-memory load).  Bound by the FMA pipe at the layer's sizes and by the latency of a k-tile
// where there are fewer tiles than SMs, so:
//   - the multiply-adds are packed pairs (fma.rn.f32x2: the same two roundings, half the instructions to issue);
//   - the next k-tile travels from global memory to registers while the current one is computed and lands in the other
//     of two shared buffers: one barrier per k-tile, no load latency in the open;
//   - both tiles lie [k][m] and [k][n], whatever the storage order.  A column is XOR-ed with a function of k that spreads the
//     scalar stores of a transposed tile over all 32 banks and keeps groups of four together.
// At n = 2048, d = 512, d' = 2048, 16 experts (8.6 GFLOP per expert product) a product takes 174-207 us here, 42-50 TFLOP/s of the
// 74 the FMA pipe has; the 64 x 64 tile with 4 x 4 results per thread, one buffer and scalar loads that this replaces
// took 445-640 us.  What is left, from the counters: the FMA pipe is busy 75 % of the time in the plain 128 x 128 tile and the
// shared-memory pipe 48 % (two CTAs of four warps on an SM do not cover all of each other's fragment loads and barriers),
// 70 % with 128 tiles on 148 SMs, 60 and 53 % where GeLU and GeLU' (erff) follow in the open; 512 tiles on 296 places
// leave the second round 0.73 full.
#include "internal.h"

namespace ecmoe {

namespace {

__device__ __forceinline__ float ldv(const float* p, int64_t i) { return p[i]; }
__device__ __forceinline__ float ldv(const bf16* p, int64_t i) { return __bfloat162float(p[i]); }
__device__ __forceinline__ void stv(float* p, int64_t i, float v) { p[i] = v; }
__device__ __forceinline__ void stv(bf16* p, int64_t i, float v) { p[i] = __float2bfloat16(v); }
// four consecutive elements (the address a multiple of four elements)
__device__ __forceinline__ void ldv4(const float* p, int64_t i, float (&f)[4]) {
  const float4 v = *reinterpret_cast<const float4*>(p + i); f[0] = v.x; f[1] = v.y; f[2] = v.z; f[3] = v.w;
}
__device__ __forceinline__ void ldv4(const bf16* p, int64_t i, float (&f)[4]) {
  const uint2 v = *reinterpret_cast<const uint2*>(p + i);
  f[0] = __uint_as_float(v.x << 16); f[1] = __uint_as_float(v.x & 0xFFFF0000u);
  f[2] = __uint_as_float(v.y << 16); f[3] = __uint_as_float(v.y & 0xFFFF0000u);
}
__device__ __forceinline__ void stv4(float* p, int64_t i, const float (&f)[4]) {
  *reinterpret_cast<float4*>(p + i) = make_float4(f[0], f[1], f[2], f[3]);
}
__device__ __forceinline__ void stv4(bf16* p, int64_t i, const float (&f)[4]) {
  __nv_bfloat162 a = __floats2bfloat162_rn(f[0], f[1]), b = __floats2bfloat162_rn(f[2], f[3]);
  *reinterpret_cast<uint2*>(p + i) = make_uint2(*reinterpret_cast<unsigned*>(&a), *reinterpret_cast<unsigned*>(&b));
}

__device__ __forceinline__ unsigned long long pair2(float a, float b) {
  return (unsigned long long)__float_as_uint(a) | ((unsigned long long)__float_as_uint(b) << 32);
}
__device__ __forceinline__ unsigned long long fma_pair(unsigned long long a, unsigned long long b, unsigned long long c) {
  unsigned long long d; asm("fma.rn.f32x2 %0, %1, %2, %3;" : "=l"(d) : "l"(a), "l"(b), "l"(c)); return d;
}

// How an operand's tile is fetched: which storage direction is contiguous and whether four elements along it can be
// taken at once (their address is 16 (fp32) or 8 (bf16) byte aligned and they are all inside or all outside).
struct Operand { int k_fast, vec; };

// An operand as the kernel sees it: p(r, k) = p[r * sr + k * sk], rows r in [0, rows), depth k in [0, kb).  A list replaces the
// row index or, with list_k, the depth.
template <typename T>
struct Source { const T* p; int64_t sr, sk; int rows, kb; const int32_t* list; int list_k; int64_t list_total; int* status; };

// One operand's share of a k-tile: ROWS x BK elements, held in registers between the load and the store to shared memory.
// Elements outside [0, rows) x [0, kb) are zero.  VEC: only operands with `vec` set come here.
template <typename T, int ROWS, int BK, int NT, bool VEC>
struct TileLoader {
  static constexpr int kQuads = ROWS * BK / 4 / NT;
  static_assert(ROWS * BK % (4 * NT) == 0, "whole quads per thread");
  static constexpr int kSwz = 32 / (BK / 4);          // see sw()
  float v[kQuads][4];
  const T* at[kQuads];                                // this thread's quads at the next k-tile
  bool in[kQuads];                                    // the quad's (first) row exists
  unsigned keep[kQuads];                              // which of the four loaded elements exist; the others become zero in store()

  // column of row r at depth k: an XOR by a multiple of four below 32
  static __device__ __forceinline__ int sw(int k, int r) { return r ^ (((k >> 2) & (BK / 4 - 1)) * kSwz); }

  // quad q: k_fast: four consecutive k of one row; else four consecutive rows at one k
  static __device__ __forceinline__ void where(int q, int k_fast, int& r, int& k) {
    const int idx = threadIdx.x % NT + q * NT;
    if (k_fast) { r = idx / (BK / 4); k = (idx % (BK / 4)) * 4; } else { r = (idx % (ROWS / 4)) * 4; k = idx / (ROWS / 4); }
  }
  __device__ __forceinline__ void init(const Source<T>& s, const Operand o, int r0, int k0) {
#pragma unroll
    for (int q = 0; q < kQuads; ++q) {
      int r, k; where(q, o.k_fast, r, k);
      r += r0; k += k0;
      int64_t ri = r;
      in[q] = r < s.rows;
      if (VEC && s.list && !s.list_k && in[q]) {
        const int sel = s.list[r];
        in[q] = idx_ok(sel, 0, s.list_total, s.status);
        ri = sel;
      }
      at[q] = in[q] ? s.p + ri * s.sr + (VEC && s.list_k ? 0 : (int64_t)k * s.sk) : s.p;
    }
  }
  // Loads the k-tile at k0; a thread asks for its k-tiles in order, `step` elements of k apart, from init's k0 on.  No
  // branch: what lies outside is read at the operand's first element and dropped, so that all loads are in flight together.
  __device__ __forceinline__ void load(const Source<T>& s, const Operand o, int r0, int k0, int step) {
#pragma unroll
    for (int q = 0; q < kQuads; ++q) {
      int r, k; where(q, o.k_fast, r, k);
      k += k0;
      if constexpr (VEC) {
        bool ok = in[q] && k < s.kb;
        const T* p = at[q];
        if (s.list_k) {                               // the rows of k are picked one by one; the four lie along r
          const int sel = s.list[k < s.kb ? k : 0];
          ok = ok && idx_ok(sel, 0, s.list_total, s.status);
          p += ok ? (int64_t)sel * s.sk : 0;
        } else {
          at[q] += step * s.sk;
        }
        ldv4(ok ? p : s.p, 0, v[q]);
        keep[q] = ok ? 15u : 0u;
      } else {
        const int64_t along = o.k_fast ? s.sk : s.sr;
#pragma unroll
        for (int j = 0; j < 4; ++j) {
          const bool ok = o.k_fast ? in[q] && k + j < s.kb : r0 + r + j < s.rows && k < s.kb;
          v[q][j] = ldv(ok ? at[q] + j * along : s.p, 0);
          keep[q] = j == 0 ? (ok ? 1u : 0u) : keep[q] | (ok ? 1u << j : 0u);
        }
        at[q] += step * s.sk;
      }
    }
  }
  __device__ __forceinline__ void store(float* tile, const Operand o) const {
#pragma unroll
    for (int q = 0; q < kQuads; ++q) {
      int r, k; where(q, o.k_fast, r, k);
      float x[4];
#pragma unroll
      for (int j = 0; j < 4; ++j) x[j] = (VEC ? keep[q] != 0u : (keep[q] >> j & 1u) != 0u) ? v[q][j] : 0.f;
      if (o.k_fast) {
#pragma unroll
        for (int j = 0; j < 4; ++j) tile[(k + j) * ROWS + sw(k, r)] = x[j];          // k is a multiple of four: one swizzle for all
      } else {
        *reinterpret_cast<float4*>(tile + k * ROWS + sw(k, r)) = make_float4(x[0], x[1], x[2], x[3]);
      }
    }
  }
};

template <typename TA, typename TB, typename TC, int EPI, int BM, int BN, int BK, int TM, int TN, int KS, int MINB, bool VEC>
__global__ void __launch_bounds__(BM / TM * (BN / TN) * KS, MINB) gemm_simt_kernel(const GemmArgs g, const Operand oa, const Operand ob, int c_vec) {
  constexpr int NT = BM / TM * (BN / TN), TX = BN / TN, GM = TM / 4, GN = TN / 4;
  static_assert(TX % 8 == 0 && TM % 4 == 0 && TN % 4 == 0, "a warp covers 4 x 8 threads");
  using LA = TileLoader<TA, BM, BK, NT, VEC>;
  using LB = TileLoader<TB, BN, BK, NT, VEC>;
  chain_enter(g.early);
  constexpr int kBuf = BK * (BM + BN);                // one k-tile of both operands
  extern __shared__ __align__(16) float simt_smem[];  // [KS groups][2 buffers][A | B]; after the main loop the other groups' sums
  const int b = blockIdx.z, grp = threadIdx.x / NT;
  float* bufs = simt_smem + grp * 2 * kBuf;
  const int m0 = blockIdx.x * BM, n0 = blockIdx.y * BN;     // row tiles on grid.x: M (tokens) is the dimension without a limit
  const int warp = (threadIdx.x % NT) >> 5, lane = threadIdx.x & 31;
  const int tx = (lane & 7) + 8 * (warp % (TX / 8)), ty = (lane >> 3) + 4 * (warp / (TX / 8));
  unsigned long long acc[TM][TN / 2];
#pragma unroll
  for (int i = 0; i < TM; ++i)
#pragma unroll
    for (int j = 0; j < TN / 2; ++j) acc[i][j] = 0ull;
  int Kb = g.K;
  if (g.k_limit > 0) { const int64_t left = g.k_limit - (int64_t)b * g.K; Kb = (int)(left < g.K ? (left > 0 ? left : 0) : g.K); }
  const Source<TA> sa = {(const TA*)g.A + (g.a_rows ? 0 : (int64_t)b * g.batch_a), g.sam, g.sak, g.M, Kb,
                         g.a_rows ? g.a_rows + (int64_t)b * g.a_rows_batch : nullptr, g.a_rows ? g.a_rows_k : 0, g.a_rows_total, g.status};
  const Source<TB> sb = {(const TB*)g.B + (int64_t)b * g.batch_b, g.sbn, g.sbk, g.N, Kb, nullptr, 0, 0, nullptr};
  LA la; LB lb;
  la.init(sa, oa, m0, grp * BK); lb.init(sb, ob, n0, grp * BK);
  auto fetch = [&](int t) { la.load(sa, oa, m0, t * BK, KS * BK); lb.load(sb, ob, n0, t * BK, KS * BK); };
  auto put = [&](float* buf) { la.store(buf, oa); lb.store(buf + BK * BM, ob); };
  auto group_sync = [&] { if constexpr (KS == 1) __syncthreads(); else asm volatile("bar.sync %0, %1;" ::"r"(1 + grp), "n"(NT) : "memory"); };
  const int kt = (Kb + BK - 1) / BK;                  // k-tiles; the groups take them in turn
  if (grp < kt) {
    fetch(grp);
    put(bufs);
    group_sync();
  }
  int cur = 0;
  for (int t = grp; t < kt; t += KS, cur ^= 1) {
    const float* as = bufs + cur * kBuf;
    const float* bs = as + BK * BM;
    if (t + KS < kt) fetch(t + KS);
#pragma unroll
    for (int kk = 0; kk < BK; ++kk) {
      if (TM == 4 && kk % 8 == 0 && kk > 0 && t * BK + kk >= Kb) break;           // the rest of the last k-tile is zeros
      float a[TM]; unsigned long long bb[TN / 2];
#pragma unroll
      for (int i = 0; i < GM; ++i) {
        const float4 v = *reinterpret_cast<const float4*>(as + kk * BM + LA::sw(kk, i * (BM / GM) + ty * 4));
        a[4 * i] = v.x; a[4 * i + 1] = v.y; a[4 * i + 2] = v.z; a[4 * i + 3] = v.w;
      }
#pragma unroll
      for (int j = 0; j < GN; ++j) {
        const ulonglong2 v = *reinterpret_cast<const ulonglong2*>(bs + kk * BN + LB::sw(kk, j * (BN / GN) + tx * 4));
        bb[2 * j] = v.x; bb[2 * j + 1] = v.y;
      }
#pragma unroll
      for (int i = 0; i < TM; ++i) {
        const unsigned long long aa = pair2(a[i], a[i]);
#pragma unroll
        for (int j = 0; j < TN / 2; ++j) acc[i][j] = fma_pair(aa, bb[j], acc[i][j]);
      }
    }
    if (t + KS < kt) {                                // the other buffer was last read before the previous barrier
      put(bufs + (cur ^ 1) * kBuf);
      group_sync();
    }
  }
  if constexpr (KS > 1) {                             // the groups' sums join in ascending order
    __syncthreads();
    float2* part = reinterpret_cast<float2*>(simt_smem);               // [TM * TN / 2][NT], one group at a time
    for (int s = 1; s < KS; ++s) {
      if (grp == s) {
#pragma unroll
        for (int i = 0; i < TM; ++i)
#pragma unroll
          for (int j = 0; j < TN / 2; ++j)
            part[(i * (TN / 2) + j) * NT + threadIdx.x % NT] = make_float2(__uint_as_float((unsigned)acc[i][j]), __uint_as_float((unsigned)(acc[i][j] >> 32)));
      }
      __syncthreads();
      if (grp == 0) {
#pragma unroll
        for (int i = 0; i < TM; ++i)
#pragma unroll
          for (int j = 0; j < TN / 2; ++j) {
            const float2 o = part[(i * (TN / 2) + j) * NT + threadIdx.x];
            acc[i][j] = pair2(__uint_as_float((unsigned)acc[i][j]) + o.x, __uint_as_float((unsigned)(acc[i][j] >> 32)) + o.y);
          }
      }
      __syncthreads();
    }
    if (grp != 0) { chain_leave(g.early); return; }
  }
  TC* C = g.C ? (TC*)g.C + (int64_t)b * g.batch_c : nullptr;
  // EPI_ADD_SLOTS: the lists of a thread's four rows are walked side by side, so that four rows of `rows` are in flight
  auto row_of = [&](int i) { return m0 + (i / 4) * (BM / GM) + ty * 4 + i % 4; };
#pragma unroll
  for (int i0 = 0; i0 < TM; i0 += 4) {
    int qa[4], qb[4];
    if constexpr (EPI == EPI_ADD_SLOTS) {
      int* st = n0 + tx == 0 ? g.status : nullptr;    // one thread of a row's records a bad index
#pragma unroll
      for (int u = 0; u < 4; ++u) {
        const int m = min(row_of(i0 + u), g.M - 1);
        qa[u] = g.row_ptr[m]; qb[u] = g.row_ptr[m + 1];
      }
#pragma unroll
      for (int u = 0; u < 4; ++u)
        if (row_of(i0 + u) >= g.M || !idx_ok(qa[u], 0, g.slots_total + 1, st) || !idx_ok(qb[u], qa[u], g.slots_total + 1, st)) qa[u] = qb[u] = 0;
    }
#pragma unroll
    for (int j = 0; j < GN; ++j) {
      const int n = n0 + j * (BN / GN) + tx * 4;
      if (n >= g.N) continue;
      const int left = min(4, g.N - n);               // 4 whenever c_vec
      float v[4][4];
#pragma unroll
      for (int u = 0; u < 4; ++u)
#pragma unroll
        for (int e = 0; e < 2; ++e) {
          const unsigned long long p = acc[i0 + u][2 * j + e];
          v[u][2 * e] = __uint_as_float((unsigned)p); v[u][2 * e + 1] = __uint_as_float((unsigned)(p >> 32));
        }
      if (g.bias) {
#pragma unroll
        for (int e = 0; e < 4; ++e) {
          const float bv = e < left ? ldv((const TC*)g.bias, (int64_t)b * g.N + n + e) : 0.f;
#pragma unroll
          for (int u = 0; u < 4; ++u) v[u][e] += bv;
        }
      }
      if constexpr (EPI == EPI_ADD_SLOTS) {
        const TC* rows = (const TC*)g.rows;
        for (int q = 0;; ++q) {
          bool any = false;
          int sid[4];
#pragma unroll
          for (int u = 0; u < 4; ++u) {
            sid[u] = qa[u] + q < qb[u] ? g.slots[qa[u] + q] : -1;
            any |= qa[u] + q < qb[u];
          }
          if (!any) break;
          float x[4][4];
#pragma unroll
          for (int u = 0; u < 4; ++u) {
            if (sid[u] >= 0 && !idx_ok(sid[u], 0, g.slots_total, n == 0 ? g.status : nullptr)) sid[u] = -1;
            const int64_t ro = (int64_t)(sid[u] < 0 ? 0 : sid[u]) * g.ld_rows + n;
            if (c_vec) ldv4(rows, ro, x[u]);
            else {
#pragma unroll
              for (int e = 0; e < 4; ++e) x[u][e] = ldv(rows, ro + (e < left ? e : 0));
            }
          }
#pragma unroll
          for (int u = 0; u < 4; ++u)
            if (sid[u] >= 0)
#pragma unroll
              for (int e = 0; e < 4; ++e) v[u][e] += x[u][e];
        }
      }
#pragma unroll
      for (int u = 0; u < 4; ++u) {
        const int m = row_of(i0 + u);
        if (m >= g.M) continue;
        const int64_t o = (int64_t)m * g.ldc + n;
        if constexpr (EPI == EPI_GELU) {
          float h[4];
#pragma unroll
          for (int e = 0; e < 4; ++e) h[e] = gelu_fwd(v[u][e], g.gelu);
          TC* H = (TC*)g.C2 + (int64_t)b * g.batch_c;
          if (c_vec) stv4(H, o, h); else for (int e = 0; e < left; ++e) stv(H, o + e, h[e]);
        } else if constexpr (EPI == EPI_GELU_GRAD) {
          const TC* Z = (const TC*)g.Zin + (int64_t)b * g.batch_c;
          float z[4] = {0.f, 0.f, 0.f, 0.f};
          if (c_vec) ldv4(Z, o, z); else for (int e = 0; e < left; ++e) z[e] = ldv(Z, o + e);
#pragma unroll
          for (int e = 0; e < 4; ++e) v[u][e] *= gelu_bwd(z[e], g.gelu);
        }
        if (C) { if (c_vec) stv4(C, o, v[u]); else for (int e = 0; e < left; ++e) stv(C, o + e, v[u][e]); }   // EPI_GELU without C: only GeLU(acc) is wanted
      }
    }
  }
  chain_leave(g.early);
}

// Column tiles sit on grid.y.  64 columns cover every width the layer takes (2^22 - 64), 32 columns the widths below 2 097 121.
// (Several launches with a column offset do it too, but one more kernel argument changed the code of the tiles that every
// layer uses: an fp32 step of 531 us took 541.)
constexpr int kMaxColTiles = 65535;

enum Tile { TILE_128x128, TILE_128x128_K2, TILE_64x64_K2, TILE_64x32 };
// The SM with the most tiles decides: its multiply-adds at the rate the tile reaches (share of the 128 per cycle), or its
// k-tiles one after the other where too few warps hide their latency.  Rates measured on the three products of the
// layer above (8.6 GFLOP each; 512, 128 and 512 tiles of 128 x 128): 194, 233 and 174 us with the plain 128 x 128 tile,
// 207, 206 and 196 us with its contraction cut in two, the better one where there is a tile per SM at most (the second
// product); 236-298 us with 64 x 64 and 262 us with 64 x 32 tiles, which win by their number on small problems.
// Against the best of the four on 34 other sizes (k 12-1813, d 32-1024, d' 32-4096, 1 to 32 experts; 102 products): the same
// or within 4.4 % in nine of ten, 1.29 times the best at worst (k = 1219, d = 164, d' = 2924, 4 experts: H . W2^T in 64 x 32
// tiles 218 us, in 64 x 64 169).
Tile pick_tile(const GemmArgs& g, int sms, double* cycles) {
  struct Form { Tile id; int bm, bn, kstep, per_sm; double alone, full; };
  static const Form forms[] = {{TILE_128x128, 128, 128, 16, 2, 0.61, 0.80}, {TILE_128x128_K2, 128, 128, 32, 1, 0.70, 0.70},
                               {TILE_64x64_K2, 64, 64, 32, 3, 0.45, 0.60}, {TILE_64x32, 64, 32, 32, 4, 0.35, 0.52}};
  constexpr double kLatency = 1000.;                  // cycles of a k-tile nobody hides
  Tile best = TILE_64x32; double least = 0.;
  for (const Form& f : forms) {
    if ((g.N + f.bn - 1) / f.bn > kMaxColTiles) continue;
    const int64_t tiles = (((int64_t)g.M + f.bm - 1) / f.bm) * ((g.N + f.bn - 1) / f.bn) * g.batches, q = (tiles + sms - 1) / sms;
    const double work = (double)q * f.bm * f.bn * g.K / 128. / (q >= f.per_sm ? f.full : f.alone);
    const double steps = (double)((q + f.per_sm - 1) / f.per_sm) * ((g.K + f.kstep - 1) / f.kstep) * kLatency;
    const double t = work > steps ? work : steps;
    if (least == 0. || t < least) { least = t; best = f.id; }
  }
  *cycles = least;
  return best;
}

template <typename TA, typename TB, typename TC, int EPI, int BM, int BN, int BK, int TM, int TN, int KS, int MINB, bool VEC>
cudaError_t launch_tile(const GemmArgs& g, const Operand& oa, const Operand& ob, int c_vec, cudaStream_t st) {
  const dim3 grid((unsigned)(((int64_t)g.M + BM - 1) / BM), (g.N + BN - 1) / BN, g.batches);
  if (grid.y > (unsigned)kMaxColTiles || grid.z > 65535u) return cudaErrorInvalidConfiguration;
  auto kern = gemm_simt_kernel<TA, TB, TC, EPI, BM, BN, BK, TM, TN, KS, MINB, VEC>;
  constexpr int bufs = KS * 2 * BK * (BM + BN) * 4, sums = KS > 1 ? BM * BN * 4 : 0, smem = bufs > sums ? bufs : sums;
  if (smem > 48 * 1024) {
    const cudaError_t e = cudaFuncSetAttribute(kern, cudaFuncAttributeMaxDynamicSharedMemorySize, smem);
    if (e != cudaSuccess) return e;
  }
  return launch_chained(kern, grid, dim3(BM / TM * (BN / TN) * KS), smem, st, g, oa, ob, c_vec);
}

// Operands whose groups of four straddle an edge (an expert count that is not a multiple of four, in the gate's gradients
// only) are loaded one element at a time, in the small tile.  No list (a_rows) and no GeLU comes here: the products that
// have them contract rows of whole 16-byte vectors.
template <typename TA, typename TB, typename TC, int EPI>
cudaError_t launch_odd(const GemmArgs& g, const Operand& oa, const Operand& ob, int c_vec, cudaStream_t st) {
  if constexpr (EPI == EPI_ADD_SLOTS) {               // the one product whose columns are the layer's width
    if (g.N > 32 * kMaxColTiles) return launch_tile<TA, TB, TC, EPI, 64, 64, 16, 8, 8, 2, 3, false>(g, oa, ob, c_vec, st);
  }
  return launch_tile<TA, TB, TC, EPI, 64, 32, 32, 4, 4, 1, 4, false>(g, oa, ob, c_vec, st);
}
template <int EPI>
cudaError_t launch_f32(const GemmArgs& g, Tile tile, const Operand& oa, const Operand& ob, int c_vec, cudaStream_t st) {
  switch (tile) {
    case TILE_128x128: return launch_tile<float, float, float, EPI, 128, 128, 16, 8, 16, 1, 2, true>(g, oa, ob, c_vec, st);
    case TILE_128x128_K2: return launch_tile<float, float, float, EPI, 128, 128, 16, 8, 16, 2, 1, true>(g, oa, ob, c_vec, st);
    case TILE_64x64_K2: return launch_tile<float, float, float, EPI, 64, 64, 16, 8, 8, 2, 3, true>(g, oa, ob, c_vec, st);
    case TILE_64x32: return launch_tile<float, float, float, EPI, 64, 32, 32, 4, 4, 1, 4, true>(g, oa, ob, c_vec, st);
  }
  return cudaErrorInvalidValue;
}

inline bool aligned4(const void* p, int dtype) { return ((uintptr_t)p & (dtype == 0 ? 15 : 7)) == 0; }

}  // namespace

cudaError_t launch_gemm_simt(const GemmArgs& g, cudaStream_t st) {
  if (g.M < 1 || g.N < 1 || g.batches < 1) return cudaErrorInvalidValue;
  int dev = 0, sms = 148;
  cudaGetDevice(&dev);
  cudaDeviceGetAttribute(&sms, cudaDevAttrMultiProcessorCount, dev);
  // Four elements at a time along the contiguous direction: every address is then a multiple of four elements, and a group
  // never straddles the end of that direction.  With k_limit the contraction ends where the last split does.
  auto operand = [&](const void* p, int dtype, int64_t sr, int64_t sk, int64_t batch, int64_t rows, bool list_contiguous) {
    Operand o;
    o.k_fast = sk == 1 ? 1 : 0;
    const int64_t ld = o.k_fast ? sr : sk, len = o.k_fast ? g.K : rows, lim = o.k_fast ? g.k_limit : 0;
    o.vec = (o.k_fast || sr == 1) && !list_contiguous && aligned4(p, dtype) && ld % 4 == 0 && len % 4 == 0 && lim % 4 == 0 &&
            (g.batches == 1 || batch % 4 == 0);
    return o;
  };
  const bool a_list_contig = g.a_rows && ((g.sak == 1) == (g.a_rows_k != 0));
  const Operand oa = operand(g.A, g.a_dtype, g.sam, g.sak, g.a_rows ? 0 : g.batch_a, g.M, a_list_contig);
  const Operand ob = operand(g.B, g.b_dtype, g.sbn, g.sbk, g.batch_b, g.N, false);
  auto out4 = [&](const void* p) { return p == nullptr || aligned4(p, g.c_dtype); };
  const int c_vec = g.N % 4 == 0 && g.ldc % 4 == 0 && (g.batches == 1 || g.batch_c % 4 == 0) && out4(g.C) && out4(g.C2) && out4(g.Zin) &&
                    out4(g.rows) && g.ld_rows % 4 == 0;
  if (g.bias && g.bias_dtype != g.c_dtype) return cudaErrorInvalidValue;
  if (g.a_rows && !(oa.vec && ob.vec)) return cudaErrorInvalidValue;         // the scalar tile does not read through a list
  if (g.a_dtype == 0 && g.b_dtype == 0 && g.c_dtype == 0) {
    if (oa.vec && ob.vec) {
      double fma_cycles; int cols = 0;
      const Tile tile = pick_tile(g, sms, &fma_cycles);
      // The tensor cores where their estimate is the lower one.  They win from a few k-blocks and tiles on: 205 against 67 us at
      // 256 x 512 x 2048 (16 experts), 14.7 against 12.9 at 58 x 584 x 180 (10); with few rows or a short or lonely contraction
      // a tile of multiply-adds is over sooner: 16.3 against 17.0 at 8 x 128 x 384 (24), 21.0 against 23.1 at 40 x 200 x 600 (16).
      const double tc_cycles = c_vec ? plan_gemm_f32_tc(g, sms, &cols) : -1.;
      if (tc_cycles >= 0. && tc_cycles < fma_cycles) {
        const cudaError_t e = launch_gemm_f32_tc(g, cols, sms, st);
        if (e != cudaErrorNotSupported) return e;    // else nothing was launched
      }
      switch (g.epi) {
        case EPI_STORE: return launch_f32<EPI_STORE>(g, tile, oa, ob, c_vec, st);
        case EPI_GELU: return launch_f32<EPI_GELU>(g, tile, oa, ob, c_vec, st);
        case EPI_GELU_GRAD: return launch_f32<EPI_GELU_GRAD>(g, tile, oa, ob, c_vec, st);
        case EPI_ADD_SLOTS: return launch_f32<EPI_ADD_SLOTS>(g, tile, oa, ob, c_vec, st);
      }
    } else {
      switch (g.epi) {
        case EPI_STORE: return launch_odd<float, float, float, EPI_STORE>(g, oa, ob, c_vec, st);
        case EPI_ADD_SLOTS: return launch_odd<float, float, float, EPI_ADD_SLOTS>(g, oa, ob, c_vec, st);
      }
    }
  }
  // the gate gradients of the bf16 path with an expert count that is not a multiple of 8 (dL stays fp32); every other
  // product of that path has rows of whole 16-byte vectors and runs on the tensor cores
  if (g.a_dtype == 1 && g.b_dtype == 0 && g.c_dtype == 0 && g.epi == EPI_STORE)
    return launch_odd<bf16, float, float, EPI_STORE>(g, oa, ob, c_vec, st);
  if (g.a_dtype == 0 && g.b_dtype == 1 && g.c_dtype == 1 && g.epi == EPI_ADD_SLOTS)
    return launch_odd<float, bf16, bf16, EPI_ADD_SLOTS>(g, oa, ob, c_vec, st);
  return cudaErrorInvalidValue;
}

}  // namespace ecmoe
