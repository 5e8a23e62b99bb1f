// fp32 expert products on the tensor cores.
//
// An fp32 value is the sum of three bf16 values, x = h + m + l: h is x rounded to bf16, m what is left rounded, l the rest,
// which fits eight bits.  The pieces are those of 2^24 x, so that the lowest bit of the smallest x is still a normal bf16 number, and
// the sums are multiplied by 2^-48 at the end: both exact.  What this range does not hold at the other end (|x| from 2^104, sums
// from 2^80, infinities) comes out infinite or NaN, and every such element is taken again by multiply-adds from global memory
// (take_again): the result is then the multiply-add kernel's.  A product of two such sums is taken as six of its nine terms,
//
//     a b  =  ah bh + (ah bm + am bh) + (am bm + ah bl + al bh)  +  terms below 2^-26 of |a b|,
//
// each exact in the multiplier of a tcgen05.mma.  What an accumulation in tensor memory rounds away (the unit truncates) is
// kept small in two ways: the five small terms of a k-block go in first, the large one last, and a k-block (64 of K) is all that
// is accumulated there; the running sums over k-blocks are fp32 registers of the epilogue warps, added with the usual rounding.
// Against 64 bits, 2-norm, 75 products of 25 layers (k 8-2048, d 32-768, d' 64-3072): 0.5e-7 to 1.5e-7, the chains of
// multiply-adds of gemm_simt_kernel 0.5e-7 to 8.2e-7 and in none of them less than this.
//
// One persistent CTA per SM, 20 warps, the registers shared out by role:
//   warps 0..7    add every finished k-block to the running sums (FN / 2 columns of 32 rows a warp: tensor memory is a ring of
//                 512 / FN buffers), then run the epilogue, through a 4 KiB staging buffer per warp that turns rows into
//                 coalesced lines;
//   warps 8..15   load the next k-block of both operands from global memory (16-byte loads, all in flight together), split it
//                 and store the six planes with the 128-byte swizzle, in the operand's own orientation (K-major or MN-major);
//   warp 16       one thread issues the 24 MMAs of a k-block (warps 17..19 only complete its register group).
// Two stages of 96 KiB (128 x 128 tile).  Bound by the SM's shared-memory and L1 data path: the MMAs read 192 KiB of operands a
// k-block, the planes are 96 KiB of stores and the loads pass 64 KiB twice, 3.3 k cycles in all, where the MMAs alone take
// 1.7 k.  At 2048 tokens, 512 x 2048, 16 experts (8.6 GFLOP a product): 67-71 us a product, 166-206 us with multiply-adds.
#include "internal.h"
#include "tc_ptx.cuh"

namespace ecmoe {

namespace {

constexpr int FM = 128, FK = 64;
constexpr int kAddWarps = 8, kSplitWarps = 8, kF32Threads = 32 * (kAddWarps + kSplitWarps + 4);
// 640 threads are launched with 96 registers (61440); the adding and splitting warps take 112 each, the last group keeps 32: as many
constexpr int kLaunchRegs = 96, kBusyRegs = 112, kIssueRegs = 32;
static_assert(32 * (kAddWarps + kSplitWarps) * kBusyRegs + 128 * kIssueRegs <= kF32Threads * kLaunchRegs, "no warp waits for registers that nobody gives back");
constexpr int kStages = 2, kStageOut = 4096;         // staging per epilogue warp: 32 rows x 128 bytes
__host__ __device__ constexpr int plane_bytes(int rows) { return rows * FK * 2; }
__host__ __device__ constexpr int f32_stage_bytes(int fn) { return 3 * (plane_bytes(FM) + plane_bytes(fn)); }
__host__ __device__ constexpr int f32_smem_bytes(int fn) { return kStages * f32_stage_bytes(fn) + kAddWarps * kStageOut + 256 + 1024; }

// One operand as the splitting warps see it: element (r, k) at p[r * ld + k] (K-major) or p[k * ld + r].  A list replaces the
// index that ld multiplies.
struct Side { const float* p; int64_t ld; int rows, kb; const int32_t* list; int64_t list_total; int* status; };

constexpr float kScaleIn = 16777216.f, kScaleOut = 1.f / 281474976710656.f;          // 2^24, 2^-48

// 2^24 x = h + m + l for two values, packed
__device__ __forceinline__ unsigned bf2(float a, float b) {
  const __nv_bfloat162 v = __floats2bfloat162_rn(a, b);
  return *reinterpret_cast<const unsigned*>(&v);
}
__device__ __forceinline__ void split2(float a, float b, unsigned& h, unsigned& m, unsigned& l) {
  const unsigned long long x = mul2(pk2(a, b), pk2(kScaleIn, kScaleIn));
  a = lo2(x); b = hi2(x);
  h = bf2(a, b);
  a -= __uint_as_float(h << 16); b -= __uint_as_float(h & 0xFFFF0000u);
  m = bf2(a, b);
  a -= __uint_as_float(m << 16); b -= __uint_as_float(m & 0xFFFF0000u);
  l = bf2(a, b);
}

// Sixteen bytes of global memory, or zeros; no branch, so that all loads of a thread are in flight together.
__device__ __forceinline__ float4 load4_if(const float* p, bool ok) {
  float4 v;
  asm volatile("{\n .reg .pred p;\n setp.ne.u32 p, %5, 0;\n mov.b32 %0, 0f00000000;\n mov.b32 %1, 0f00000000;\n mov.b32 %2, 0f00000000;\n mov.b32 %3, 0f00000000;\n"
               " @p ld.global.L1::no_allocate.v4.f32 {%0, %1, %2, %3}, [%4];\n}\n"
               : "=&f"(v.x), "=&f"(v.y), "=&f"(v.z), "=&f"(v.w) : "l"(p), "r"((unsigned)ok) : "memory");
  return v;
}

// A thread's share of an operand's k-block: Q groups of four elements along the contiguous direction, so that a warp's load is
// two runs of 256 bytes.  (Groups of eight per thread make each load touch eight lines with half of every sector: asking for a
// k-block then takes 2400 cycles, longer than its MMAs.)  A 128-byte row of the shared image holds 64 elements of that
// direction; four elements g4 of row r lie at r * 128 + (((g4 / 2) ^ (r & 7)) << 4) + (g4 & 1) * 8.  K-major: row r is the
// operand's row r; MN-major: rows 64 b .. 64 b + 63 are the 64 depths of the operand's rows 64 b .. 64 b + 63.
template <int ROWS, bool K_MAJOR, bool LIST>
struct SplitLoader {
  static constexpr int Q = ROWS * 16 / (kSplitWarps * 32), RP = kSplitWarps * 2;     // image rows of one go of all threads
  float4 v[Q];
  int row[LIST && K_MAJOR ? Q : 1];                  // with a list: the groups' rows of the operand, -1 for none
  __device__ __forceinline__ void init(const Side& s, int r0, int tt) {
    if constexpr (LIST && K_MAJOR) {
#pragma unroll
      for (int q = 0; q < Q; ++q) {
        const int r = r0 + (tt >> 4) + RP * q;
        row[q] = r < s.rows ? s.list[r] : -1;
        if (r < s.rows && !idx_ok(row[q], 0, s.list_total, s.status)) row[q] = -1;
      }
    }
  }
  __device__ __forceinline__ void load(const Side& s, int r0, int k0, int tt) {
    const int g = (tt & 15) * 4;
    if constexpr (K_MAJOR) {
      const bool in = k0 + g < s.kb;
      const float* p = s.p + (LIST ? 0 : (int64_t)(r0 + (tt >> 4)) * s.ld) + k0 + g;
#pragma unroll
      for (int q = 0; q < Q; ++q) {
        if constexpr (LIST) v[q] = load4_if(p + row[q] * s.ld, in && row[q] >= 0);
        else { v[q] = load4_if(p, in && r0 + (tt >> 4) + RP * q < s.rows); p += RP * s.ld; }
      }
    } else {
      const float* p = s.p + (LIST ? 0 : (int64_t)(k0 + (tt >> 4)) * s.ld) + r0 + g;
      const int64_t step = RP * s.ld;
#pragma unroll
      for (int q = 0; q < Q; ++q) {
        const int k = k0 + (((tt >> 4) + RP * q) & 63), c = RP * q / 64 * 64;
        bool ok = r0 + g + c < s.rows && k < s.kb;
        if constexpr (LIST) {
          const int sel = ok ? s.list[k] : 0;
          ok = ok && idx_ok(sel, 0, s.list_total, s.status);
          v[q] = load4_if(p + sel * s.ld + c, ok);
        } else {
          v[q] = load4_if(p + (RP * q & 63) / RP * step + c, ok);
        }
      }
    }
  }
  __device__ __forceinline__ void store(uint8_t* planes, int tt) const {
    uint8_t* dst = planes + (tt >> 4) * 128 + ((((tt & 15) >> 1) ^ ((tt >> 4) & 7)) << 4) + (tt & 1) * 8;
#pragma unroll
    for (int q = 0; q < Q; ++q) {
      uint2 h, m, l;
      split2(v[q].x, v[q].y, h.x, m.x, l.x); split2(v[q].z, v[q].w, h.y, m.y, l.y);
      *reinterpret_cast<uint2*>(dst + q * (RP * 128)) = h;
      *reinterpret_cast<uint2*>(dst + q * (RP * 128) + plane_bytes(ROWS)) = m;
      *reinterpret_cast<uint2*>(dst + q * (RP * 128) + 2 * plane_bytes(ROWS)) = l;
    }
  }
};

// The MMAs of a k-block whose planes lie at `st` (A: h, m, l; B behind them), small terms first; `left` of K are left, what lies
// beyond is zeros.  A descriptor's low word moves by constants from MMA to MMA.
template <bool A_K, bool B_K, int FN>
__device__ __forceinline__ void issue_terms(uint32_t st, uint32_t d_tmem, int left) {
  constexpr int kAP = plane_bytes(FM), kBP = plane_bytes(FN);
  constexpr uint32_t idesc = (1u << 4) | (1u << 7) | (1u << 10) | ((A_K ? 0u : 1u) << 15) | ((B_K ? 0u : 1u) << 16) |
                             ((uint32_t)(FN >> 3) << 17) | ((uint32_t)(FM >> 4) << 24);
  constexpr uint32_t a_step = A_K ? 32 : 2048, b_step = B_K ? 32 : 2048;
  const uint64_t a0 = make_desc(st, A_K ? 16 : FK * 128, 1024), b0 = make_desc(st + 3 * kAP, B_K ? 16 : FK * 128, 1024);
  constexpr int kTermA[6] = {2, 0, 1, 1, 0, 0}, kTermB[6] = {0, 2, 1, 0, 1, 0};
#pragma unroll
  for (int t = 0; t < 6; ++t)
#pragma unroll
    for (int kk = 0; kk < FK / 16; ++kk)
      if (kk == 0 || kk * 16 < left) tc_mma(d_tmem, a0 + ((kTermA[t] * kAP + kk * a_step) >> 4), b0 + ((kTermB[t] * kBP + kk * b_step) >> 4), idesc, (t | kk) != 0);
}

// Four at once: the form is asked for once, not per value (a step of 2048 x 512 x 2048, 16 experts: 517 -> 501 us)
template <int FORM> __device__ __forceinline__ float4 gelu_fwd4(float4 v) {
  return make_float4(gelu_fwd(v.x, FORM), gelu_fwd(v.y, FORM), gelu_fwd(v.z, FORM), gelu_fwd(v.w, FORM));
}
template <int FORM> __device__ __forceinline__ float4 gelu_bwd4(float4 v) {
  return make_float4(gelu_bwd(v.x, FORM), gelu_bwd(v.y, FORM), gelu_bwd(v.z, FORM), gelu_bwd(v.w, FORM));
}

// What the pieces could not hold: the marked elements of row `row`, bit j for column n0 + j, by multiply-adds in ascending k, four columns
// at a time.  NaN four times ends a sum.  Not inlined: in the epilogue's own loop it costs a step 20 us, like this 4.
template <int EPI, bool A_K, bool B_K, bool LIST>
__device__ __noinline__ void take_again(const GemmArgs& g, int b, int row, int n0, unsigned long long bad) {
  if (row >= g.M) return;
  const float* A = (const float*)g.A + (LIST ? 0 : (int64_t)b * g.batch_a);
  const int32_t* list = LIST ? g.a_rows + (int64_t)b * g.a_rows_batch : nullptr;
  const int64_t lda = A_K ? g.sam : g.sak, ldb = B_K ? g.sbn : g.sbk;
  for (; bad != 0; bad >>= 4, n0 += 4) {
    if ((bad & 15ull) == 0 || n0 >= g.N) continue;
    const float* B = (const float*)g.B + (int64_t)b * g.batch_b + (B_K ? n0 * ldb : n0);
    float acc[4] = {0.f, 0.f, 0.f, 0.f};
#pragma unroll 4
    for (int k = 0; k < g.K; ++k) {
      int64_t line = A_K ? row : k;
      bool ok = true;
      if constexpr (LIST) { line = list[line]; ok = idx_ok(line, 0, g.a_rows_total, g.status); }
      const float a = ok ? A[line * lda + (A_K ? k : row)] : 0.f;
#pragma unroll
      for (int j = 0; j < 4; ++j) acc[j] = fmaf(a, B_K ? B[j * ldb + k] : B[k * ldb + j], acc[j]);
      if ((k & 63) == 63 && isnan(acc[0]) && isnan(acc[1]) && isnan(acc[2]) && isnan(acc[3])) break;
    }
    for (int j = 0; j < 4; ++j) {
      if (!(bad >> j & 1ull)) continue;
      const int64_t o = (int64_t)b * g.batch_c + (int64_t)row * g.ldc + n0 + j;
      float v = acc[j] + (g.bias ? ((const float*)g.bias)[(int64_t)b * g.N + n0 + j] : 0.f);
      if constexpr (EPI == EPI_GELU) ((float*)g.C2)[o] = gelu_fwd(v, g.gelu);
      if constexpr (EPI == EPI_GELU_GRAD) v *= gelu_bwd(((const float*)g.Zin)[o], g.gelu);
      if (g.C) ((float*)g.C)[o] = v;
    }
  }
}

template <int EPI, int FN, bool A_K, bool B_K, bool LIST>
__global__ void __launch_bounds__(kF32Threads, 1) gemm_f32_tc_kernel(const __grid_constant__ GemmArgs g, int tiles_m, int tiles_n, int total_tiles) {
  constexpr int kAP = plane_bytes(FM), kBP = plane_bytes(FN), kStage = f32_stage_bytes(FN);
  constexpr int kRing = 512 / FN, kCols = FN / 2;    // accumulator buffers; columns of an epilogue warp
  extern __shared__ uint8_t f32_smem[];
  uint8_t* smem = (uint8_t*)(((uintptr_t)f32_smem + 1023) & ~(uintptr_t)1023);
  uint64_t* bars = (uint64_t*)(smem + kStages * kStage + kAddWarps * kStageOut);     // full, empty [stages]; accumulator full, empty [ring]
  uint32_t* tmem_slot = (uint32_t*)(bars + 2 * kStages + 2 * kRing);
  volatile int* abort_flag = (volatile int*)(tmem_slot + 1);
  const uint32_t full0 = smem_u32(bars), empty0 = full0 + 8 * kStages, tfull0 = empty0 + 8 * kStages, tempty0 = tfull0 + 8 * kRing;
  const int warp = threadIdx.x >> 5, lane = threadIdx.x & 31;
  constexpr int kMmaWarp = kAddWarps + kSplitWarps;
  if (threadIdx.x == 0) {
    for (int s = 0; s < kStages; ++s) { mbar_init(full0 + 8 * s, kSplitWarps); mbar_init(empty0 + 8 * s, 1); }
    for (int b = 0; b < kRing; ++b) { mbar_init(tfull0 + 8 * b, 1); mbar_init(tempty0 + 8 * b, kAddWarps); }
    *abort_flag = 0;
    asm volatile("fence.mbarrier_init.release.cluster;" ::: "memory");
  }
  if (warp == kMmaWarp) {
    asm volatile("tcgen05.alloc.cta_group::1.sync.aligned.shared::cta.b32 [%0], %1;" ::"r"(smem_u32(tmem_slot)), "r"(512) : "memory");
    asm volatile("tcgen05.relinquish_alloc_permit.cta_group::1.sync.aligned;" ::: "memory");
  }
  tc_fence_before();
  __syncthreads();
  tc_fence_after();
  chain_enter(g.early);
  const uint32_t tmem_base = *tmem_slot;
  const int kblocks = (g.K + FK - 1) / FK;
  auto place = [&](int tile, int& b, int& m0, int& n0) {               // row tiles fastest: CTAs that run together share columns of B
    b = tile / (tiles_m * tiles_n); m0 = tile % tiles_m * FM; n0 = tile / tiles_m % tiles_n * FN;
  };

  
  if (warp >= kAddWarps && warp < kMmaWarp) {
    asm volatile("setmaxnreg.inc.sync.aligned.u32 %0;" ::"n"(kBusyRegs));
    const int tt = threadIdx.x - kAddWarps * 32;
    int stage = 0, tile = blockIdx.x, kb = 0, m0 = 0, n0 = 0; uint32_t phase = 0;
    Side sa, sb; SplitLoader<FM, A_K, LIST> la; SplitLoader<FN, B_K, false> lb;
    auto enter_tile = [&] {
      int b; place(tile, b, m0, n0);
      sa = {(const float*)g.A + (LIST ? 0 : (int64_t)b * g.batch_a), A_K ? g.sam : g.sak, g.M, g.K, LIST ? g.a_rows + (int64_t)b * g.a_rows_batch : nullptr,
            g.a_rows_total, g.status};
      sb = {(const float*)g.B + (int64_t)b * g.batch_b, B_K ? g.sbn : g.sbk, g.N, g.K, nullptr, 0, nullptr};
      la.init(sa, m0, tt);
    };
    bool more = tile < total_tiles;
    if (more) { enter_tile(); la.load(sa, m0, 0, tt); lb.load(sb, n0, 0, tt); }
    while (more) {
      const bool ok = mbar_wait(empty0 + 8 * stage, phase ^ 1, abort_flag, g.status, 1);
      if (!__all_sync(0xffffffffu, ok)) break;
      if (++kb == kblocks) { kb = 0; tile += gridDim.x; more = tile < total_tiles; if (more) enter_tile(); }     // the next k-block, maybe of the next tile
      uint8_t* st = smem + stage * kStage;
      la.store(st, tt);                              // A's next loads travel while B is split
      if (more) la.load(sa, m0, kb * FK, tt);
      lb.store(st + 3 * kAP, tt);
      fence_async_smem();
      __syncwarp();
      if (lane == 0) mbar_arrive(full0 + 8 * stage);
      if (more) lb.load(sb, n0, kb * FK, tt);
      if (++stage == kStages) { stage = 0; phase ^= 1; }
    }
  } else if (warp >= kMmaWarp) {
    asm volatile("setmaxnreg.dec.sync.aligned.u32 %0;" ::"n"(kIssueRegs));
    if (warp == kMmaWarp && lane == 0) {
      int stage = 0, buf = 0; uint32_t phase = 0, tphase = 0; bool gave_up = false;
      for (int tile = blockIdx.x; tile < total_tiles && !gave_up; tile += gridDim.x) {
#pragma unroll 1
        for (int kb = 0; kb < kblocks; ++kb) {
          if (!mbar_wait(tempty0 + 8 * buf, tphase ^ 1, abort_flag, g.status, 2) || !mbar_wait(full0 + 8 * stage, phase, abort_flag, g.status, 3)) { gave_up = true; break; }
          tc_fence_after();
          issue_terms<A_K, B_K, FN>(smem_u32(smem) + stage * kStage, tmem_base + buf * FN, g.K - kb * FK);
          tc_commit(empty0 + 8 * stage);
          tc_commit(tfull0 + 8 * buf);
          if (++stage == kStages) { stage = 0; phase ^= 1; }
          if (++buf == kRing) { buf = 0; tphase ^= 1; }
        }
      }
    }
  } else {
    asm volatile("setmaxnreg.inc.sync.aligned.u32 %0;" ::"n"(kBusyRegs));
    const int q = warp & 3, half = warp >> 2;
    uint8_t* stg = smem + kStages * kStage + warp * kStageOut;
    int buf = 0; uint32_t tphase = 0; bool gave_up = false;
    for (int tile = blockIdx.x; tile < total_tiles && !gave_up; tile += gridDim.x) {
      int b, m0, n0; place(tile, b, m0, n0);
      float acc[kCols];
#pragma unroll
      for (int j = 0; j < kCols; ++j) acc[j] = 0.f;
#pragma unroll 1
      for (int kb = 0; kb < kblocks; ++kb) {
        const bool ok = mbar_wait(tfull0 + 8 * buf, tphase, abort_flag, g.status, 4);
        if (!__all_sync(0xffffffffu, ok)) { gave_up = true; break; }
        tc_fence_after();
        const uint32_t t = tmem_base + ((uint32_t)(q * 32) << 16) + buf * FN + half * kCols;
#pragma unroll
        for (int c = 0; c < kCols; c += 32) {
          uint32_t r[32]; tc_ld32(t + c, r);
#pragma unroll
          for (int j = 0; j < 32; ++j) acc[c + j] += __uint_as_float(r[j]);
        }
        tc_fence_before();
        __syncwarp();
        if (lane == 0) mbar_arrive(tempty0 + 8 * buf);
        if (++buf == kRing) { buf = 0; tphase ^= 1; }
      }
      if (gave_up) break;
      unsigned long long zero = 0ull, bad = 0ull;    // zero: NaN as soon as one of this lane's elements is not finite; bad: which ones
#pragma unroll
      for (int j = 0; j < kCols; j += 2) zero = fma2(pk2(acc[j], acc[j + 1]), pk2(0.f, 0.f), zero);
      const bool redo = __any_sync(0xffffffffu, lo2(zero) + hi2(zero) != 0.f);
      if (redo) {
#pragma unroll
        for (int j = 0; j < kCols; ++j) bad |= (unsigned long long)!isfinite(acc[j]) << j;
      }
#pragma unroll
      for (int c = 0; c < kCols; c += 32) {
        // rows of 32 columns into the staging buffer (swizzled: no bank conflicts either way), back as lines: eight lanes a row
        const int n = n0 + half * kCols + c + (lane & 7) * 4, mr = m0 + q * 32 + (lane >> 3);
        float4 bias = make_float4(0.f, 0.f, 0.f, 0.f);
        if (g.bias && n < g.N) bias = *reinterpret_cast<const float4*>((const float*)g.bias + (int64_t)b * g.N + n);
#pragma unroll
        for (int j = 0; j < 8; ++j)
          *reinterpret_cast<float4*>(stg + lane * 128 + ((j ^ (lane & 7)) << 4)) = make_float4(acc[c + 4 * j], acc[c + 4 * j + 1], acc[c + 4 * j + 2], acc[c + 4 * j + 3]);
        __syncwarp();
        const int64_t o0 = (int64_t)b * g.batch_c + (int64_t)mr * g.ldc + n;
        auto z_at = [&](int i) {
          return mr + 4 * i < g.M && n < g.N ? *reinterpret_cast<const float4*>((const float*)g.Zin + o0 + 4 * i * g.ldc) : make_float4(0.f, 0.f, 0.f, 0.f);
        };
        float4 zn[2];                                // Z of the next two rows
        if constexpr (EPI == EPI_GELU_GRAD) { zn[0] = z_at(0); zn[1] = z_at(1); }
#pragma unroll 2
        for (int i = 0; i < 8; ++i) {
          const int r = 4 * i + (lane >> 3);
          float4 z = make_float4(0.f, 0.f, 0.f, 0.f);
          if constexpr (EPI == EPI_GELU_GRAD) { z = zn[i & 1]; if (i < 6) zn[i & 1] = z_at(i + 2); }
          float4 v = *reinterpret_cast<const float4*>(stg + r * 128 + (((lane & 7) ^ (r & 7)) << 4));
          if (mr + 4 * i >= g.M || n >= g.N) continue;
          const int64_t o = o0 + 4 * i * g.ldc;
          v.x = fmaf(v.x, kScaleOut, bias.x); v.y = fmaf(v.y, kScaleOut, bias.y); v.z = fmaf(v.z, kScaleOut, bias.z); v.w = fmaf(v.w, kScaleOut, bias.w);
          // GeLU as the multiply-add kernel takes it, exact at both ends.  (Packed polynomials save 13 us of a 524 us step at 2048 x 512 x
          // 2048, 16 experts, but their gate is off by 5e-8 for every z beyond 5.3 and by 1.0e-7 before, where erff's is within 6e-8.)
          if constexpr (EPI == EPI_GELU) {
            *reinterpret_cast<float4*>((float*)g.C2 + o) = g.gelu == 0 ? gelu_fwd4<0>(v) : gelu_fwd4<1>(v);
          } else if constexpr (EPI == EPI_GELU_GRAD) {
            z = g.gelu == 0 ? gelu_bwd4<0>(z) : gelu_bwd4<1>(z);
            v.x *= z.x; v.y *= z.y; v.z *= z.z; v.w *= z.w;
          }
          if (g.C) *reinterpret_cast<float4*>((float*)g.C + o) = v;
        }
        __syncwarp();
      }
      if (redo) take_again<EPI, A_K, B_K, LIST>(g, b, m0 + q * 32 + lane, n0 + half * kCols, bad);
    }
  }

  // ------------------------------------------------------------------ orderly exit
  __syncwarp();
  if (*abort_flag) {                                 // let MMAs still in flight drain
    const unsigned long long t0 = globaltimer();
    while (globaltimer() - t0 < 200000ull) __nanosleep(1000);
  }
  tc_fence_before();
  __syncthreads();
  if (warp == kMmaWarp) {
    tc_fence_after();
    asm volatile("tcgen05.dealloc.cta_group::1.sync.aligned.b32 %0, %1;" ::"r"(tmem_base), "r"(512) : "memory");
  }
  chain_leave(g.early);
}

template <int EPI, int FN, bool A_K, bool B_K, bool LIST>
cudaError_t launch_f32_tc_one(const GemmArgs& g, int sms, cudaStream_t st) {
  auto kern = gemm_f32_tc_kernel<EPI, FN, A_K, B_K, LIST>;
  constexpr int smem = f32_smem_bytes(FN);
  cudaFuncAttributes at;                             // the split of the registers relies on what the compiler gave the kernel
  cudaError_t e = cudaFuncGetAttributes(&at, kern);
  if (e != cudaSuccess) return e;
  if (at.numRegs != kLaunchRegs) return cudaErrorNotSupported;
#ifdef EC_DEBUG
  if (g.other_regs) return cudaErrorNotSupported;
#endif
  if ((e = cudaFuncSetAttribute(kern, cudaFuncAttributeMaxDynamicSharedMemorySize, smem)) != cudaSuccess) return e;
  const int tm = (g.M + FM - 1) / FM, tn = (g.N + FN - 1) / FN, total = tm * tn * g.batches;
  return launch_chained(kern, dim3(total < sms ? total : sms), dim3(kF32Threads), smem, st, g, tm, tn, total);
}
// The layer's products: X W1 and dX_e W2 (rows of K times rows of N), H W2^T and dZ W1^T (rows of K both), the weight gradients
template <int FN>
cudaError_t launch_f32_tc_n(const GemmArgs& g, int sms, cudaStream_t st) {
  const bool ak = g.sak == 1, bk = g.sbk == 1;
  if (g.a_rows) {
    return ak ? launch_f32_tc_one<EPI_GELU, FN, true, false, true>(g, sms, st) : launch_f32_tc_one<EPI_STORE, FN, false, false, true>(g, sms, st);
  }
  if (ak && !bk) switch (g.epi) {
    case EPI_STORE: return launch_f32_tc_one<EPI_STORE, FN, true, false, false>(g, sms, st);
    case EPI_GELU: return launch_f32_tc_one<EPI_GELU, FN, true, false, false>(g, sms, st);
    case EPI_GELU_GRAD: return launch_f32_tc_one<EPI_GELU_GRAD, FN, true, false, false>(g, sms, st);
  }
  if (ak && bk && g.epi == EPI_STORE) return launch_f32_tc_one<EPI_STORE, FN, true, true, false>(g, sms, st);
  if (!ak && !bk && g.epi == EPI_STORE) return launch_f32_tc_one<EPI_STORE, FN, false, false, false>(g, sms, st);
  return cudaErrorInvalidValue;
}

}  // namespace

// Estimated cycles with `cols` columns per tile: per k-block what the data path takes (measured with all SMs busy), per tile the
// epilogue that is left in the open
static double f32_tc_cycles(const GemmArgs& g, int cols, int sms) {
  const int64_t tiles = (((int64_t)g.M + FM - 1) / FM) * ((g.N + cols - 1) / cols) * g.batches;
  return (double)((tiles + sms - 1) / sms) * ((g.K + FK - 1) / FK * (cols == 64 ? 3000. : 3400.) + 2500.);
}
double plan_gemm_f32_tc(const GemmArgs& g, int sms, int* cols) {
  const bool ak = g.sak == 1, bk = g.sbk == 1;
  const bool form = ak && !bk ? g.epi == EPI_STORE || g.epi == EPI_GELU || g.epi == EPI_GELU_GRAD : ak == bk && g.epi == EPI_STORE;
  const bool list = !g.a_rows || (ak && !bk && g.epi == EPI_GELU) || (!ak && !bk);
  const int64_t tiles = (((int64_t)g.M + FM - 1) / FM) * ((g.N + 63) / 64) * g.batches;
  if (!form || !list || g.k_limit > 0 || g.status == nullptr || tiles > 0x7FFFFFFF) return -1.;
  const double narrow = f32_tc_cycles(g, 64, sms), wide = f32_tc_cycles(g, 128, sms);
  *cols = narrow < wide ? 64 : 128;
  return narrow < wide ? narrow : wide;
}
cudaError_t launch_gemm_f32_tc(const GemmArgs& g, int cols, int sms, cudaStream_t st) {
  return cols == 64 ? launch_f32_tc_n<64>(g, sms, st) : launch_f32_tc_n<128>(g, sms, st);
}

}  // namespace ecmoe
