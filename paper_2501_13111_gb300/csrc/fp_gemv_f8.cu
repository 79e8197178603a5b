// Decode linear for int4 group-128 weights at up to 32 tokens on the tcgen05
// tensor cores with 8-bit operands.
//
// y[m][n] = sum_g s[n][g] sum_{k in g} (q[n][k] - z[n][g]) x[m][k].
//
// An int4 code placed in a byte is the e4m3 number q 2^-9, exactly: e4m3's
// subnormals (bytes 0-7) and its first binade (8-15) share one spacing.  So a
// packed word becomes two operand words by one shift and two masks (0.4
// instructions a code; the bf16 expansion takes two), and the weights stay
// exact.  x is split beforehand, per token and group (beyond 16 tokens per token), into
// two e4m3 pieces (split_x_kernel):
//   x 2^e = hi + lo / 32,  e the power of two with the largest |x| 2^e in [128, 256).
// hi keeps four significant bits and lo the next four, so a bf16 x is carried
// exactly down to 2^-13 of the largest |x| of its group (token) and, below, with an
// error of at most 2^-22 of that largest.  hi and lo are columns of their own, so N = 2
// x tokens; the group's products are summed in fp32, and lo / 32, the zero point times
// the group's sum of x, 2^-e and the scale are applied in fp32 to its accumulator.
// To 16 tokens: with one exponent a token, one large element cost the small elements of
// every group their bits.  Relative error of rows of N(0, 0.05) and one element of 30000
// whose own weights are zero (2-norm; an exponent a group / a token / the mma.sync GEMV,
// whose fp32 sums hold 1024 + q times x; the result's rounding is 0.0017 of each):
//   4608 x 4096 0.0088 / 0.046 / 1.6   5120 x 13824 0.0049 / 0.047 / 0.55   65536 x 256 0.032 / 0.046 / 2.9
// and with the whole group's weights zero 0.0017 / 0.03-0.05 / 0.0017.
// Beyond 16 tokens the sums' warps set the pace and the group's exponent would cost 12 us
// of 100; the path that this kernel replaces there takes any bf16 x as it is (one element of
// 2^18 beside unit normals, its weights zero: 0.0027, here 0.054; infinities).  So the
// split adds up what each token loses, and a third kernel, that path, runs again over the
// result if that is more than its own rounding, else returns (1.2-2 us).
//
// One CTA per SM, 20 warps; an item is two groups of one row tile:
//   warps 0-7   codes to operands, one row per thread, shared memory to TMEM:
//               warps 0-3 the even items, 4-7 the odd ones;
//   warps 8-15  the group sums to fp32 accumulators, one row per thread: warps
//               8-11 the even items, 12-15 the odd ones; at the end of a row
//               tile each takes half of the tokens (exchanged through shared
//               memory) to the output;
//   warp 16     TMA of the weights, [128 rows][128 bytes] boxes (SwiGLU: 64
//               gate and the matching 64 up rows), into a ring;
//   warp 17     copies of the items' x pieces (already in the swizzled layout)
//               and sums into rings of their own;
//   warps 18-19 issue the MMAs of the even and of the odd items (M 128 weight
//               rows from TMEM, N 2 MT, K 32), one accumulator per group; warp
//               18 owns the 512 TMEM columns.
// A warp's pass over an item is a chain of waits and round trips (1400 cycles
// for the operands, 1100-2600 for the sums) while an item may take 780, hence
// two of each kind: with every warp on every item the 57344 x 8192 SwiGLU took
// 155 us at 8 tokens, so 61.  More warps did not help (four teams for the operands
// 64 us), nor did one polling lane per warp (80).
// The (row tile, item) pairs are cut into equal contiguous ranges, one per
// CTA.  A row tile shared by several CTAs is finished by the last of them from
// fp32 partials (a ticket per 32 rows and half of the tokens; sums in CTA
// order, nothing spins).  SwiGLU tiles always go through the partials, which
// bring a gate row and its up row together.
//
// What bounds it: an item's 17 KB of codes and scales take 780 cycles of an SM
// at the copy rate and its MMAs 360; the hand-offs between the roles keep it at
// about 1070 (57344 x 8192, 252 MB, 8 tokens: 61.5 us, 4.1 TB/s; without any copy
// after the rings' first fill 61).
// Every mbarrier wait is bounded; past the limit the thread records error 2,
// the CTA stops and releases TMEM after its copies and MMAs have completed.
#include <algorithm>

#include <cuda_fp16.h>
#include <cuda_fp8.h>

#include "common.cuh"
#include "kernels.cuh"
#include "tc.cuh"

namespace fpk {

constexpr int kF8Rows = 128, kF8RowBytes = 128;           // an item's weight box
constexpr int kF8WStage = kF8Rows * kF8RowBytes;           // 16 KB
constexpr int kF8WarpEpi = 8, kF8WarpW = 16, kF8WarpX = 17, kF8WarpMma = 18;
constexpr int kF8Threads = 20 * 32;
constexpr int kF8SlotCols = 64;                            // an A operand slot in TMEM (two groups)
constexpr int kF8XsRing = 10;                              // stages of group sums

template <int MT>
struct F8Geom {
  static constexpr int kN = 2 * MT;                        // hi columns, then lo columns
  static constexpr int kGroupBytes = kN * 128;             // x pieces of one group
  static constexpr int kXStage = 2 * kGroupBytes;
  static constexpr int kAccs = MT == 32 ? 2 : 4;           // items whose two accumulators are in TMEM
  static constexpr int kSlots = MT == 8 ? 6 : 4;           // items whose A operands are
  static constexpr int kACol = kAccs * 2 * kN;             // the first column of the A operands
  static constexpr int kWStages = MT == 32 ? 8 : 10;
  static constexpr int kXStages = 4;
  static constexpr int kXsStage = 2 * 2 * MT * 4;          // two groups' sums and powers of two
  static constexpr int kSwap = kF8Rows * MT * 4;           // the tokens' halves changing hands
  static constexpr int kSmem = kWStages * kF8WStage + kXStages * kXStage + kF8XsRing * kXsStage + kSwap + 1024;
  static_assert(kACol + kSlots * kF8SlotCols <= 512, "TMEM columns");
  static_assert(kSlots % 2 == 0, "each issuer and converting team keeps to slots of its own");
  static_assert(kXStages <= kSlots, "an x stage is freed by the commit of its item");
  // sums are read while the MMAs are at most kAccs items ahead and the copies kXStages beyond
  static_assert(kF8XsRing >= kXStages + kAccs + 2, "ring of group sums");
  static_assert(kSmem <= 227 * 1024, "shared memory");
};

FP_DEV long long f8_cta_of(long long i, long long C, long long total) { return ((i + 1) * C - 1) / total; }

// ------------------------------------------------------------------ x pieces
// pieces [groups][2 MT][128 bytes], row m token m's hi and row MT + m its lo (tokens past
// M: zeros), 16-byte chunk c of a row at c ^ (row % 8) (the 128-byte swizzle), and within
// each eight elements the order in which masking a packed int4 word yields them; sums
// [groups][2][MT] = 2^-9 sum of the group's pieces, then 2^-e, NaN where the exponent's
// elements hold an infinity or a NaN.  perm (GPTQ4): element j is x[perm[j]].
// TOKEN false: an exponent a (token, group), CTAs x tokens, eight elements a thread.  True
// (17 tokens and more): an exponent a token, one CTA each, which reads the row twice and
// leaves in range[m] the token's squares lost and kept (f8_wide), and in xp, if given, x in
// the order of perm for the kernel that takes over then.
// Bound by latency (2 K bytes read and written per token).
constexpr int kSplitThreads = 256, kSplitRowThreads = 1024;

// |x| as bf16 bits orders like the values, infinities and NaN on top.
FP_DEV uint32_t f8_amax(uint32_t a, const uint4& v) {
  const uint32_t w[4] = {v.x, v.y, v.z, v.w};
#pragma unroll
  for (int i = 0; i < 4; ++i) a = max(a, max(w[i] & 0x7FFFu, (w[i] >> 16) & 0x7FFFu));
  return a;
}

template <bool TOKEN>
__global__ void __launch_bounds__(TOKEN ? kSplitRowThreads : kSplitThreads)
    split_x_kernel(const uint16_t* __restrict__ x, int M, int MT, int K, const int32_t* __restrict__ perm,
                   uint8_t* __restrict__ pieces, float* __restrict__ sums, float2* __restrict__ range,
                   uint16_t* __restrict__ xp, int32_t* err) {
  pdl_trigger();
  pdl_wait();
  const int m = blockIdx.y, lane = threadIdx.x & 31, chunks = K / 8;  // whole groups of 16 chunks
  const uint16_t* xr = x + (long long)m * K;
  bool bad = false;
  auto load = [&](int c) {  // eight elements; past the row or the tokens: zeros
    uint4 v = make_uint4(0, 0, 0, 0);
    if (m < M && c < chunks) {
      if (perm == nullptr) {
        v = ld_nc16(xr + c * 8);
      } else {
        uint32_t e[8];
#pragma unroll
        for (int i = 0; i < 8; ++i) {
          const int k = perm[c * 8 + i];
          const bool ok = (unsigned)k < (unsigned)K;
          bad |= !ok;
          e[i] = ok ? (uint32_t)xr[k] : 0u;
        }
        v = make_uint4(e[0] | (e[1] << 16), e[2] | (e[3] << 16), e[4] | (e[5] << 16), e[6] | (e[7] << 16));
      }
    }
    return v;
  };
  uint32_t row = 0;  // TOKEN: the row's largest
  __shared__ uint32_t red[TOKEN ? kSplitRowThreads / 32 : 1];
  __shared__ float2 part[TOKEN ? kSplitRowThreads / 32 : 1];
  if constexpr (TOKEN) {
    for (int c = threadIdx.x; c < chunks; c += kSplitRowThreads) {
      const uint4 v = load(c);
      if (xp != nullptr && m < M) *reinterpret_cast<uint4*>(xp + (long long)m * K + c * 8) = v;
      row = f8_amax(row, v);
    }
    row = __reduce_max_sync(0xffffffffu, row);
    if (lane == 0) red[threadIdx.x >> 5] = row;
    __syncthreads();
    row = __reduce_max_sync(0xffffffffu, red[lane]);
  }
  float lost = 0.f, all = 0.f, few = 0.f;  // squares: what the pieces lose, x, x below 2^-8 of the largest
  int small = 0;
  // (groups: one round, of whose threads all take part in the reductions)
  int c0 = blockIdx.x * blockDim.x + (threadIdx.x & ~31);
  do {
    const int c = c0 + lane;
    const uint4 v = load(c);
    const uint32_t w[4] = {v.x, v.y, v.z, v.w};
    uint32_t am = TOKEN ? row : f8_amax(0, v);
    if constexpr (!TOKEN) {
      bool over = false;  // beyond the fp16 range but not NaN
#pragma unroll
      for (int i = 0; i < 4; ++i) {
        const uint32_t a = w[i] & 0x7FFFu, b = (w[i] >> 16) & 0x7FFFu;
        over |= (a >= 0x4780u && a <= 0x7F80u) || (b >= 0x4780u && b <= 0x7F80u);
      }
      // tokens that a kernel staging x in fp16 refuses are refused here too
      if (over && err) atomicExch(err, 3);
#pragma unroll
      for (int o = 8; o > 0; o >>= 1) am = max(am, __shfl_xor_sync(0xffffffffu, am, o));  // the group's 16 lanes
    }
    // e = 134 - biased exponent of the largest, kept where 2^e and 2^-e are normal
    const int ex = (int)(am >> 7);
    const int e = am == 0 || ex == 255 ? 0 : min(126, 134 - ex);
    const float mul = __uint_as_float((uint32_t)(127 + e) << 23);
    float hi_sum = 0.f, lo_sum = 0.f;
    uint32_t hb[4], lb[4];  // e4m3 pairs (2i, 2i + 1)
#pragma unroll
    for (int i = 0; i < 4; ++i) {
      float2 f = bf2x2f(w[i]);
      f.x *= mul;
      f.y *= mul;
      const __nv_fp8x2_storage_t h = __nv_cvt_float2_to_fp8x2(f, __NV_SATFINITE, __NV_E4M3);
      const float2 hf = __half22float2(__half2(__nv_cvt_fp8x2_to_halfraw2(h, __NV_E4M3)));
      const float2 r = make_float2((f.x - hf.x) * 32.f, (f.y - hf.y) * 32.f);
      const __nv_fp8x2_storage_t l = __nv_cvt_float2_to_fp8x2(r, __NV_SATFINITE, __NV_E4M3);
      const float2 lf = __half22float2(__half2(__nv_cvt_fp8x2_to_halfraw2(l, __NV_E4M3)));
      hi_sum += hf.x + hf.y;
      lo_sum += lf.x + lf.y;
      if constexpr (TOKEN) {
        const float dx = r.x - lf.x, dy = r.y - lf.y;  // 32 times what the pieces lose
        lost += dx * dx + dy * dy;
        all += f.x * f.x + f.y * f.y;
        if (fabsf(f.x) < 1.f) few += f.x * f.x, small += c < chunks;
        if (fabsf(f.y) < 1.f) few += f.y * f.y, small += c < chunks;
      }
      hb[i] = h;
      lb[i] = l;
    }
    // a packed int4 word masked with 0x0F0F0F0F holds elements 0, 4, 1, 5, and
    // shifted by four bits 2, 6, 3, 7
    const uint2 ho = make_uint2(__byte_perm(hb[0], hb[2], 0x5140), __byte_perm(hb[1], hb[3], 0x5140));
    const uint2 lo = make_uint2(__byte_perm(lb[0], lb[2], 0x5140), __byte_perm(lb[1], lb[3], 0x5140));
    float sum = hi_sum + lo_sum * (1.f / 32.f);
#pragma unroll
    for (int o = 8; o > 0; o >>= 1) sum += __shfl_xor_sync(0xffffffffu, sum, o);
    if (c < chunks) {
      const int g = c >> 4, ch = (c & 15) >> 1, half = c & 1;
      uint8_t* base = pieces + (long long)g * (2 * MT * 128);
      *reinterpret_cast<uint2*>(base + m * 128 + ((ch ^ (m & 7)) << 4) + half * 8) = ho;
      *reinterpret_cast<uint2*>(base + (MT + m) * 128 + ((ch ^ ((MT + m) & 7)) << 4) + half * 8) = lo;
      if ((c & 15) == 0) {
        float* o = sums + (long long)g * (2 * MT) + m;
        o[0] = sum * (1.f / 512.f);
        o[MT] = __uint_as_float(ex == 255 ? 0x7FC00000u : (uint32_t)(127 - e) << 23);
      }
    }
  } while (TOKEN && (c0 += kSplitRowThreads) < chunks);
  if (bad && err) atomicExch(err, 1);
  if constexpr (TOKEN) {
    // the token's squares; where most of its elements are below 2^-8 of the largest, only
    // those count as kept
    const int warp = threadIdx.x >> 5;
    const float most = warp_sum(few);
    lost = warp_sum(lost);
    all = warp_sum(all);
    small = __reduce_add_sync(0xffffffffu, small);
    __shared__ float smalls[kSplitRowThreads / 32];
    __shared__ int counts[kSplitRowThreads / 32];
    if (lane == 0) part[warp] = make_float2(lost, all), smalls[warp] = most, counts[warp] = small;
    __syncthreads();
    if (warp == 0) {
      lost = warp_sum(part[lane].x);
      all = warp_sum(part[lane].y);
      few = warp_sum(smalls[lane]);
      small = __reduce_add_sync(0xffffffffu, counts[lane]);
      if (lane == 0)
        range[m] = (row >> 7) == 255 ? make_float2(1.f, 0.f)  // an infinity or a NaN: lost
                                     : make_float2(lost / 1024.f, 2 * small >= K ? few : all);
    }
  }
}

// ------------------------------------------------------------------ helpers
// d = a b + c on two fp32 lanes at once.
FP_DEV float2 ffma2(float2 a, float2 b, float2 c) {
  float2 d;
  asm("{\n .reg .b64 a, b, c, d;\n mov.b64 a, {%2, %3};\n mov.b64 b, {%4, %5};\n mov.b64 c, {%6, %7};\n"
      " fma.rn.f32x2 d, a, b, c;\n mov.b64 {%0, %1}, d;\n}\n"
      : "=f"(d.x), "=f"(d.y)
      : "f"(a.x), "f"(a.y), "f"(b.x), "f"(b.y), "f"(c.x), "f"(c.y));
  return d;
}
// d = a b on two fp32 lanes at once.
FP_DEV float2 fmul2(float2 a, float2 b) {
  float2 d;
  asm("{\n .reg .b64 a, b, d;\n mov.b64 a, {%2, %3};\n mov.b64 b, {%4, %5};\n"
      " mul.rn.f32x2 d, a, b;\n mov.b64 {%0, %1}, d;\n}\n"
      : "=f"(d.x), "=f"(d.y)
      : "f"(a.x), "f"(a.y), "f"(b.x), "f"(b.y));
  return d;
}

// Output column `row` of tokens m0 .. m0 + T - 1 (those below M) from their
// sums v (SwiGLU: gate sums v, up sums w), times the tokens' powers of two (UN).  The
// residuals are read before any store (R may be Y itself).
template <int EPI, int T, bool UN>
FP_DEV void f8_store(const float* v, const float* w, int M, int m0, int row, int Nout, const float* __restrict__ unscale,
                     const uint16_t* R, void* Y) {
  float un[T], rv[T];
#pragma unroll
  for (int t = 0; t < T; ++t) {
    const int m = min(m0 + t, M - 1);
    un[t] = UN ? __ldg(unscale + m) : 1.f;
    rv[t] = EPI == FP_EPI_RESID ? bf2f(R[(long long)m * Nout + row]) : 0.f;
  }
#pragma unroll
  for (int t = 0; t < T; ++t) {
    if (m0 + t >= M) break;
    const float a = UN ? v[t] * un[t] : v[t];
    uint16_t* y = (uint16_t*)Y + (long long)(m0 + t) * Nout + row;
    if constexpr (EPI == FP_EPI_STORE) *y = f2bf(a);
    else if constexpr (EPI == FP_EPI_RESID) *y = f2bf(rv[t] + a);
    else *y = f2bf(silu(a) * (UN ? w[t] * un[t] : w[t]));
  }
}

// The same from the partials of cnt CTAs, `slot` floats apart, summed in CTA
// order (deterministic) with the loads of several CTAs in flight together
// (one after the other they took 4 us of a 5120 x 5120 matrix).  Not inlined:
// its registers would crowd the loop over the items.
template <int EPI, int T, bool UN>
__device__ __noinline__ void f8_sum_store(const float* p0, size_t slot, int cnt, int M, int m0, int row, int Nout,
                                          const float* __restrict__ unscale, const uint16_t* R, void* Y) {
  constexpr bool GLU = EPI == FP_EPI_SWIGLU;
  constexpr int B = T < 8 ? T : 8, U = GLU ? 2 : 4;
  if (row >= Nout) return;
#pragma unroll
  for (int t0 = 0; t0 < T; t0 += B) {
    float v[B], w[B];
#pragma unroll
    for (int k = 0; k < B; ++k) v[k] = w[k] = 0.f;
    for (int cc = 0; cc < cnt; cc += U) {
      const float* pc = p0 + (size_t)cc * slot + (size_t)(m0 + t0) * kF8Rows;
      float a[U][B], e[U][B];
#pragma unroll
      for (int u = 0; u < U; ++u)
#pragma unroll
        for (int k = 0; k < B; ++k) {
          const bool in = cc + u < cnt && m0 + t0 + k < M;
          a[u][k] = in ? __ldcg(pc + u * slot + k * kF8Rows) : 0.f;
          e[u][k] = GLU && in ? __ldcg(pc + u * slot + k * kF8Rows + kF8Rows / 2) : 0.f;
        }
#pragma unroll
      for (int u = 0; u < U; ++u)
#pragma unroll
        for (int k = 0; k < B; ++k) v[k] += a[u][k], w[k] += e[u][k];
    }
    f8_store<EPI, B, UN>(v, w, M, m0 + t0, row, Nout, unscale, R, Y);
  }
}

// ------------------------------------------------------------------ kernel
// S: groups per row; SI = ceil(S / 2) items per row tile.
template <int MT, int EPI>
__global__ void __launch_bounds__(kF8Threads, 1)
    gemv_f8_kernel(const __grid_constant__ CUtensorMap map_w, const uint8_t* __restrict__ pieces,
                   const float* __restrict__ sums, int M, int N,
                   const uint16_t* __restrict__ scales, const uint16_t* __restrict__ zeros, const uint16_t* R, void* Y,
                   long long total, int S, float* __restrict__ ws, unsigned* __restrict__ counters, int32_t* err) {
  using G = F8Geom<MT>;
  constexpr bool GLU = EPI == FP_EPI_SWIGLU;
  constexpr bool GE = MT <= 16;  // an exponent a group, not a token
  constexpr int WS = G::kWStages, XS = G::kXStages, NA = G::kSlots, ND = G::kAccs, TH = MT / 2;
  constexpr int TR = GLU ? kF8Rows / 2 : kF8Rows;  // output rows per tile
  extern __shared__ __align__(1024) uint8_t smem_raw[];
  __shared__ uint64_t wfull[WS], wempty[WS], xfull[XS], afull[NA], idone[NA], dempty[ND], sfull[kF8XsRing],
      given[2][4], taken[2][4], mma_done[2];
  __shared__ uint32_t tmem_base;
  __shared__ int abort_word;
  volatile int* abort_flag = &abort_word;
  uint8_t* smem = (uint8_t*)(((uintptr_t)smem_raw + 1023) & ~(uintptr_t)1023);
  uint8_t* w_ring = smem;
  uint8_t* x_ring = smem + WS * kF8WStage;
  float* xs_ring = reinterpret_cast<float*>(x_ring + XS * G::kXStage);
  float* swap = xs_ring + kF8XsRing * 4 * MT;
  const int warp = threadIdx.x >> 5, lane = threadIdx.x & 31;
  const int Nout = GLU ? N / 2 : N;
  const long long C = gridDim.x, c = blockIdx.x;
  const long long begin = c * total / C, end = (c + 1) * total / C;
  const int L = (int)(end - begin), SI = (S + 1) / 2;
  const int b_first = (int)(begin / SI), i_first = (int)(begin % SI);  // (row tile, item) of the range's start
  auto fail = [&]() {
    *abort_flag = 1;
    if (err) atomicExch(err, 2);
  };

  pdl_trigger();
  if (threadIdx.x == 0) {
    for (int i = 0; i < WS; ++i) mbar_init(&wfull[i], 1), mbar_init(&wempty[i], 4);
    for (int i = 0; i < XS; ++i) mbar_init(&xfull[i], 1);
    for (int i = 0; i < NA; ++i) mbar_init(&afull[i], 4), mbar_init(&idone[i], 1);
    for (int i = 0; i < ND; ++i) mbar_init(&dempty[i], 4);
    for (int i = 0; i < kF8XsRing; ++i) mbar_init(&sfull[i], 1);
    for (int i = 0; i < 8; ++i) mbar_init(&given[i >> 2][i & 3], 1), mbar_init(&taken[i >> 2][i & 3], 1);
    mbar_init(&mma_done[0], 1);
    mbar_init(&mma_done[1], 1);
    *abort_flag = 0;
    asm volatile("fence.mbarrier_init.release.cluster;" ::: "memory");
  }
  if (warp == kF8WarpMma) {
    asm volatile("tcgen05.alloc.cta_group::1.sync.aligned.shared::cta.b32 [%0], 512;" ::"r"(smem_u32(&tmem_base))
                 : "memory");
    asm volatile("tcgen05.relinquish_alloc_permit.cta_group::1.sync.aligned;" ::: "memory");
  }
  tc_fence_before();
  __syncthreads();
  tc_fence_after();
  const uint32_t tmem = tmem_base;

  if (warp == kF8WarpW) {
    // ---------------- the weights are constant: their ring fills before the
    // kernel that splits x has finished
    if (lane == 0) {
      int b = b_first, i = i_first, issued = 0;
      for (int q = 0; q < L; ++q) {
        const int s = q % WS;
        if (q >= WS && (!mbar_wait(&wempty[s], ((q / WS) & 1) ^ 1) || *abort_flag)) {
          fail();
          break;
        }
        uint8_t* d = w_ring + s * kF8WStage;
        mbar_expect_tx(&wfull[s], kF8WStage);
        tma_load_2d(d, &map_w, i * kF8RowBytes, b * TR, &wfull[s]);
        if (GLU) tma_load_2d(d + kF8WStage / 2, &map_w, i * kF8RowBytes, Nout + b * TR, &wfull[s]);
        issued = q + 1;
        if (++i == SI) i = 0, ++b;
      }
      // copies still in flight land before the CTA leaves (their stages are its shared memory)
      for (int j = max(0, issued - WS); j < issued; ++j) mbar_wait(&wfull[j % WS], (j / WS) & 1);
    }
  } else if (warp == kF8WarpX) {
    // ---------------- pieces, group sums and powers of two of x
    if (lane == 0) {
      pdl_wait();
      asm volatile("fence.proxy.async;" ::: "memory");  // they were written by generic stores
      int i = i_first, issued = 0;
      for (int q = 0; q < L; ++q) {
        // stage q % XS: item q - XS has been multiplied
        if (q >= XS && (!mbar_wait(&idone[(q - XS) % NA], ((q - XS) / NA) & 1) || *abort_flag)) {
          fail();
          break;
        }
        const int g0 = 2 * i, nv = min(2, S - g0), s = q % XS, r = q % kF8XsRing;
        mbar_expect_tx(&xfull[s], nv * G::kGroupBytes);
        bulk_load(x_ring + s * G::kXStage, pieces + (long long)g0 * G::kGroupBytes, nv * G::kGroupBytes, &xfull[s]);
        mbar_expect_tx(&sfull[r], nv * 2 * MT * 4);
        bulk_load(xs_ring + r * (4 * MT), sums + (long long)g0 * (2 * MT), nv * 2 * MT * 4, &sfull[r]);
        issued = q + 1;
        if (++i == SI) i = 0;
      }
      for (int j = max(0, issued - XS); j < issued; ++j) mbar_wait(&xfull[j % XS], (j / XS) & 1);
      for (int j = max(0, issued - kF8XsRing); j < issued; ++j) mbar_wait(&sfull[j % kF8XsRing], (j / kF8XsRing) & 1);
    }
  } else if (warp >= kF8WarpMma) {
    // ---------------- MMA issuers of the even and the odd items
    constexpr uint32_t idesc = tc_idesc_e4m3(kF8Rows, G::kN);
    const uint64_t xd0 = sdesc(smem_u32(x_ring));
    const int par = warp - kF8WarpMma;
    bool ok = true;
    int i = i_first + par;
    for (int q = par; q < L; q += 2, i += 2) {
      const int a = q % NA;
      while (i >= SI) i -= SI;
      const bool two = 2 * i + 1 < S;
      // operands are there, and the sums of item q - ND, which used this
      // accumulator, have been read
      ok = mbar_wait(&xfull[q % XS], (q / XS) & 1) && mbar_wait(&afull[a], (q / NA) & 1) &&
           (q < ND || mbar_wait(&dempty[q % ND], ((q / ND) & 1) ^ 1)) && !*abort_flag;
      ok = __all_sync(0xffffffffu, ok);
      if (!ok) break;
      tc_fence_after();
      const uint64_t xd = xd0 + (uint64_t)(((q % XS) * G::kXStage) >> 4);
      const uint32_t ta = tmem + G::kACol + a * kF8SlotCols, td = tmem + (q % ND) * 2 * G::kN;
      if (elect_one()) {
#pragma unroll
        for (int kk = 0; kk < 4; ++kk) {  // 32 k: eight A columns, 32 bytes of an x row
          tc_mma_ts_f8(td, ta + kk * 8, xd + kk * 2, idesc, kk > 0 ? 1u : 0u);
          if (two)
            tc_mma_ts_f8(td + G::kN, ta + kF8SlotCols / 2 + kk * 8, xd + (G::kGroupBytes >> 4) + kk * 2, idesc,
                         kk > 0 ? 1u : 0u);
        }
        tc_commit(&idone[a]);  // the sums are complete, A slot a and x stage q % XS have been read
      }
      __syncwarp();
    }
    if (!ok && lane == 0) fail();
    if (elect_one()) tc_commit(&mma_done[par]);  // every MMA issued has completed before TMEM is released
    __syncwarp();
    mbar_wait(&mma_done[par], 0);
  } else if (warp < kF8WarpEpi) {
    // ---------------- codes to operands
    const int par = warp >> 2, qd = warp & 3, row = qd * 32 + lane;
    const uint32_t ta = tmem + ((uint32_t)(qd * 32) << 16) + G::kACol;
    const uint8_t* src = w_ring + row * kF8RowBytes;
    const int sw = row & 7;
    for (int q = par; q < L; q += 2) {
      bool ok = mbar_wait(&wfull[q % WS], (q / WS) & 1);
      const int a = q % NA;
      uint4 w[8];
#pragma unroll
      for (int i = 0; i < 8; ++i)
        w[i] = *reinterpret_cast<const uint4*>(src + (q % WS) * kF8WStage + ((i ^ sw) << 4));
      if (q >= NA) ok = mbar_wait(&idone[a], ((q / NA) & 1) ^ 1) && ok;
      if (!__all_sync(0xffffffffu, ok)) {
        if (lane == 0) fail();
        break;
      }
      tc_fence_after();
      if (lane == 0) mbar_arrive(&wempty[q % WS]);  // every lane has its row in registers
#pragma unroll
      for (int j = 0; j < 2; ++j) {
        uint32_t o[32];
#pragma unroll
        for (int i = 0; i < 4; ++i) {
          const uint4 v = w[4 * j + i];
          const uint32_t ww[4] = {v.x, v.y, v.z, v.w};
#pragma unroll
          for (int t = 0; t < 4; ++t) {
            o[i * 8 + t * 2] = ww[t] & 0x0F0F0F0Fu;
            o[i * 8 + t * 2 + 1] = (ww[t] >> 4) & 0x0F0F0F0Fu;
          }
        }
        tc_st32(ta + a * kF8SlotCols + j * (kF8SlotCols / 2), o);
      }
      tc_wait_st();
      tc_fence_before();
      __syncwarp();
      if (lane == 0) mbar_arrive(&afull[a]);
    }
  } else {
    // ---------------- group sums to accumulators, row tiles to the output
    const int qd = warp & 3, lr = qd * 32 + lane, par = (warp - kF8WarpEpi) >> 2;
    const uint32_t lane_base = tmem + ((uint32_t)(qd * 32) << 16);
    constexpr int CH = MT <= 16 ? MT : 16;  // tokens per TMEM load
    // scales and zeros of this thread's weight row, the two groups of its next item
    auto wrow = [&](int bb) -> long long {  // the row of the weight matrix (clamped: rows past the end are not stored)
      if (GLU) return min(bb * TR + (lr & (TR - 1)), Nout - 1) + (lr >= TR ? (long long)Nout : 0LL);
      return min(bb * TR + lr, Nout - 1);
    };
    auto pair_of = [&](const uint16_t* p, long long idx, int i) -> uint32_t {
      if ((S & 1) == 0) return __ldg(reinterpret_cast<const unsigned int*>(p + idx));
      const uint32_t lo = __ldg(reinterpret_cast<const unsigned short*>(p + idx));
      return 2 * i + 1 < S ? lo | ((uint32_t)__ldg(reinterpret_cast<const unsigned short*>(p + idx + 1)) << 16) : lo;
    };
    int nb = b_first, ni = i_first;  // (row tile, item) whose scales are loaded next
    uint32_t s_nxt = 0, z_nxt = 0;
    auto load_scales = [&]() {
      const long long idx = wrow(nb) * S + 2 * ni;
      s_nxt = pair_of(scales, idx, ni);
      z_nxt = pair_of(zeros, idx, ni);
    };
    auto skip = [&](int n) {
      for (ni += n; ni >= SI; ni -= SI) ++nb;
    };
    skip(par);
    if (par < L) load_scales();
    pdl_wait();
    const int m0 = par * TH;  // the tokens this warp takes to the output
    float2 acc[MT / 2];
#pragma unroll
    for (int t = 0; t < MT / 2; ++t) acc[t] = make_float2(0.f, 0.f);
    int b = b_first, i = i_first, seg = 0;
    for (int q = 0; q < L; ++q) {
      if ((q & 1) == par) {
        const uint32_t sp = s_nxt, zp = z_nxt;
        if (q + 2 < L) {
          skip(2);
          load_scales();
        }
        const int r = q % kF8XsRing, nv = min(2, S - 2 * i);
        const bool ok = mbar_wait(&sfull[r], (q / kF8XsRing) & 1) && mbar_wait(&idone[q % NA], (q / NA) & 1);
        if (!__all_sync(0xffffffffu, ok)) {
          if (lane == 0) fail();
          break;
        }
        tc_fence_after();
#pragma unroll
        for (int j = 0; j < 2; ++j) {
          if (j < nv) {
            const float s = __uint_as_float(j ? sp & 0xFFFF0000u : sp << 16);
            const float z = __uint_as_float(j ? zp & 0xFFFF0000u : zp << 16);
            const float2 s2 = make_float2(s, s), nz2 = make_float2(-z, -z), r32 = make_float2(1.f / 32.f, 1.f / 32.f);
            const float* xs = xs_ring + r * (4 * MT) + j * (2 * MT);
            const uint32_t d = lane_base + (q % ND) * 2 * G::kN + j * G::kN;
#pragma unroll
            for (int c0 = 0; c0 < MT; c0 += CH) {
              float4 xv[CH / 4], uv[CH / 4];  // read while the sums come from TMEM
#pragma unroll
              for (int t = 0; t < CH / 4; ++t) {
                xv[t] = *reinterpret_cast<const float4*>(xs + c0 + 4 * t);
                if (GE) uv[t] = *reinterpret_cast<const float4*>(xs + MT + c0 + 4 * t);
              }
              uint32_t hi[CH], lo[CH];
              tc_ld_pair<CH>(d + c0, d + MT + c0, hi, lo);
#pragma unroll
              for (int k = 0; k < CH; k += 2) {
                const float4 x4 = xv[k / 4], u4 = GE ? uv[k / 4] : make_float4(1.f, 1.f, 1.f, 1.f);
                const float2 xx = k & 2 ? make_float2(x4.z, x4.w) : make_float2(x4.x, x4.y);
                const float2 uu = k & 2 ? make_float2(u4.z, u4.w) : make_float2(u4.x, u4.y);
                float2 v = ffma2(nz2, xx, make_float2(__uint_as_float(hi[k]), __uint_as_float(hi[k + 1])));
                v = ffma2(make_float2(__uint_as_float(lo[k]), __uint_as_float(lo[k + 1])), r32, v);
                acc[(c0 + k) / 2] = ffma2(s2, GE ? fmul2(uu, v) : v, acc[(c0 + k) / 2]);
              }
            }
          }
        }
        tc_fence_before();
        __syncwarp();
        if (lane == 0) mbar_arrive(&dempty[q % ND]);
      }
      const int tb = b;
      if (++i == SI) i = 0, ++b;
      if (i != 0 && q != L - 1) continue;

      // ---- this CTA's part of row tile tb is summed, in the even and the odd
      // warps: this warp keeps tokens [m0, m0 + TH) and hands the others over
      float av[TH];
      {
        float* mine = swap + (par * TH) * kF8Rows + lr;          // [token][row] for this warp's tokens
        float* theirs = swap + ((par ^ 1) * TH) * kF8Rows + lr;
        bool ok = seg == 0 || mbar_wait(&taken[par ^ 1][qd], (seg - 1) & 1);  // the partner has read the last ones
        if (__all_sync(0xffffffffu, ok)) {
#pragma unroll
          for (int t = 0; t < TH / 2; ++t) {
            const float2 v = par ? acc[t] : acc[TH / 2 + t];
            theirs[(2 * t) * kF8Rows] = v.x;
            theirs[(2 * t + 1) * kF8Rows] = v.y;
          }
          __syncwarp();
          if (lane == 0) mbar_arrive(&given[par][qd]);
          ok = mbar_wait(&given[par ^ 1][qd], seg & 1);
        }
        if (!__all_sync(0xffffffffu, ok) || __any_sync(0xffffffffu, *abort_flag != 0)) {
          if (lane == 0) fail();
          break;
        }
#pragma unroll
        for (int t = 0; t < TH / 2; ++t) {
          const float2 v = par ? acc[TH / 2 + t] : acc[t];
          // the operands were q 2^-9
          const float x = mine[(2 * t) * kF8Rows], y = mine[(2 * t + 1) * kF8Rows];
          av[2 * t] = (v.x + x) * 512.f;
          av[2 * t + 1] = (v.y + y) * 512.f;
        }
        __syncwarp();
        if (lane == 0) mbar_arrive(&taken[par][qd]);
        ++seg;
      }
#pragma unroll
      for (int t = 0; t < MT / 2; ++t) acc[t] = make_float2(0.f, 0.f);

      const int row = tb * TR + (GLU ? (lr & (TR - 1)) : lr);
      const long long c0 = f8_cta_of((long long)tb * SI, C, total);
      const long long c1 = f8_cta_of((long long)(tb + 1) * SI - 1, C, total);
      if (!GLU && c0 == c1) {
        constexpr int B = TH < 8 ? TH : 8;
        if (row < Nout) {
#pragma unroll
          for (int t = 0; t < TH; t += B) f8_store<EPI, B, !GE>(av + t, av + t, M, m0 + t, row, Nout, sums + MT, R, Y);
        }
        continue;
      }
      // partial slot tb + c: distinct for every (row tile, CTA) pair that meets
      const size_t slot = (size_t)M * kF8Rows;
      float* part = ws + (size_t)(tb + c) * slot + lr;
#pragma unroll
      for (int t = 0; t < TH; ++t)
        if (m0 + t < M) part[(size_t)(m0 + t) * kF8Rows] = av[t];
      __threadfence();
      __syncwarp();
      // one ticket per 32 output rows and half of the tokens; with SwiGLU the
      // warps of the gate and of the up rows draw from the same one
      unsigned* ticket = counters + (GLU ? (tb * 2 + par) * 2 + (qd & 1) : (tb * 2 + par) * 4 + qd);
      const unsigned last = (unsigned)((c1 - c0 + 1) * (GLU ? 2 : 1) - 1);
      unsigned t = 0;
      if (lane == 0) t = atomicAdd(ticket, 1u);
      t = __shfl_sync(0xffffffffu, t, 0);
      if (t != last) continue;
      __threadfence();
      f8_sum_store<EPI, TH, !GE>(ws + (size_t)(tb + c0) * slot + (GLU ? (lr & (TR - 1)) : lr), slot, (int)(c1 - c0) + 1, M, m0,
                            row, Nout, sums + MT, R, Y);
      if (lane == 0) *ticket = 0u;
    }
  }
  tc_fence_before();
  __syncthreads();
  if (warp == kF8WarpMma) {
    tc_fence_after();
    asm volatile("tcgen05.dealloc.cta_group::1.sync.aligned.b32 %0, 512;" ::"r"(tmem) : "memory");
  }
}

// ------------------------------------------------------------------ host side
static int f8_sms() {
  static int n = 0;
  if (!n) {
    int dev = 0;
    if (cudaGetDevice(&dev) != cudaSuccess || cudaDeviceGetAttribute(&n, cudaDevAttrMultiProcessorCount, dev) != cudaSuccess ||
        n <= 0)
      n = 152;
  }
  return n;
}

static int f8_mt(int M) { return M <= 8 ? 8 : M <= 16 ? 16 : 32; }

// fp32 partials, then the x pieces and their group sums and powers of two; beyond 16
// tokens, behind what the kernel that may take over writes, the range sums and x in the
// order of perm.
struct F8Plan {
  long long tiles, total;
  int ctas, S;
  size_t pieces, sums, range, xp, bytes;  // offsets
};

static F8Plan f8_plan(int epi, int M, int N, int K) {
  F8Plan p{};
  const bool glu = epi == FP_EPI_SWIGLU;
  const long long nout = glu ? N / 2 : N;
  const int tr = glu ? kF8Rows / 2 : kF8Rows, mt = f8_mt(M);
  p.S = K / 128;
  p.tiles = (nout + tr - 1) / tr;
  p.total = p.tiles * ((p.S + 1) / 2);
  p.ctas = (int)std::min<long long>(p.total, f8_sms());
  auto up = [](size_t b) { return (b + 127) / 128 * 128; };
  p.pieces = (size_t)kLinTicketSlots * 4 + up((size_t)(p.tiles + p.ctas) * M * kF8Rows * 4);
  p.sums = p.pieces + (size_t)p.S * 2 * mt * 128;
  p.range = p.sums + up((size_t)p.S * 2 * mt * 4);
  if (M > 16) p.range = up(std::max(p.range, q4tc_ws_bytes(epi, M, N, K)));
  p.xp = p.range + (M > 16 ? up((size_t)mt * sizeof(float2)) : 0);
  p.bytes = p.xp + (M > 16 ? up((size_t)M * K * 2) : 0);
  return p;
}

// Where it is the faster path.  Measured in a graph over copies of the weights that
// exceed L2, microseconds here / the mma.sync GEMV:
//   tokens            1             8             9             16
//   1024 x 512      6.6 /  3.7    6.7 /  4.4    7.9 /  4.7    7.9 /  4.9
//   4096 x 4096     9.8 /  7.7   10.0 /  8.8   11.7 / 12.7   12.2 / 14.1
//   2048 x 8192    10.3 / 11.6   10.6 / 12.3   12.4 / 20.8   13.1 / 22.1
//   8192 x 4096    13.4 / 12.1   13.7 / 13.5   15.4 / 19.5   15.7 / 21.2
//   10240 x 8192   19.0 / 25.4   19.3 / 26.8   23.3 / 31.4   23.6 / 33.0
//   5120 x 13824   17.7 / 27.9   18.2 / 29.7   22.0 / 32.1   22.3 / 34.1
//   57344 x 8192   59.7 /  109   61.5 /  113   73.8 /  133   74.4 /  135 (SwiGLU)
//   tokens           17            32          (SwiGLU; here / the bf16 expansion in TMEM)
//   57344 x 8192   98.2 / 104    100.1 / 108
// The line was set at 8 MB of codes before the mma.sync GEMV had clusters; matrices of
// 8 to 20 MB that are wider than long have since been 1-2 us faster there at up to 8
// tokens, with larger errors.  From 17 tokens only the largest gate and up matrices gain.
static bool f8_pays(int epi, int M, int N, int K) {
  const long long weights = (long long)N * K;
  return M <= 16 ? weights >= (1LL << 24)
                 : M <= 32 && epi == FP_EPI_SWIGLU && weights >= (1LL << 28) && q4tc_ok(FP_W_INT4_G128, epi, M, N, K);
}

bool f8_ok(int wquant, int epi, int M, int N, int K) {
  if (wquant != FP_W_INT4_G128 || epi == FP_EPI_F32 || M < 1 || N < 1 || K < 128 || K % 128 != 0) return false;
  if (!f8_pays(epi, M, N, K) || (epi == FP_EPI_SWIGLU && N % 2 != 0)) return false;
  const long long nout = epi == FP_EPI_SWIGLU ? N / 2 : N;
  const long long tiles = (nout + kF8Rows - 1) / kF8Rows;  // eight tickets per 128 output rows
  return tiles * 8 <= kLinTicketSlots && tensor_maps_available();
}

size_t f8_ws_bytes(int epi, int M, int N, int K) { return f8_plan(epi, M, N, K).bytes; }

template <int MT, int EPI>
static cudaError_t launch_f8_t(const CUtensorMap& mw, const F8Plan& p, char* ws, int M, int N, const uint16_t* scales,
                               const uint16_t* zeros, const uint16_t* R, void* Y, int32_t* err, cudaStream_t s) {
  auto kern = gemv_f8_kernel<MT, EPI>;
  // above half an SM whatever MT is: one CTA (and one owner of the TMEM) per SM
  constexpr int smem = F8Geom<MT>::kSmem;
  static_assert(smem > 116 * 1024, "one CTA per SM");
  static std::atomic<unsigned long long> attr{0};
  FP_CUDA_TRY(smem_limit_once(kern, smem, &attr));
  return launch_early(kern, dim3(p.ctas), dim3(kF8Threads), (size_t)smem, s, mw, (const uint8_t*)(ws + p.pieces),
                      (const float*)(ws + p.sums), M, N, scales, zeros, R, Y, p.total,
                      p.S, (float*)(ws + (size_t)kLinTicketSlots * 4), (unsigned*)ws, err);
}

template <int MT>
static cudaError_t launch_f8_m(int epi, const CUtensorMap& mw, const F8Plan& p, char* ws, int M, int N,
                               const uint16_t* scales, const uint16_t* zeros, const uint16_t* R, void* Y, int32_t* err,
                               cudaStream_t s) {
  switch (epi) {
    case FP_EPI_STORE: return launch_f8_t<MT, FP_EPI_STORE>(mw, p, ws, M, N, scales, zeros, R, Y, err, s);
    case FP_EPI_RESID: return launch_f8_t<MT, FP_EPI_RESID>(mw, p, ws, M, N, scales, zeros, R, Y, err, s);
    default: return launch_f8_t<MT, FP_EPI_SWIGLU>(mw, p, ws, M, N, scales, zeros, R, Y, err, s);
  }
}

cudaError_t launch_f8(int epi, const uint16_t* x, const int32_t* perm, int M, int N, int K, const void* codes,
                      const uint16_t* scales, const uint16_t* zeros, const uint16_t* residual, void* y, void* ws,
                      size_t ws_bytes, int32_t* err, cudaStream_t s) {
  if (!f8_ok(FP_W_INT4_G128, epi, M, N, K)) return cudaErrorInvalidValue;
  const F8Plan p = f8_plan(epi, M, N, K);
  if (!ws || ws_bytes < p.bytes) return cudaErrorInvalidValue;
  const int mt = f8_mt(M);
  CUtensorMap mw;
  // codes [N][K / 2] bytes, box [128 rows (SwiGLU 64)][128]; past the row's end zeros
  if (!make_tensor_map(&mw, codes, N, K / 2, 1, epi == FP_EPI_SWIGLU ? kF8Rows / 2 : kF8Rows, kF8RowBytes, 128))
    return cudaErrorInvalidValue;
  char* w = (char*)ws;
  uint8_t* pieces = (uint8_t*)(w + p.pieces);
  float* sums = (float*)(w + p.sums);
  float2* range = (float2*)(w + p.range);
  uint16_t* xp = M > 16 && perm ? (uint16_t*)(w + p.xp) : nullptr;
  if (M <= 16)
    FP_CUDA_TRY(launch(split_x_kernel<false>, dim3((K / 8 + kSplitThreads - 1) / kSplitThreads, mt), dim3(kSplitThreads), 0,
                       s, x, M, mt, K, perm, pieces, sums, range, xp, err));
  else
    FP_CUDA_TRY(launch(split_x_kernel<true>, dim3(1, mt), dim3(kSplitRowThreads), 0, s, x, M, mt, K, perm, pieces, sums,
                       range, xp, err));
  switch (mt) {
    case 8: return launch_f8_m<8>(epi, mw, p, w, M, N, scales, zeros, residual, y, err, s);
    case 16: return launch_f8_m<16>(epi, mw, p, w, M, N, scales, zeros, residual, y, err, s);
    default:  // SwiGLU: no residual that y may be
      FP_CUDA_TRY((launch_f8_t<32, FP_EPI_SWIGLU>(mw, p, w, M, N, scales, zeros, residual, y, err, s)));
      return launch_q4tc_if_wide(xp ? xp : x, M, N, K, codes, scales, zeros, y, ws, ws_bytes, err, s, range);
  }
}

}  // namespace fpk
