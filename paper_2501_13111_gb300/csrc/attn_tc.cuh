// Pieces shared by the tcgen05 prefill attention kernels (fp_attn_tc.cu,
// fp_attn_short.cu): operand descriptors, conversions, launch limits.
#pragma once

#include "attn_items.h"
#include "kernels.cuh"
#include "tc.cuh"

namespace fpk {

constexpr int kPaHD = 128;
constexpr int kPaHalf = kPaB * 128;          // bytes of one [128 rows][64 bf16] swizzled half
constexpr int kPaTile = 2 * kPaHalf;         // one [128][128] bf16 operand
constexpr int kPaStage = 32 * 64;            // a warp's 32 output rows, 32 columns at a time
constexpr float kPaLog2e = 1.4426950408889634f;

// Shared-memory descriptor of an MN-major operand with 128-byte swizzle:
// 64-element atoms along MN `lbo` bytes apart, 8-row groups along K 1024
// bytes apart.
FP_DEV uint64_t sdesc_mn(uint32_t saddr, uint32_t lbo) {
  uint64_t d = 0;
  d |= (uint64_t)((saddr & 0x3FFFF) >> 4);
  d |= (uint64_t)((lbo >> 4) & 0x3FFF) << 16;
  d |= (uint64_t)(1024 >> 4) << 32;
  d |= (uint64_t)1 << 46;
  d |= (uint64_t)2 << 61;
  return d;
}

// 2^x by the hardware approximation (subnormal results flush to zero: P
// values below 2^-126 carry no weight next to the row's maximum of 1 .. 256).
FP_DEV float pa_ex2(float x) {
  float y;
  asm("ex2.approx.ftz.f32 %0, %1;" : "=f"(y) : "f"(x));
  return y;
}

// (lo, hi) -> bf16x2, round to nearest even.
FP_DEV uint32_t pa_pack(float lo, float hi) {
  uint32_t r;
  asm("cvt.rn.bf16x2.f32 %0, %1, %2;" : "=r"(r) : "f"(hi), "f"(lo));
  return r;
}

// (lo, hi) -> fp16x2, round to nearest even.
FP_DEV uint32_t pa_pack_h(float lo, float hi) {
  uint32_t r;
  asm("cvt.rn.f16x2.f32 %0, %1, %2;" : "=r"(r) : "f"(hi), "f"(lo));
  return r;
}

// Signed bytes a and b of w as the fp16 pair (q_a, q_b), exact: the byte
// permute places q + 128 under the fp16 exponent of 1024 (0x64nn = 1024 + nn),
// one fp16x2 subtraction of 1152 leaves q.
FP_DEV uint32_t pa_i8h2(uint32_t u, uint32_t sel) {
  uint32_t h = __byte_perm(u, 0x64646464u, sel);
  asm("sub.rn.f16x2 %0, %0, %1;" : "+r"(h) : "r"(0x64806480u));
  return h;
}

// 32 rows of an output tile (this warp's TMEM lanes), COLS columns from x0 on, to out
// (rows from `pos` on, those below S; `ld` elements apart).  load(x, r) gives
// columns x .. x + 31 of the thread's row.  Through shared memory, four lanes to a
// row's 64 bytes (16 bytes of 32 rows a store took 5 us a tile); chunk c of row r
// is staged at c ^ (r / 2 % 4).
template <int COLS, typename F>
FP_DEV void pa_write_rows(F load, int x0, uint8_t* stage, uint16_t* out, long long ld, int pos, int S) {
  const int lane = threadIdx.x & 31;
#pragma unroll
  for (int x1 = 0; x1 < COLS; x1 += 32, x0 += 32) {
    float r[32];
    load(x0, r);
#pragma unroll
    for (int c = 0; c < 4; ++c) {
      uint32_t o[4];
#pragma unroll
      for (int y = 0; y < 4; ++y)
        o[y] = pa_pack(r[8 * c + 2 * y], r[8 * c + 2 * y + 1]);
      *reinterpret_cast<uint4*>(stage + lane * 64 + ((c ^ ((lane >> 1) & 3)) << 4)) = make_uint4(o[0], o[1], o[2], o[3]);
    }
    __syncwarp();
#pragma unroll
    for (int y = 0; y < 4; ++y) {
      const int rr = 8 * y + (lane >> 2), c = lane & 3;
      const uint4 o = *reinterpret_cast<const uint4*>(stage + rr * 64 + ((c ^ ((rr >> 1) & 3)) << 4));
      if (pos + rr < S) *reinterpret_cast<uint4*>(out + (long long)rr * ld + x0 + c * 8) = o;
    }
    __syncwarp();
  }
}

// 32 columns of an output accumulator in TMEM, times inv.
FP_DEV void pa_load_out(uint32_t to, float inv, float* r) {
  tc_ld<32>(to, reinterpret_cast<uint32_t*>(r));
#pragma unroll
  for (int y = 0; y < 32; ++y) r[y] *= inv;
}

// Prompts of at most kPaB tokens (fp_attn_short.cu), from launch_attention_prefill_tc.
cudaError_t launch_attention_prefill_short(const CUtensorMap& mq, const CUtensorMap& mk, const CUtensorMap& mv, int B,
                                           int S, int n_heads, const fp_kv_view& kv, uint16_t* out, int32_t* err,
                                           cudaStream_t s);

}  // namespace fpk
