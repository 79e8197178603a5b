// Prefill attention on the tcgen05 tensor cores: paged cache of bf16 or int8
// codes with per-(token, KV head) fp32 scales, head_dim 128.
//
// o = softmax(q K^T / sqrt(hd) + causal mask) V for the S query rows of every
// (sequence, head) against cache positions 0..S-1 (Sec. 5.1: the block's
// attention), for prompts of more than 128 tokens (fp_attn_short.cu takes most of
// the shorter ones).  One persistent CTA per SM walks work items of two query tiles
// of 128 rows that read the same keys and values: two heads of one KV head's
// group where groups are even, else 256 consecutive rows of a head.  Key tiles of
// 128.  Where pairs would leave SMs idle or one CTA's share too long, an item is
// one query tile whose key tiles the two softmax groups take in turn (`split`),
// each with its own maximum, row sum and accumulator; they are added at the end,
// half of the columns by each group.
// Tensor memory holds, for each of the two tiles, its scores (128 columns, P
// written over them as 16-bit pairs) and its output accumulator (128 columns):
//   warps 0-3   softmax of tile 0, warps 4-7 of tile 1: one query row (TMEM
//               lane) per thread, the tile's 128 scores held in registers
//               between the row maximum and P = 2^(s - m).  The reference
//               maximum m only moves when a tile raises it by more than 2^8 (O
//               and the row sum are rescaled then); P never exceeds 256, and
//               o / l is exact either way.  At the end of an item they write
//               their rows of O;
//   warp 8      TMA: the item's Q tiles (two 64-column boxes each), then (bf16
//               cache) per key tile its K rows and its V rows page by page (a
//               [16][64] box per 16-token page and half of head_dim, 128-byte
//               swizzle, one box per lane) into rings of two tiles each;
//   warp 9      owns the TMEM and issues the MMAs.  For each key tile and query
//               tile in turn: O += P(t) V(t) (A = P from TMEM, V read MN-major),
//               then S(t + 1) = Q K(t + 1)^T over the scores that P(t) V(t) has
//               read (one thread's MMAs execute in order), so one tile's softmax
//               runs while the other tile's two products do.
//   int8 cache: both products run on fp16 operands.  Warps 10-15 convert the
//               item's Q tiles to fp16 in place once, then widen the codes: each
//               loads its rows' 16-byte code chunks and turns each pair into the
//               fp16 pair (1024 + q + 128) by one byte permute, minus 1152 --
//               exact -- in the same swizzled layout the TMA writes, and stages
//               the tile's K scales and its V scales times 2^sigma; the softmax
//               multiplies each score column by its K scale and each P column by
//               its scaled V scale in fp32 (the row sum takes the unscaled P)
//               and packs P as fp16.  sigma, one per item, is the largest power
//               of two keeping 256 * (largest V scale of the item's keys) *
//               2^sigma within 65280, so P stays in the fp16 normal range; the
//               output divides it out.  A q beyond the fp16 range sets status 3.
// What bounds it: a key tile's products take 2 x 16 MMAs of 65 cycles for the two
// query tiles, 2080 cycles, which also fill shared memory's bandwidth; a step
// takes 4100 (the softmax of a tile about 1600, its P V and next scores 1040, and
// the hand-offs between the roles), with the int8 cache 8700 (the scales of the
// keys are read by every row, and the widening shares the issue slots).
// Measured, whole launches, bf16 cache, 4 x 2048 tokens, 64 / 8 heads | 8 x 1024,
// 40 heads | int8 cache, the first shape:
//   one 128-row tile per CTA, two CTAs per SM (before)       338 | 151 | 982 us
//   two tiles per CTA                                        333 | 161 | 725
//   every lane runs the MMA loop (one lane's issue took 144
//     cycles for an MMA that runs 65)                        297 | 138 | 641
//   output rows through shared memory                        285 | 126 | 617
//   the items longest first, block by block of heads         255 | 123 | 540
// A query tile's keys in turn by the two groups, bf16 | int8 cache: 8 heads, 1 x 1024
// tokens 19.7 | 39.5 us, 1 x 4096 61 | 133, 40 heads, 1 x 1024 27.1 | 52 (one 128-row
// tile per CTA 20.4 | 49.5, 70 | 211, 31.5 | 71; with two V tiles in the ring, as for
// pairs, 23.7, 82 and 31.2 with the bf16 cache: V held up the copies of K).
// Key tiles in halves of 64, so that a tile's own two products overlap its
// softmax, took 360 us: the waits cost more than they hid.
// Every mbarrier wait is bounded (error 2 past the limit); a page id out of
// range reads zeros and sets error 1.
#include <algorithm>
#include <type_traits>

#include "attn_items.h"
#include "attn_tc.cuh"
#include "common.cuh"

namespace fpk {

constexpr int kPaWarpTma = 8, kPaWarpMma = 9, kPaWarpWiden = 10;
constexpr int kPaWiden = 6;                                 // int8 cache: warps widening codes
constexpr int kPaWRows = (kPaB + 4 * kPaWiden - 1) / (4 * kPaWiden);  // tile rows per widening thread
template <bool KV8>
constexpr int pa_threads() { return KV8 ? (kPaWarpWiden + kPaWiden) * 32 : 384; }
// Registers a thread, moved to the softmax, which holds a row of scores: bf16
// cache 168 at launch (384 threads), 2 x 208 + 88 = 3 x 168; int8 cache 128 (512
// threads), 2 x 160 + 2 x 96 = 4 x 128
template <bool KV8>
constexpr int pa_reg_soft() { return KV8 ? 160 : 208; }
template <bool KV8>
constexpr int pa_reg_other() { return KV8 ? 96 : 88; }
constexpr uint32_t kPaTmemCols = 512;
constexpr uint32_t kPaO = 256;               // O of tile j at kPaO + 128 j, its scores at 128 j
constexpr int kPaRing = 2;                   // K tiles in shared memory, and V tiles; a shared query
                                             // tile leaves room for a third V tile
constexpr int kPaScl = 4;                    // tiles of int8 scales
constexpr int kPaSmem = (2 + 2 * kPaRing) * kPaTile + 8 * kPaStage + 1024;  // Q, K, V, output, alignment
constexpr float kPaSlack = 8.f;  // log2 of the largest P allowed before the reference maximum moves

// Two fp32 lanes at once: a b + c, a b, a + b.
FP_DEV float2 pa_fma2(float2 a, float2 b, float2 c) {
  float2 d;
  asm("{\n .reg .b64 a, b, c, d;\n mov.b64 a, {%2, %3};\n mov.b64 b, {%4, %5};\n mov.b64 c, {%6, %7};\n"
      " fma.rn.f32x2 d, a, b, c;\n mov.b64 {%0, %1}, d;\n}\n"
      : "=f"(d.x), "=f"(d.y)
      : "f"(a.x), "f"(a.y), "f"(b.x), "f"(b.y), "f"(c.x), "f"(c.y));
  return d;
}
FP_DEV float2 pa_mul2(float2 a, float2 b) {
  float2 d;
  asm("{\n .reg .b64 a, b, d;\n mov.b64 a, {%2, %3};\n mov.b64 b, {%4, %5};\n"
      " mul.rn.f32x2 d, a, b;\n mov.b64 {%0, %1}, d;\n}\n"
      : "=f"(d.x), "=f"(d.y)
      : "f"(a.x), "f"(a.y), "f"(b.x), "f"(b.y));
  return d;
}
FP_DEV float2 pa_add2(float2 a, float2 b) {
  float2 d;
  asm("{\n .reg .b64 a, b, d;\n mov.b64 a, {%2, %3};\n mov.b64 b, {%4, %5};\n"
      " add.rn.f32x2 d, a, b;\n mov.b64 {%0, %1}, d;\n}\n"
      : "=f"(d.x), "=f"(d.y)
      : "f"(a.x), "f"(a.y), "f"(b.x), "f"(b.y));
  return d;
}

// split: the two softmax groups share a query tile (plan.pair == 0)
template <bool KV8, bool split>
__global__ void __launch_bounds__(pa_threads<KV8>(), 1)
    attn_prefill_tc_kernel(const __grid_constant__ CUtensorMap map_q, const __grid_constant__ CUtensorMap map_k,
                           const __grid_constant__ CUtensorMap map_v, const int8_t* __restrict__ k8,
                           const int8_t* __restrict__ v8, const float* __restrict__ k_scale,
                           const float* __restrict__ v_scale, int S, int H, int Hkv, int page_size,
                           const int32_t* __restrict__ page_table, int pages_per_seq, int n_pages, PaPlan plan,
                           uint16_t* __restrict__ out, int32_t* err) {
  constexpr int RV = split ? kPaRing + 1 : kPaRing;
  extern __shared__ __align__(1024) uint8_t smem_raw[];
  __shared__ uint64_t qfull, qconv, qempty, kfull[kPaRing], kempty[kPaRing], vfull[RV], vempty[RV], sfull[2],
      pfull[2], ofull[2], oempty[2], vmet, met, mma_done;
  __shared__ float s_vmax[2][kPaWiden];  // int8: the widening warps' largest V scales, by item parity
  __shared__ float s_unscale[4];          // int8: 2^-sigma, removed from the output; by item % 4
  __shared__ float2 s_ml[2][2][split ? kPaB : 1];  // reference maximum and row sum; by item parity, group
  __shared__ uint32_t tmem_base;
  __shared__ int abort_word;
  __shared__ __align__(16) float s_scl[KV8 ? 2 * kPaScl * kPaB : 4];  // int8: [K, V][tile % 4][key] scales
  volatile int* abort_flag = &abort_word;
  uint8_t* smem = (uint8_t*)(((uintptr_t)smem_raw + 1023) & ~(uintptr_t)1023);
  uint8_t* sQ = smem;
  uint8_t* sK = smem + (split ? 1 : 2) * kPaTile;
  uint8_t* sV = sK + kPaRing * kPaTile;
  const int warp = threadIdx.x >> 5, lane = threadIdx.x & 31;
  auto item = [](int n) { return pa_item(n, blockIdx.x, gridDim.x); };
  auto fail = [&]() {
    *abort_flag = 1;
    if (err) atomicExch(err, 2);
  };

  pdl_trigger();
  if (threadIdx.x == 0) {
    mbar_init(&qfull, 1);
    mbar_init(&qconv, kPaWiden);  // int8: the widening warps converted Q to fp16
    mbar_init(&qempty, 1);
    mbar_init(&vmet, kPaWiden);
    for (int i = 0; i < kPaRing; ++i) {
      mbar_init(&kfull[i], KV8 ? kPaWiden : 1);
      mbar_init(&kempty[i], 1);
    }
    for (int i = 0; i < RV; ++i) {
      mbar_init(&vfull[i], KV8 ? kPaWiden : 1);
      mbar_init(&vempty[i], 1);
    }
    for (int j = 0; j < 2; ++j) {
      mbar_init(&sfull[j], 1);
      mbar_init(&pfull[j], 4);
      mbar_init(&ofull[j], 1);
      mbar_init(&oempty[j], split ? 8 : 4);
    }
    mbar_init(&met, 8);
    mbar_init(&mma_done, 1);
    *abort_flag = 0;
    asm volatile("fence.mbarrier_init.release.cluster;" ::: "memory");
  }
  if (warp == kPaWarpMma) {
    asm volatile("tcgen05.alloc.cta_group::1.sync.aligned.shared::cta.b32 [%0], %1;" ::"r"(smem_u32(&tmem_base)),
                 "r"(kPaTmemCols)
                 : "memory");
    asm volatile("tcgen05.relinquish_alloc_permit.cta_group::1.sync.aligned;" ::: "memory");
  }
  tc_fence_before();
  __syncthreads();
  tc_fence_after();
  const uint32_t tmem = tmem_base;
  pdl_wait();

  if (warp >= kPaWarpTma) asm volatile("setmaxnreg.dec.sync.aligned.u32 %0;" ::"n"(pa_reg_other<KV8>()));
  if (warp == kPaWarpTma) {
    // ---------------- TMA producer: lane 0 copies Q; lanes 0-15 each copy one
    // [16][64] box of a key tile (page lane & 7, head_dim half lane >> 3).  The
    // next tile's page ids are read while this one is in flight.
    if (lane == 0 && !KV8) {
      asm volatile("prefetch.tensormap [%0];" ::"l"(&map_k) : "memory");
      asm volatile("prefetch.tensormap [%0];" ::"l"(&map_v) : "memory");
    }
    const int pg = lane & 7, half = (lane >> 3) & 1;
    int n = 0, kn = 0, iss[3] = {0, 0, 0};  // items, key tiles; copies issued of Q, K, V
    bool ok = true;
    for (int i = item(0); i < plan.items && ok; i = item(++n)) {
      const PaItem w(i, S, H, Hkv, plan);
      if (n > 0) ok = __all_sync(0xffffffffu, mbar_wait(&qempty, (n - 1) & 1)) && !*abort_flag;
      if (!__all_sync(0xffffffffu, ok)) break;
      iss[0] = n + 1;
      if (lane == 0) {
        mbar_expect_tx(&qfull, (w.nt[1] > 0 ? 2 : 1) * kPaTile);
#pragma unroll
        for (int j = 0; j < 2; ++j)
          if (w.nt[j] > 0) {
            tma_load_2d(sQ + j * kPaTile, &map_q, w.h[j] * kPaHD, w.b * S + w.q0[j], &qfull);
            tma_load_2d(sQ + j * kPaTile + kPaHalf, &map_q, w.h[j] * kPaHD + 64, w.b * S + w.q0[j], &qfull);
          }
      }
      if constexpr (!KV8) {
        const int32_t* pt = page_table + (long long)w.b * pages_per_seq;
        auto page_row = [&](int t) {  // pool row of this lane's page of tile t; -16 reads zeros
          const int key0 = t * kPaB + pg * 16;
          if (lane >= 16 || key0 >= S) return -16;
          const int id = __ldg(pt + key0 / page_size);
          if (id >= 0 && id < n_pages) return (id * Hkv + w.kvh) * page_size;
          if (err && half == 0) atomicExch(err, 1);
          return -16;
        };
        const int nt = w.tiles();
        int row = page_row(0);
        for (int t = 0; t < nt && ok; ++t, ++kn) {
#pragma unroll
          for (int v = 0; v < 2 && ok; ++v) {
            const int ring = v ? RV : kPaRing, s = kn % ring, ph = ((kn / ring) & 1) ^ 1;
            uint64_t* full = v ? &vfull[s] : &kfull[s];
            if (kn >= ring) ok = mbar_wait(v ? &vempty[s] : &kempty[s], ph);
            ok = __all_sync(0xffffffffu, ok && !*abort_flag);
            if (!ok) break;
            if (lane == 0) mbar_expect_tx(full, kPaTile);
            __syncwarp();
            if (lane < 16)
              tma_load_2d((v ? sV : sK) + s * kPaTile + half * kPaHalf + pg * 2048, v ? &map_v : &map_k, half * 64, row,
                          full);
            iss[1 + v] = kn + 1;
          }
          if (t + 1 < nt) row = page_row(t + 1);
        }
      }
    }
    if (lane == 0) {
      if (!ok) fail();
      // copies still in flight land before the CTA leaves
      if (iss[0] > 0) mbar_wait(&qfull, (iss[0] - 1) & 1);
#pragma unroll
      for (int v = 0; v < 2; ++v)
        for (int t = max(0, iss[1 + v] - (v ? RV : kPaRing)); t < iss[1 + v]; ++t)
          mbar_wait(v ? &vfull[t % RV] : &kfull[t % kPaRing], (t / (v ? RV : kPaRing)) & 1);
    }
  } else if (warp == kPaWarpMma) {
    // ---------------- MMA issuer: every lane runs the loop, one issues.
    // Q, K both K-major; V MN-major.  int8 cache: fp16 operands (A and B
    // of one MMA always share their type), bf16 cache: bf16
    constexpr uint32_t f16 = KV8 ? ((1u << 7) | (1u << 10)) : 0u;
    constexpr uint32_t idesc_s = tc_idesc(kPaB, kPaB) & ~f16;
    constexpr uint32_t idesc_o = (tc_idesc(kPaB, kPaHD) | (1u << 16)) & ~f16;
    const uint64_t qd = sdesc(smem_u32(sQ)), kd = sdesc(smem_u32(sK)), vd = sdesc_mn(smem_u32(sV), kPaHalf);
    int n = 0, kn = 0, pn[2] = {0, 0}, on[2] = {0, 0};
    bool ok = true;
    // descriptor start addresses count 16-byte units
    auto scores = [&](int j, int s) {  // S_j = Q_j K^T of ring tile s (issuing lane only)
      const uint64_t qj = qd + (split ? 0 : j) * (kPaTile >> 4), ks = kd + s * (kPaTile >> 4);
#pragma unroll
      for (int kk = 0; kk < kPaHD / 16; ++kk) {
        const int off = ((kk >> 2) * kPaHalf + (kk & 3) * 32) >> 4;
        tc_mma(tmem + j * kPaB, qj + off, ks + off, idesc_s, kk > 0 ? 1u : 0u);
      }
      tc_commit(&sfull[j]);
    };
    auto values = [&](int j, int s, bool first) {  // O_j (+)= P_j V of ring tile s (issuing lane only)
      const uint64_t vs = vd + s * (kPaTile >> 4);
#pragma unroll
      for (int kk = 0; kk < kPaB / 16; ++kk)  // 16 keys: two 8-row groups of the V tile
        tc_mma_ts(tmem + kPaO + j * kPaHD, tmem + j * kPaB + kk * 8, vs + kk * (2048 >> 4), idesc_o,
                  (!first || kk > 0) ? 1u : 0u);
    };
    for (int i = item(0); i < plan.items && ok; i = item(++n)) {
      const PaItem w(i, S, H, Hkv, plan);
      const int nt = w.tiles();
      ok = mbar_wait(KV8 ? &qconv : &qfull, n & 1) && mbar_wait(&kfull[kn % kPaRing], (kn / kPaRing) & 1) && !*abort_flag;
      ok = __all_sync(0xffffffffu, ok);
      if (!ok) break;
      tc_fence_after();
      if constexpr (split) {
        // one query tile: key tile t is group t % 2's, scores two tiles ahead
        if (elect_one()) {
          scores(0, kn % kPaRing);
          tc_commit(&kempty[kn % kPaRing]);
          if (nt == 1) tc_commit(&qempty);
        }
        __syncwarp();
        if (nt > 1) {
          ok = __all_sync(0xffffffffu, mbar_wait(&kfull[(kn + 1) % kPaRing], ((kn + 1) / kPaRing) & 1));
          if (!ok) break;
          if (elect_one()) {
            scores(1, (kn + 1) % kPaRing);
            tc_commit(&kempty[(kn + 1) % kPaRing]);
            if (nt == 2) tc_commit(&qempty);
          }
          __syncwarp();
        }
        for (int t = 0; t < nt && ok; ++t, ++kn) {
          const int s = kn % kPaRing, sv = kn % RV, j = t & 1;  // s: of key tiles t and t + 2
          const int p = j ? pn[1] : pn[0], o = j ? on[1] : on[0];
          ok = mbar_wait(&vfull[sv], (kn / RV) & 1) &&
               (t + 2 >= nt || mbar_wait(&kfull[s], ((kn + kPaRing) / kPaRing) & 1)) && mbar_wait(&pfull[j], p & 1) &&
               (t > 1 || o == 0 || mbar_wait(&oempty[j], (o - 1) & 1)) && !*abort_flag;
          ok = __all_sync(0xffffffffu, ok);
          if (!ok) break;
          tc_fence_after();
          if (elect_one()) {
            values(j, sv, t < 2);
            tc_commit(&vempty[sv]);
            if (t + 2 < nt) {
              scores(j, s);
              tc_commit(&kempty[s]);
            } else {
              tc_commit(&ofull[j]);
            }
            if (t + 3 == nt) tc_commit(&qempty);
          }
          __syncwarp();
          if (j) ++pn[1], on[1] += t + 2 >= nt;
          else ++pn[0], on[0] += t + 2 >= nt;
        }
        continue;
      }
      if (elect_one()) {
#pragma unroll
        for (int j = 0; j < 2; ++j)
          if (w.nt[j] > 0) scores(j, kn % kPaRing);
        tc_commit(&kempty[kn % kPaRing]);
        if (nt == 1) tc_commit(&qempty);
      }
      __syncwarp();
      for (int t = 0; t < nt && ok; ++t, ++kn) {
        const int s = kn % kPaRing, s1 = (kn + 1) % kPaRing;
        ok = mbar_wait(&vfull[s], (kn / kPaRing) & 1);
        if (t + 1 < nt) ok = ok && mbar_wait(&kfull[s1], ((kn + 1) / kPaRing) & 1);
#pragma unroll
        for (int j = 0; j < 2; ++j) {
          if (t >= w.nt[j] || !ok) continue;
          // P_j(t) is written, and (first tile) the last item's output has been read
          ok = mbar_wait(&pfull[j], pn[j] & 1) && (t > 0 || on[j] == 0 || mbar_wait(&oempty[j], (on[j] - 1) & 1)) &&
               !*abort_flag;
          ok = __all_sync(0xffffffffu, ok);
          if (!ok) continue;
          ++pn[j];
          tc_fence_after();
          if (elect_one()) {
            values(j, s, t == 0);
            if (t + 1 < w.nt[j]) scores(j, s1);
            else tc_commit(&ofull[j]);
          }
          __syncwarp();
          if (t + 1 >= w.nt[j]) ++on[j];
        }
        ok = __all_sync(0xffffffffu, ok);
        if (!ok) break;
        if (elect_one()) {
          tc_commit(&vempty[s]);
          if (t + 1 < nt) tc_commit(&kempty[s1]);
          if (t + 2 == nt) tc_commit(&qempty);  // the item's last scores: Q may be overwritten
        }
        __syncwarp();
      }
    }
    if (!ok && lane == 0) fail();
    if (elect_one()) tc_commit(&mma_done);
    __syncwarp();
    mbar_wait(&mma_done, 0);
  } else if (KV8 && warp >= kPaWarpWiden) {
    // ---------------- int8 cache: Q to fp16, then widening of the key tiles
    const int wi = (warp - kPaWarpWiden) * 32 + lane;  // 0 .. 191
    constexpr int WT = 32 * kPaWiden;
    const int c = wi & 7;                                     // code chunk: head_dim 16c .. 16c + 15
    const int rbase = wi >> 3;                                // tile rows rbase + 24i (< 128)
    // its bf16 form is chunks cb, cb + 1 of half c / 4 of the swizzled row;
    // the lanes of the upper half store the odd chunk first, so the eight
    // lanes of one row write eight distinct 16-byte bank groups
    const int cb = 2 * (c & 3), half_off = (c >> 2) * kPaHalf;
    int n = 0, kn = 0;
    bool ok = true;
    for (int i = item(0); i < plan.items && ok; i = item(++n)) {
      const PaItem w(i, S, H, Hkv, plan);
      const int nt = w.tiles();
      const int32_t* pt = page_table + (long long)w.b * pages_per_seq;
      // sigma: from the largest V scale over the keys the item reads
      float vmax = 0.f;
      const int nkeys = min(nt * kPaB, S);
#pragma unroll 4
      for (int key = wi; key < nkeys; key += WT) {
        const int pg = __ldg(pt + key / page_size);
        if (pg >= 0 && pg < n_pages) vmax = fmaxf(vmax, __ldg(v_scale + (pg * Hkv + w.kvh) * page_size + key % page_size));
      }
      vmax = warp_max(vmax);
      // (a warp that reaches the next item's meeting has read this item's values)
      if (lane == 0) {
        s_vmax[n & 1][warp - kPaWarpWiden] = vmax;
        mbar_arrive(&vmet);
      }
      ok = __all_sync(0xffffffffu, mbar_wait(&vmet, n & 1));
#pragma unroll
      for (int x = 0; x < kPaWiden; ++x) vmax = fmaxf(vmax, s_vmax[n & 1][x]);
      // 2^sigma with 256 * vmax * 2^sigma <= 65280 (vmax = 0: no V weight at all)
      const int sigma = vmax > 0.f ? min(60, max(-60, (int)floorf(log2f(255.f / vmax)))) : 0;
      const float vmul = exp2f((float)sigma);
      // Q to fp16 in place (the element order of the swizzled tiles is kept)
      ok = ok && __all_sync(0xffffffffu, mbar_wait(&qfull, n & 1));
      if (ok) {
        bool over = false;
        const int q16 = (w.nt[1] > 0 ? 2 : 1) * (kPaTile / 16);
#pragma unroll 4
        for (int x = wi; x < q16; x += WT) {
          uint4* p = reinterpret_cast<uint4*>(sQ) + x;
          const uint4 v = *p;
          const uint32_t w4[4] = {v.x, v.y, v.z, v.w};
          uint32_t o[4];
#pragma unroll
          for (int j = 0; j < 4; ++j) {
            const float2 f = bf2x2f(w4[j]);
            over |= fabsf(f.x) > 65504.f || fabsf(f.y) > 65504.f;
            o[j] = pa_pack_h(f.x, f.y);
          }
          *p = make_uint4(o[0], o[1], o[2], o[3]);
        }
        if (over && err) atomicExch(err, 3);  // q outside the fp16 range: the output is invalid
        // published with Q, which every score of the item follows; this slot's
        // last reader was the epilogue of item n - 4: the scores of item n - 1,
        // whose last use of Q preceded this item's Q, follow P of item n - 2 and
        // so that tile's epilogue of item n - 3
        if (wi == 0) s_unscale[n & 3] = exp2f((float)-sigma);
        fence_proxy_async();
      }
      __syncwarp();
      if (lane == 0) mbar_arrive(&qconv);
      for (int t = 0; t < nt && ok; ++t, ++kn) {
        int rowi[kPaWRows];  // pool row of each of the thread's keys (< 2^31); -1 reads zeros
#pragma unroll
        for (int r = 0; r < kPaWRows; ++r) {
          const int row = rbase + 4 * kPaWiden * r, key = t * kPaB + row;
          rowi[r] = -1;
          if (row < kPaB && key < S) {
            const int pg = __ldg(pt + key / page_size);
            if (pg >= 0 && pg < n_pages) rowi[r] = (pg * Hkv + w.kvh) * page_size + key % page_size;
            else if (err && c == 0) atomicExch(err, 1);
          }
        }
        // the tile's K and V scales go out with its K codes: the softmax reads
        // both once S(t) is complete, which only the K tile's barrier precedes
        float sck[kPaWRows], scv[kPaWRows];
#pragma unroll
        for (int r = 0; r < kPaWRows; ++r) {
          sck[r] = (c == 0 && rowi[r] >= 0) ? __ldg(k_scale + rowi[r]) : 0.f;
          scv[r] = (c == 0 && rowi[r] >= 0) ? __ldg(v_scale + rowi[r]) * vmul : 0.f;
        }
#pragma unroll 1
        for (int which = 0; which < 2; ++which) {
          const int8_t* pool = which ? v8 : k8;
          const int ring = which ? RV : kPaRing, s = kn % ring, ph = ((kn / ring) & 1) ^ 1;
          uint4 cw[kPaWRows];
          // the codes are read before the wait for the buffer
#pragma unroll
          for (int r = 0; r < kPaWRows; ++r)
            cw[r] = rowi[r] >= 0 ? ld_nc16(pool + (long long)rowi[r] * kPaHD + c * 16) : make_uint4(0, 0, 0, 0);
          if (kn >= ring) ok = mbar_wait(which ? &vempty[s] : &kempty[s], ph);
          if (!__all_sync(0xffffffffu, ok) || __any_sync(0xffffffffu, *abort_flag != 0)) {
            ok = false;
            break;
          }
          uint8_t* dst = (which ? sV : sK) + s * kPaTile + half_off;
#pragma unroll
          for (int r = 0; r < kPaWRows; ++r) {
            const int row = rbase + 4 * kPaWiden * r, sw = row & 7;
            if (row >= kPaB) break;
            const uint32_t ww[4] = {cw[r].x ^ 0x80808080u, cw[r].y ^ 0x80808080u, cw[r].z ^ 0x80808080u,
                                    cw[r].w ^ 0x80808080u};
            uint32_t o[8];
#pragma unroll
            for (int j = 0; j < 8; ++j) o[j] = pa_i8h2(ww[j >> 1], (j & 1) ? 0x4342 : 0x4140);
            const uint4 e = make_uint4(o[0], o[1], o[2], o[3]), f = make_uint4(o[4], o[5], o[6], o[7]);
            uint8_t* rp = dst + row * 128;
            if (c < 4) {
              *reinterpret_cast<uint4*>(rp + ((cb ^ sw) << 4)) = e;
              *reinterpret_cast<uint4*>(rp + (((cb + 1) ^ sw) << 4)) = f;
            } else {
              *reinterpret_cast<uint4*>(rp + (((cb + 1) ^ sw) << 4)) = f;
              *reinterpret_cast<uint4*>(rp + ((cb ^ sw) << 4)) = e;
            }
            if (which == 0 && c == 0) {
              // slot kn % 4 was last read by the softmax of tile kn - 4; K tile
              // kn - 2 has been multiplied, which its P V (of tile kn - 3) preceded
              s_scl[(kn % kPaScl) * kPaB + row] = sck[r];
              s_scl[(kPaScl + kn % kPaScl) * kPaB + row] = scv[r];
            }
          }
          fence_proxy_async();  // the MMAs read the tile through the async proxy
          __syncwarp();
          if (lane == 0) mbar_arrive(which ? &vfull[s] : &kfull[s]);
        }
      }
    }
    if (!ok && lane == 0) fail();
  } else if (warp < kPaWarpTma) {
    // ---------------- softmax: thread = query row (TMEM lane 32 (warp % 4) + lane) of tile j
    asm volatile("setmaxnreg.inc.sync.aligned.u32 %0;" ::"n"(pa_reg_soft<KV8>()));
    const int j = warp >> 2, quad = warp & 3, row = quad * 32 + lane;
    const uint32_t lane_base = tmem + ((uint32_t)(quad * 32) << 16);
    const uint32_t ts = lane_base + j * kPaB, to = lane_base + kPaO + j * kPaHD;
    const float scale = kPaLog2e * rsqrtf((float)kPaHD);
    const int jq = split ? 0 : j, first = split ? j : 0, stride = split ? 2 : 1;  // query tile; this group's key tiles
    int n = 0, kn = 0, sn = 0, on = 0;  // items, key tiles, this group's scores and outputs
    bool ok = true;
    for (int i = item(0); i < plan.items && ok; i = item(++n)) {
      const PaItem w(i, S, H, Hkv, plan);
      const int nt = w.key_tiles(jq), qrow = w.row0(jq) + row;  // position in the sequence
      float m = -INFINITY;                            // reference maximum (log2 domain)
      float2 l2[4];                                   // row sum
#pragma unroll
      for (int y = 0; y < 4; ++y) l2[y] = make_float2(0.f, 0.f);
      for (int t = first; t < nt; t += stride, ++sn) {
        ok = mbar_wait(&sfull[j], sn & 1);
        if (!__all_sync(0xffffffffu, ok)) {
          ok = false;
          break;
        }
        tc_fence_after();
        uint32_t r[kPaB];
        tc_ld<64>(ts, r);
        tc_ld<64>(ts + 64, r + 64);
        float* v = reinterpret_cast<float*>(r);
        const int key0 = t * kPaB;
        const float* ks = s_scl + ((kn + t) % kPaScl) * kPaB;
        if constexpr (KV8) {
#pragma unroll
          for (int x = 0; x < kPaB; x += 4) {  // K scale of each key column
            const float4 f = *reinterpret_cast<const float4*>(ks + x);
            const float2 a = pa_mul2(make_float2(v[x], v[x + 1]), make_float2(f.x, f.y));
            const float2 b = pa_mul2(make_float2(v[x + 2], v[x + 3]), make_float2(f.z, f.w));
            v[x] = a.x, v[x + 1] = a.y, v[x + 2] = b.x, v[x + 3] = b.y;
          }
        }
        if (t == nt - 1) {  // the diagonal tile: keys after this row (and so past S) are masked
#pragma unroll
          for (int x = 0; x < kPaB; ++x)
            if (key0 + x > qrow) v[x] = -INFINITY;
        }
        float m4[4] = {-INFINITY, -INFINITY, -INFINITY, -INFINITY};
#pragma unroll
        for (int x = 0; x < kPaB; x += 8)
#pragma unroll
          for (int y = 0; y < 4; ++y) m4[y] = fmaxf(m4[y], fmaxf(v[x + 2 * y], v[x + 2 * y + 1]));
        const float mx = fmaxf(fmaxf(m4[0], m4[1]), fmaxf(m4[2], m4[3])) * scale;
        // move the reference when the tile would exceed it by more than 2^kPaSlack
        float corr = 1.f;
        if (mx > m + kPaSlack) {
          corr = exp2f(m - mx);  // 0 on the first tile
          m = mx;
#pragma unroll
          for (int y = 0; y < 4; ++y) l2[y] = pa_mul2(l2[y], make_float2(corr, corr));
        }
        if (t > first && __any_sync(0xffffffffu, corr != 1.f)) {
          // O holds P V of the earlier tiles (complete: S(t) was issued after it)
#pragma unroll 1
          for (int x = 0; x < kPaHD / 16; ++x) {
            uint32_t o[16];
            tc_ld<16>(to + x * 16, o);
#pragma unroll
            for (int y = 0; y < 16; ++y) o[y] = __float_as_uint(__uint_as_float(o[y]) * corr);
            tc_st16(to + x * 16, o);
          }
        }
        // P = 2^(s scale - m) as 16-bit pairs over the score columns
        const float mref = m == -INFINITY ? 0.f : m;
        const float2 sc2 = make_float2(scale, scale), nm2 = make_float2(-mref, -mref);
        const float* vs = s_scl + (kPaScl + (kn + t) % kPaScl) * kPaB;
#pragma unroll
        for (int x0 = 0; x0 < kPaB; x0 += 32) {
          uint32_t pw[16];
#pragma unroll
          for (int x = 0; x < 32; x += 2) {
            const float2 e = pa_fma2(make_float2(v[x0 + x], v[x0 + x + 1]), sc2, nm2);
            float2 p = make_float2(pa_ex2(e.x), pa_ex2(e.y));
            l2[(x >> 1) & 3] = pa_add2(l2[(x >> 1) & 3], p);
            if constexpr (KV8) {
              // V scale of each key column: P V then takes the codes as they are
              p = pa_mul2(p, *reinterpret_cast<const float2*>(vs + x0 + x));
              pw[x / 2] = pa_pack_h(p.x, p.y);
            } else {
              pw[x / 2] = pa_pack(p.x, p.y);
            }
          }
          tc_st16(ts + x0 / 2, pw);
        }
        tc_wait_st();
        tc_fence_before();
        __syncwarp();
        if (lane == 0) mbar_arrive(&pfull[j]);
      }
      kn += w.tiles();
      if (!ok) break;
      if (nt == 0) continue;
      const float l = ((l2[0].x + l2[0].y) + (l2[1].x + l2[1].y)) + ((l2[2].x + l2[2].y) + (l2[3].x + l2[3].y));
      // ---- the item's output
      const int pos = w.row0(jq) + quad * 32;
      uint8_t* stage = sV + RV * kPaTile + warp * kPaStage;
      uint16_t* dst = out + ((long long)w.b * S + pos) * ((long long)H * kPaHD) + (long long)w.head(jq) * kPaHD;
      const long long ld = (long long)H * kPaHD;
      // int8 cache: P carried the V scales times 2^sigma
      if constexpr (split) {
        // the groups' sums over their key tiles, each with its own reference
        // maximum, added; each group finishes half of the columns
        const bool both = nt > 1;
        s_ml[n & 1][j][row] = make_float2(m, l);
        __syncwarp();
        if (lane == 0) mbar_arrive(&met);
        ok = __all_sync(0xffffffffu, mbar_wait(&met, n & 1) && mbar_wait(&ofull[0], n & 1) &&
                                         (!both || mbar_wait(&ofull[1], on & 1)));
        if (!ok) break;
        on += both;
        tc_fence_after();
        const float2 ml0 = s_ml[n & 1][0][row], ml1 = s_ml[n & 1][1][row];
        const float mm = fmaxf(ml0.x, ml1.x);
        float a0 = 1.f, a1 = 0.f, ls = ml0.y;
        if (both) {
          a0 = exp2f(ml0.x - mm), a1 = exp2f(ml1.x - mm);
          ls = a0 * ml0.y + a1 * ml1.y;
        }
        const float inv = (KV8 ? s_unscale[n & 3] : 1.f) / ls;
        a0 *= inv, a1 *= inv;
        pa_write_rows<kPaHD / 2>(
            [&](int x, float* r) {
              pa_load_out(lane_base + kPaO + x, a0, r);
              if (both) {
                uint32_t u[32];
                tc_ld<32>(lane_base + kPaO + kPaHD + x, u);
#pragma unroll
                for (int y = 0; y < 32; ++y) r[y] = fmaf(a1, __uint_as_float(u[y]), r[y]);
              }
            },
            j * (kPaHD / 2), stage, dst, ld, pos, S);
        tc_fence_before();
        __syncwarp();
        if (lane == 0) {
          mbar_arrive(&oempty[0]);
          if (both) mbar_arrive(&oempty[1]);
        }
        continue;
      }
      ok = __all_sync(0xffffffffu, mbar_wait(&ofull[j], on & 1));
      if (!ok) break;
      ++on;
      tc_fence_after();
      const float inv = (KV8 ? s_unscale[n & 3] : 1.f) / l;
      pa_write_rows<kPaHD>(
          [&](int x, float* r) {
            pa_load_out(to + x, inv, r);
            if (x + 32 == kPaHD) {
              tc_fence_before();
              __syncwarp();
              if (lane == 0) mbar_arrive(&oempty[j]);
            }
          },
          0, stage, dst, ld, pos, S);
    }
    if (!ok && lane == 0) fail();
  }
  tc_fence_before();
  __syncthreads();
  if (warp == kPaWarpMma) {
    tc_fence_after();
    asm volatile("tcgen05.dealloc.cta_group::1.sync.aligned.b32 %0, %1;" ::"r"(tmem), "r"(kPaTmemCols) : "memory");
  }
}

bool attention_prefill_tc_ok(int B, int S, int n_heads, const fp_kv_view& kv, const void* q, int q_stride) {
  const bool kv8 = kv.kvquant == FP_KV_INT8;
  return (kv.kvquant == FP_KV_BF16 || (kv8 && kv.k_scale && kv.v_scale)) && kv.head_dim == kPaHD &&
         kv.page_size == 16 && B >= 1 && S >= 1 && n_heads % kv.n_kv_heads == 0 && q_stride % 8 == 0 &&
         ((uintptr_t)q & 15) == 0 && ((uintptr_t)kv.k_pool & 15) == 0 && ((uintptr_t)kv.v_pool & 15) == 0 &&
         (long long)kv.n_pages * kv.n_kv_heads * kv.page_size < (1LL << 31) &&
         (long long)B * n_heads * ((S + kPaB - 1) / kPaB) < (1LL << 26) && tensor_maps_available();
}

template <bool KV8, bool SPLIT>
static cudaError_t launch_pa_plan(const PaPlan& plan, int ctas, const CUtensorMap& mq, const CUtensorMap& mk,
                                  const CUtensorMap& mv, int S, int n_heads, const fp_kv_view& kv, uint16_t* out,
                                  int32_t* err, cudaStream_t s) {
  static std::atomic<unsigned long long> attr{0};
  FP_CUDA_TRY(smem_limit_once(attn_prefill_tc_kernel<KV8, SPLIT>, kPaSmem, &attr));
  return launch(attn_prefill_tc_kernel<KV8, SPLIT>, dim3(ctas), dim3(pa_threads<KV8>()), (size_t)kPaSmem, s, mq, mk, mv,
                (const int8_t*)kv.k_pool, (const int8_t*)kv.v_pool, (const float*)kv.k_scale, (const float*)kv.v_scale,
                S, n_heads, kv.n_kv_heads, kv.page_size, kv.page_table, kv.pages_per_seq, kv.n_pages, plan, out, err);
}

static int pa_sms() {
  static int sms = 0;
  if (!sms) {
    int dev = 0;
    if (cudaGetDevice(&dev) != cudaSuccess || cudaDeviceGetAttribute(&sms, cudaDevAttrMultiProcessorCount, dev) != cudaSuccess ||
        sms <= 0)
      sms = 152;
  }
  return sms;
}

template <bool KV8>
static cudaError_t launch_pa_tc(const CUtensorMap& mq, const CUtensorMap& mk, const CUtensorMap& mv, int B, int S,
                                int n_heads, const fp_kv_view& kv, uint16_t* out, int32_t* err, cudaStream_t s) {
  const int sms = pa_sms();
  const PaPlan plan = pa_plan(B, S, n_heads, n_heads / kv.n_kv_heads, sms);
  const int ctas = std::min(plan.items, sms);
  return plan.pair ? launch_pa_plan<KV8, false>(plan, ctas, mq, mk, mv, S, n_heads, kv, out, err, s)
                   : launch_pa_plan<KV8, true>(plan, ctas, mq, mk, mv, S, n_heads, kv, out, err, s);
}

cudaError_t launch_attention_prefill_tc(const uint16_t* q, int q_stride, int B, int S, int n_heads,
                                        const fp_kv_view& kv, uint16_t* out, int32_t* err, cudaStream_t s) {
  CUtensorMap mq, mk, mv;
  const long long pool_rows = (long long)kv.n_pages * kv.n_kv_heads * kv.page_size;
  // q [B S][q_stride] bf16, box [128 rows][64]
  if (!make_tensor_map(&mq, q, (long long)B * S, q_stride, 2, kPaB, 64, 128)) return cudaErrorInvalidValue;
  // B: the grid's y extent.  Pairs of heads that share keys and values take over where the
  // short kernel (two CTAs an SM) has more than a round (int8 cache, whose codes it widens
  // once a head) or three.  H 64 on 8, 128 tokens, short / pairs, us: int8 4 prompts 13.5 / 14.1,
  // 8 24.8 / 21.7, 32 93 / 69; bf16 8 13.2 / 15.1, 16 24.8 / 24.1, 32 49 / 39
  const bool kv8 = kv.kvquant == FP_KV_INT8, shared = n_heads / kv.n_kv_heads % 2 == 0;
  const bool one_tile = S <= kPaB && B <= 65535 && !(shared && (long long)B * n_heads > (kv8 ? 2 : 6) * pa_sms());
  if (kv8)
    return one_tile ? launch_attention_prefill_short(mq, mq, mq, B, S, n_heads, kv, out, err, s)
                    : launch_pa_tc<true>(mq, mq, mq, B, S, n_heads, kv, out, err, s);
  // bf16 pools [pages Hkv 16][128], box [16 rows][64]
  if (!make_tensor_map(&mk, kv.k_pool, pool_rows, kPaHD, 2, 16, 64, 128) ||
      !make_tensor_map(&mv, kv.v_pool, pool_rows, kPaHD, 2, 16, 64, 128))
    return cudaErrorInvalidValue;
  return one_tile ? launch_attention_prefill_short(mq, mk, mv, B, S, n_heads, kv, out, err, s)
                  : launch_pa_tc<false>(mq, mk, mv, B, S, n_heads, kv, out, err, s);
}

}  // namespace fpk
