// Prefill attention for prompts of at most 128 tokens (one key tile) on the
// tcgen05 tensor cores: paged cache of bf16 or int8 codes, head_dim 128.
//
// One CTA per (sequence, head), two per SM (256 TMEM columns and 97 KiB of shared
// memory each): with a single key tile there is nothing to pipeline inside a CTA,
// so two of them overlap instead.  Bound by latency, one chain of copy, product,
// softmax, product per CTA.  8 prompts of 128 tokens, 32 heads, bf16 / int8 cache:
// 7.7 / 13.2 us here, 12.4 / 20.6 on the persistent kernel of fp_attn_tc.cu (one CTA
// per SM).
//   warp 0      TMA: the Q tile (two 64-column boxes), then (bf16 cache) the K
//               rows and the V rows page by page, one box per lane;
//   warp 1      owns the TMEM, issues S = Q K^T, then O = P V;
//   warps 2-5   softmax, one query row per thread, over 32-column chunks: the row
//               maximum, then P = 2^(s - m) as 16-bit pairs over the scores
//               already read; then the output;
//   int8 cache: warps 0, 6 and 7 convert Q to fp16 in place, widen the codes to
//               fp16 exactly and stage the K scales and the V scales times
//               2^sigma, as in fp_attn_tc.cu.
// TMEM columns: scores [0, 128) with P over [0, 64), O [128, 256).  Every mbarrier
// wait is bounded (error 2 past the limit); a page id out of range reads zeros and
// sets error 1; a q beyond the fp16 range (int8 cache) sets status 3.
#include "attn_tc.cuh"
#include "common.cuh"

namespace fpk {

constexpr int kPsWiden = 3;                                           // warps 0, 6, 7
constexpr int kPsRows = (kPaB + 4 * kPsWiden - 1) / (4 * kPsWiden);   // tile rows per widening thread
constexpr int kPsSmem = 3 * kPaTile + 1024;                           // Q, K, V, alignment
constexpr int kPsCW = 32;                                             // score columns per TMEM load
constexpr uint32_t kPsO = 128;

template <bool KV8>
__global__ void __launch_bounds__(KV8 ? 256 : 192, 2)
    attn_prefill_short_kernel(const __grid_constant__ CUtensorMap map_q, const __grid_constant__ CUtensorMap map_k,
                              const __grid_constant__ CUtensorMap map_v, const int8_t* __restrict__ k8,
                              const int8_t* __restrict__ v8, const float* __restrict__ k_scale,
                              const float* __restrict__ v_scale, int S, int H, int Hkv, int page_size,
                              const int32_t* __restrict__ page_table, int pages_per_seq, int n_pages,
                              uint16_t* __restrict__ out, int32_t* err) {
  extern __shared__ __align__(1024) uint8_t smem_raw[];
  __shared__ uint64_t qfull, qconv, kfull, vfull, sfull, pfull, ofull, vmet;
  __shared__ float s_vmax[kPsWiden];  // int8: the widening warps' largest V scales
  __shared__ float s_unscale;          // int8: 2^-sigma, removed from the output
  __shared__ uint32_t tmem_base;
  __shared__ int abort_word;
  __shared__ __align__(16) float s_scl[KV8 ? 2 * kPaB : 4];  // int8: K, V scales of the keys
  volatile int* abort_flag = &abort_word;
  uint8_t* smem = (uint8_t*)(((uintptr_t)smem_raw + 1023) & ~(uintptr_t)1023);
  uint8_t* sQ = smem;
  uint8_t* sK = smem + kPaTile;
  uint8_t* sV = smem + 2 * kPaTile;
  const int warp = threadIdx.x >> 5, lane = threadIdx.x & 31;
  const int h = blockIdx.x, b = blockIdx.y, kvh = h / (H / Hkv);
  auto fail = [&]() {
    *abort_flag = 1;
    if (err) atomicExch(err, 2);
  };

  pdl_trigger();
  if (threadIdx.x == 0) {
    mbar_init(&qfull, 1);
    mbar_init(&qconv, kPsWiden);
    mbar_init(&kfull, KV8 ? kPsWiden : 1);
    mbar_init(&vfull, KV8 ? kPsWiden : 1);
    mbar_init(&sfull, 1);
    mbar_init(&pfull, 4);
    mbar_init(&ofull, 1);
    mbar_init(&vmet, kPsWiden);
    *abort_flag = 0;
    asm volatile("fence.mbarrier_init.release.cluster;" ::: "memory");
  }
  if (warp == 1) {
    asm volatile("tcgen05.alloc.cta_group::1.sync.aligned.shared::cta.b32 [%0], 256;" ::"r"(smem_u32(&tmem_base))
                 : "memory");
    asm volatile("tcgen05.relinquish_alloc_permit.cta_group::1.sync.aligned;" ::: "memory");
  }
  tc_fence_before();
  __syncthreads();
  tc_fence_after();
  const uint32_t tmem = tmem_base;
  pdl_wait();

  const int32_t* pt = page_table + (long long)b * pages_per_seq;
  if (warp == 0 || warp >= 6) {
    if (warp == 0 && lane == 0) {
      mbar_expect_tx(&qfull, kPaTile);
      tma_load_2d(sQ, &map_q, h * kPaHD, b * S, &qfull);
      tma_load_2d(sQ + kPaHalf, &map_q, h * kPaHD + 64, b * S, &qfull);
    }
    if constexpr (!KV8) {
      // ---------------- lanes 0-15 each copy one [16][64] box of K and of V
      // (page lane & 7, head_dim half lane >> 3)
      const int pg = lane & 7, half = (lane >> 3) & 1;
      int row = -16;  // pool row of this lane's page; -16 reads zeros
      if (lane < 16 && pg * 16 < S) {
        const int id = __ldg(pt + pg * 16 / page_size);
        if (id >= 0 && id < n_pages) row = (id * Hkv + kvh) * page_size;
        else if (err && half == 0) atomicExch(err, 1);
      }
      if (lane == 0) mbar_expect_tx(&kfull, kPaTile), mbar_expect_tx(&vfull, kPaTile);
      __syncwarp();
      if (lane < 16) {
        tma_load_2d(sK + half * kPaHalf + pg * 2048, &map_k, half * 64, row, &kfull);
        tma_load_2d(sV + half * kPaHalf + pg * 2048, &map_v, half * 64, row, &vfull);
      }
      if (lane == 0) {  // the copies land before the CTA leaves
        mbar_wait(&qfull, 0);
        mbar_wait(&kfull, 0);
        mbar_wait(&vfull, 0);
      }
    } else {
      // ---------------- int8 cache: widening
      const int wi = (warp == 0 ? 0 : warp - 5) * 32 + lane;  // 0 .. 95
      constexpr int WT = 32 * kPsWiden;
      const int c = wi & 7, rbase = wi >> 3;  // code chunk (head_dim 16c .. 16c + 15); tile rows rbase + 12i
      int rowi[kPsRows];                       // pool row of each of the thread's keys; -1 reads zeros
#pragma unroll
      for (int r = 0; r < kPsRows; ++r) {
        const int key = rbase + 4 * kPsWiden * r;
        rowi[r] = -1;
        if (key < S) {  // S <= 128
          const int pg = __ldg(pt + key / page_size);
          if (pg >= 0 && pg < n_pages) rowi[r] = (pg * Hkv + kvh) * page_size + key % page_size;
          else if (err && c == 0) atomicExch(err, 1);
        }
      }
      float vmax = 0.f;
#pragma unroll
      for (int r = 0; r < kPsRows; ++r)
        if (rowi[r] >= 0) vmax = fmaxf(vmax, __ldg(v_scale + rowi[r]));
      vmax = warp_max(vmax);
      if (lane == 0) {
        s_vmax[warp == 0 ? 0 : warp - 5] = vmax;
        mbar_arrive(&vmet);
      }
      bool ok = __all_sync(0xffffffffu, mbar_wait(&vmet, 0));
      vmax = fmaxf(fmaxf(s_vmax[0], s_vmax[1]), s_vmax[2]);
      // 2^sigma with 256 * vmax * 2^sigma <= 65280 (vmax = 0: no V weight at all)
      const int sigma = vmax > 0.f ? min(60, max(-60, (int)floorf(log2f(255.f / vmax)))) : 0;
      const float vmul = exp2f((float)sigma);
      // 16-bit form of chunk c: chunks cb, cb + 1 of half c / 4 of the swizzled
      // row; the lanes of the upper half store the odd chunk first, so the
      // eight lanes of one row write eight distinct 16-byte bank groups
      const int cb = 2 * (c & 3), half_off = (c >> 2) * kPaHalf;
      // the scales are read here, so that their loads are in flight together: read
      // row by row where they are stored, 47 prompts of 126 tokens, 32 heads take
      // 84.1 us instead of 69.4
      float sck[kPsRows], scv[kPsRows];
#pragma unroll
      for (int r = 0; r < kPsRows; ++r) {
        sck[r] = c == 0 && rowi[r] >= 0 ? __ldg(k_scale + rowi[r]) : 0.f;
        scv[r] = c == 0 && rowi[r] >= 0 ? __ldg(v_scale + rowi[r]) * vmul : 0.f;
      }
#pragma unroll 1
      for (int which = 0; which < 2; ++which) {
        const int8_t* pool = which ? v8 : k8;
        uint4 cw[kPsRows];
#pragma unroll
        for (int r = 0; r < kPsRows; ++r)
          cw[r] = rowi[r] >= 0 ? ld_nc16(pool + (long long)rowi[r] * kPaHD + c * 16) : make_uint4(0, 0, 0, 0);
        uint8_t* dst = (which ? sV : sK) + half_off;
#pragma unroll
        for (int r = 0; r < kPsRows; ++r) {
          const int row = rbase + 4 * kPsWiden * r, sw = row & 7;
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
          if (which == 0 && c == 0) {  // the scales go out with the K codes
            s_scl[row] = sck[r];
            s_scl[kPaB + row] = scv[r];
          }
        }
        if (which == 0 && wi == 0) s_unscale = exp2f((float)-sigma);
        fence_proxy_async();  // the MMAs read the tile through the async proxy
        __syncwarp();
        if (lane == 0) mbar_arrive(which ? &vfull : &kfull);
        if (which == 0) {  // Q to fp16 in place (the element order of the swizzled tile is kept)
          ok = ok && __all_sync(0xffffffffu, mbar_wait(&qfull, 0));
          bool over = false;
          for (int i = wi; ok && i < kPaTile / 16; i += WT) {
            uint4* p = reinterpret_cast<uint4*>(sQ) + i;
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
          fence_proxy_async();
          __syncwarp();
          if (lane == 0) mbar_arrive(&qconv);
        }
      }
      if (!ok && lane == 0) fail();
    }
  } else if (warp == 1) {
    // ---------------- MMA issuer.  int8 cache: fp16 operands (A and B of one
    // MMA always share their type), bf16 cache: bf16
    constexpr uint32_t f16 = KV8 ? ((1u << 7) | (1u << 10)) : 0u;
    constexpr uint32_t idesc_s = tc_idesc(kPaB, kPaB) & ~f16;
    constexpr uint32_t idesc_o = (tc_idesc(kPaB, kPaHD) | (1u << 16)) & ~f16;
    const uint64_t qd = sdesc(smem_u32(sQ)), kd = sdesc(smem_u32(sK)), vd = sdesc_mn(smem_u32(sV), kPaHalf);
    bool ok = mbar_wait(KV8 ? &qconv : &qfull, 0) && mbar_wait(&kfull, 0);
    ok = __all_sync(0xffffffffu, ok);
    if (ok) {
      tc_fence_after();
      if (elect_one()) {
#pragma unroll
        for (int kk = 0; kk < kPaHD / 16; ++kk) {  // descriptor start addresses count 16-byte units
          const int off = ((kk >> 2) * kPaHalf + (kk & 3) * 32) >> 4;
          tc_mma(tmem, qd + off, kd + off, idesc_s, kk > 0 ? 1u : 0u);
        }
        tc_commit(&sfull);
      }
      __syncwarp();
      ok = __all_sync(0xffffffffu, mbar_wait(&vfull, 0) && mbar_wait(&pfull, 0));
    }
    if (ok) {
      tc_fence_after();
      if (elect_one()) {
#pragma unroll
        for (int kk = 0; kk < kPaB / 16; ++kk)  // 16 keys: two 8-row groups of the V tile
          tc_mma_ts(tmem + kPsO, tmem + kk * 8, vd + kk * (2048 >> 4), idesc_o, kk > 0 ? 1u : 0u);
      }
      __syncwarp();
    } else if (lane == 0) {
      fail();
    }
    if (elect_one()) tc_commit(&ofull);  // every MMA issued has completed before TMEM is released
    __syncwarp();
    mbar_wait(&ofull, 0);
  } else {
    // ---------------- softmax: thread = query row (TMEM lane 32 (warp % 4) + lane)
    const int quad = warp & 3, row = quad * 32 + lane;
    const uint32_t lane_base = tmem + ((uint32_t)(quad * 32) << 16);
    const float scale = kPaLog2e * rsqrtf((float)kPaHD);
    bool ok = __all_sync(0xffffffffu, mbar_wait(&sfull, 0));
    float l = 1.f;
    if (ok) {
      tc_fence_after();
      // scores of chunk c; keys after this row (and so past S) read -inf
      auto load = [&](int c, float* v) {
        tc_ld<kPsCW>(lane_base + c * kPsCW, reinterpret_cast<uint32_t*>(v));
        if constexpr (KV8) {
          const float4* k4 = reinterpret_cast<const float4*>(s_scl + c * kPsCW);
#pragma unroll
          for (int i = 0; i < kPsCW / 4; ++i) {
            const float4 f = k4[i];
            v[4 * i] *= f.x, v[4 * i + 1] *= f.y, v[4 * i + 2] *= f.z, v[4 * i + 3] *= f.w;
          }
        }
#pragma unroll
        for (int i = 0; i < kPsCW; ++i)
          if (c * kPsCW + i > row) v[i] = -INFINITY;
      };
      float m4[4] = {-INFINITY, -INFINITY, -INFINITY, -INFINITY};
#pragma unroll 1
      for (int c = 0; c < kPaB / kPsCW; ++c) {
        float v[kPsCW];
        load(c, v);
#pragma unroll
        for (int i = 0; i < kPsCW; ++i) m4[i & 3] = fmaxf(m4[i & 3], v[i]);
      }
      const float m = fmaxf(fmaxf(m4[0], m4[1]), fmaxf(m4[2], m4[3])) * scale;
      const float mref = m == -INFINITY ? 0.f : m;
      float p4[4] = {0.f, 0.f, 0.f, 0.f};
#pragma unroll 1
      for (int c = 0; c < kPaB / kPsCW; ++c) {
        float v[kPsCW];
        load(c, v);
        uint32_t pw[kPsCW / 2];
#pragma unroll
        for (int i = 0; i < kPsCW; i += 2) {
          const float p0 = pa_ex2(fmaf(v[i], scale, -mref)), p1 = pa_ex2(fmaf(v[i + 1], scale, -mref));
          p4[i & 3] += p0;
          p4[(i + 1) & 3] += p1;
          if constexpr (KV8) {
            // V scale of each key column: P V then takes the codes as they are
            const float2 vs = *reinterpret_cast<const float2*>(s_scl + kPaB + c * kPsCW + i);
            pw[i / 2] = pa_pack_h(p0 * vs.x, p1 * vs.y);
          } else {
            pw[i / 2] = pa_pack(p0, p1);
          }
        }
        tc_st16(lane_base + c * (kPsCW / 2), pw);
      }
      l = (p4[0] + p4[1]) + (p4[2] + p4[3]);
      tc_wait_st();
      tc_fence_before();
      __syncwarp();
      if (lane == 0) mbar_arrive(&pfull);
      ok = __all_sync(0xffffffffu, mbar_wait(&ofull, 0)) && !*abort_flag;
      ok = __all_sync(0xffffffffu, ok);
    }
    if (ok) {
      tc_fence_after();
      // int8 cache: P carried the V scales times 2^sigma.  Q has been read: its
      // tile serves as the staging buffer
      const float inv = (KV8 ? s_unscale : 1.f) / l;
      const int pos = quad * 32;
      pa_write_rows<kPaHD>([&](int x, float* r) { pa_load_out(lane_base + kPsO + x, inv, r); }, 0, sQ + quad * kPaStage,
                           out + ((long long)b * S + pos) * ((long long)H * kPaHD) + (long long)h * kPaHD,
                           (long long)H * kPaHD, pos, S);
    } else if (lane == 0) {
      fail();
    }
  }
  tc_fence_before();
  __syncthreads();
  if (warp == 1) {
    tc_fence_after();
    asm volatile("tcgen05.dealloc.cta_group::1.sync.aligned.b32 %0, 256;" ::"r"(tmem) : "memory");
  }
}

template <bool KV8>
static cudaError_t launch_short_t(const CUtensorMap& mq, const CUtensorMap& mk, const CUtensorMap& mv, int B, int S,
                                  int n_heads, const fp_kv_view& kv, uint16_t* out, int32_t* err, cudaStream_t s) {
  static std::atomic<unsigned long long> attr{0};
  FP_CUDA_TRY(smem_limit_once(attn_prefill_short_kernel<KV8>, kPsSmem, &attr));
  return launch(attn_prefill_short_kernel<KV8>, dim3(n_heads, B), dim3(KV8 ? 256 : 192), (size_t)kPsSmem, s, mq, mk, mv,
                (const int8_t*)kv.k_pool, (const int8_t*)kv.v_pool, (const float*)kv.k_scale,
                (const float*)kv.v_scale, S, n_heads, kv.n_kv_heads, kv.page_size, kv.page_table, kv.pages_per_seq,
                kv.n_pages, out, err);
}

cudaError_t launch_attention_prefill_short(const CUtensorMap& mq, const CUtensorMap& mk, const CUtensorMap& mv, int B,
                                           int S, int n_heads, const fp_kv_view& kv, uint16_t* out, int32_t* err,
                                           cudaStream_t s) {
  return kv.kvquant == FP_KV_INT8 ? launch_short_t<true>(mq, mk, mv, B, S, n_heads, kv, out, err, s)
                                  : launch_short_t<false>(mq, mk, mv, B, S, n_heads, kv, out, err, s);
}

}  // namespace fpk
