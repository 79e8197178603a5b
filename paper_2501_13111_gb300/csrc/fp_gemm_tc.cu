// Prefill weight-only linear on the 5th-generation tensor cores.
//
// y[M][N] = x[M][K] W[N][K]^T for M > 64 (prefill), the dense contraction of
// the block's linear layers.  Persistent: a pair of CTAs (on two SMs) walks
// 256 x 256 output tiles, each over the whole K, or, where that needs more rounds,
// one CTA 128 x 256 tiles:
//   warp 0      TMA producer: x tile [128][64] and W tile [256][64] (bf16,
//               128-byte swizzled, K-major; half of the W tile in each CTA of a
//               pair) into a 4-stage (6-stage) shared ring, completion counted
//               in bytes on mbarrier full[s] (of the even CTA);
//   warp 1      allocates 512 TMEM columns (two fp32 accumulators) and, from
//               one thread, issues tcgen05.mma (M 128, N 256, K 16);
//               tcgen05.commit frees each stage (empty[s]) and signals a full
//               accumulator (tfull[b]);
//   warps 2-5   epilogue: tcgen05.ld of the accumulator (one TMEM lane per
//               output row), per-column int8 scale, residual add / SwiGLU /
//               fp32 store; then the buffer goes back to the MMA thread
//               (tempty[b]) while the next tile accumulates in the other.
// Quantised weights are first expanded to bf16 into a scratch matrix by
// dequant_kernel (int8: the code itself, exact, with its row scale applied
// in the epilogue; int4: bf16((q - z) * s)).
//
// Every mbarrier wait is bounded: past the limit the thread records an error
// in the error word, the CTA stops issuing work and falls through to the TMEM
// release, so a fault in the pipeline surfaces as a status, not a hang.
#include <cuda.h>

#include <algorithm>

#include "common.cuh"
#include "kernels.cuh"
#include "tc.cuh"

// Rounds after which the MMA thread's wait for a stage gives up: kTcSpinLimit,
// unless a test lowers it through fp_debug_set_wait_limit to run the failure
// path (every other wait keeps kTcSpinLimit, so copies and MMAs in flight are
// still drained before the CTA leaves).
static __device__ long long g_stage_wait_limit = fpk::kTcSpinLimit;

namespace fpk {

constexpr int kTcBM = 128, kTcBN = 256, kTcBK = 64;
constexpr int kTcThreads = 192;
// Shared memory of a stage and the ring's depth, one CTA / each CTA of a pair
// (which holds its own 128 rows of x and half of the 256 weight rows).
template <bool PAIR>
struct TcGeom {
  static constexpr int kBRows = PAIR ? kTcBN / 2 : kTcBN;
  static constexpr uint32_t kStageBytes = (kTcBM + kBRows) * kTcBK * 2;  // 48 / 32 KiB
  static constexpr int kStages = PAIR ? 6 : 4;
  static constexpr int kSmem = kStages * kStageBytes + 1024;
};
constexpr uint32_t kTcTmemCols = 512;  // two 256-column fp32 accumulators

// ------------------------------------------------------------------ kernel
// Persistent: CTA c takes output tiles c, c + gridDim.x, ... in grouped
// order (16 M tiles share each sweep over the N tiles, so a wave's x rows
// and weight columns stay in L2).  The shared ring runs across tiles, and
// the fp32 accumulator is double-buffered in TMEM (2 x 256 columns): the MMA
// thread fills one buffer while the epilogue warps drain the other.
// SCALE: multiply output column n by bf16 scales[n] (int8 weights; SwiGLU:
// the up column by scales[up_off + n]).  Output (and residual) rows are ldy
// elements apart, so a launch can fill a band of columns of a wider output.
// PAIR: clusters of two CTAs on a 256 x 256 tile (cta_group::2): CTA r of a pair
// keeps rows 128 r .. of x and of the output, and loads half of the weight rows,
// which both read; the even CTA issues the MMAs.
template <int EPI, bool SCALE, bool PAIR>
__global__ void __launch_bounds__(kTcThreads, 1)
    gemm_tc_kernel(const __grid_constant__ CUtensorMap map_x, const __grid_constant__ CUtensorMap map_w, int M, int N,
                   int K, const uint16_t* __restrict__ scales, long long up_off, const uint16_t* R, void* Y,
                   int ldy, int32_t* err) {
  using G = TcGeom<PAIR>;
  constexpr int ST = G::kStages, CG = PAIR ? 2 : 1;
  extern __shared__ __align__(1024) uint8_t smem_raw[];
  __shared__ uint64_t full[ST], empty[ST], tfull[2], tempty[2], mma_done, never;
  __shared__ uint32_t tmem_base;
  __shared__ int abort_word;
  volatile int* abort_flag = &abort_word;  // set by a role that gave up waiting
  // stage buffers must be 1024-byte aligned for the 128-byte swizzle
  uint8_t* smem = (uint8_t*)(((uintptr_t)smem_raw + 1023) & ~(uintptr_t)1023);
  const int warp = threadIdx.x >> 5, lane = threadIdx.x & 31;
  const int rank = PAIR ? (int)cluster_rank() : 0;
  constexpr int NR = EPI == FP_EPI_SWIGLU ? 2 : 1;
  const int Nout = NR == 2 ? N / 2 : N;
  constexpr int BNout = kTcBN / NR;
  const int tiles_m = (M + CG * kTcBM - 1) / (CG * kTcBM), tiles_n = (Nout + BNout - 1) / BNout;
  const int ntiles = tiles_m * tiles_n;
  const int kblocks = (K + kTcBK - 1) / kTcBK;
  // (the tile loops read the grid's registers themselves: through variables the single
  // CTA's instance took 2.5 % longer, 4096^3 111.6 us against 109.4, the pairs' 2.3 %)
  auto tile_origin = [&](int t, int& m0, int& n0) {
    constexpr int GM = 16 / CG;
    const int span = GM * tiles_n;
    const int first = (t / span) * GM;
    const int gs = min(GM, tiles_m - first);
    const int r = t % span;
    m0 = (first + r % gs) * (CG * kTcBM) + rank * kTcBM;
    n0 = (r / gs) * BNout;
  };
  auto fail = [&]() {
    if constexpr (PAIR) {  // both CTAs stop
      for (uint32_t r = 0; r < 2; ++r)
        asm volatile("st.shared::cluster.u32 [%0], %1;" ::"r"(cluster_addr(&abort_word, r)), "r"(1) : "memory");
    } else {
      *abort_flag = 1;
    }
    if (err) atomicExch(err, 2);
  };

  pdl_trigger();
  if (threadIdx.x == 0) {
    for (int s = 0; s < ST; ++s) {
      mbar_init(&full[s], 1);
      mbar_init(&empty[s], 1);
    }
    for (int b = 0; b < 2; ++b) {
      mbar_init(&tfull[b], 1);        // tcgen05.commit of the tile's last MMAs
      mbar_init(&tempty[b], 4 * CG);  // one arrival per epilogue warp (of both CTAs)
    }
    mbar_init(&mma_done, 1);
    mbar_init(&never, 1);
    *abort_flag = 0;
    asm volatile("fence.mbarrier_init.release.cluster;" ::: "memory");
  }
  if constexpr (PAIR) cluster_sync();  // the peer's barriers are up before anything signals them
  if (warp == 1) {
    if constexpr (PAIR) {
      asm volatile("tcgen05.alloc.cta_group::2.sync.aligned.shared::cta.b32 [%0], %1;" ::"r"(smem_u32(&tmem_base)),
                   "r"(kTcTmemCols)
                   : "memory");
      asm volatile("tcgen05.relinquish_alloc_permit.cta_group::2.sync.aligned;" ::: "memory");
    } else {
      asm volatile("tcgen05.alloc.cta_group::1.sync.aligned.shared::cta.b32 [%0], %1;" ::"r"(smem_u32(&tmem_base)),
                   "r"(kTcTmemCols)
                   : "memory");
      asm volatile("tcgen05.relinquish_alloc_permit.cta_group::1.sync.aligned;" ::: "memory");
    }
  }
  tc_fence_before();
  __syncthreads();
  if constexpr (PAIR) cluster_sync();  // both tensor memories are allocated
  tc_fence_after();
  const uint32_t tmem = tmem_base;
  pdl_wait();

  if (warp == 0) {
    // ---------------- TMA producer
    if (lane == 0) {
      int it = 0;  // k-blocks issued, across tiles
      for (int t = blockIdx.x / CG; t < ntiles && !*abort_flag; t += gridDim.x / CG) {
        int m0, n0;
        tile_origin(t, m0, n0);
        for (int kb = 0; kb < kblocks; ++kb, ++it) {
          const int s = it % ST;
          if (!mbar_wait(&empty[s], ((it / ST) & 1) ^ 1) || *abort_flag) {
            fail();
            break;
          }
          uint8_t* a = smem + s * G::kStageBytes;
          uint8_t* b = a + kTcBM * kTcBK * 2;
          if constexpr (PAIR) {
            // the bytes of both CTAs count on the even CTA's barrier
            if (rank == 0) mbar_expect_tx(&full[s], 2 * G::kStageBytes);
            const uint32_t bar = cluster_addr(&full[s], 0);
            const int wrow = NR == 2 ? (rank ? Nout + n0 : n0) : n0 + rank * G::kBRows;  // SwiGLU: gate rows | up rows
            tma_load_2d_pair(a, &map_x, kb * kTcBK, m0, bar);
            tma_load_2d_pair(b, &map_w, kb * kTcBK, wrow, bar);
          } else {
            mbar_expect_tx(&full[s], G::kStageBytes);
            tma_load_2d(a, &map_x, kb * kTcBK, m0, &full[s]);
            tma_load_2d(b, &map_w, kb * kTcBK, n0, &full[s]);  // SwiGLU: gate rows
            if (NR == 2) tma_load_2d(b + 128 * kTcBK * 2, &map_w, kb * kTcBK, Nout + n0, &full[s]);  // up rows
          }
        }
      }
      // copies still in flight land before the CTA leaves (their stages are its
      // shared memory); a pair leaves together, after the even CTA has seen both's.
      // After an abort the two may have issued different numbers of copies: a
      // bounded wait for what never comes outlasts them
      if (rank == 0)
        for (int j = max(0, it - ST); j < it; ++j) mbar_wait(&full[j % ST], (j / ST) & 1);
      if (PAIR && *abort_flag) mbar_wait(&never, 0);
    }
  } else if (warp == 1) {
    // ---------------- MMA issuer
    if (lane == 0 && rank == 0) {
      constexpr uint32_t idesc = tc_idesc(CG * kTcBM, kTcBN);
      const long long stage_limit = g_stage_wait_limit;
      auto commit = [&](uint64_t* bar) {
        if constexpr (PAIR) tc_commit_pair(bar);
        else tc_commit(bar);
      };
      int it = 0, lt = 0;
      for (int t = blockIdx.x / CG; t < ntiles && !*abort_flag; t += gridDim.x / CG, ++lt) {
        const int acc = lt & 1;
        // the epilogue has drained this accumulator (local tile lt - 2)
        if (!mbar_wait(&tempty[acc], ((lt >> 1) & 1) ^ 1) || *abort_flag) {
          fail();
          break;
        }
        tc_fence_after();
        const uint32_t d = tmem + (uint32_t)acc * kTcBN;
        bool ok = true;
        for (int kb = 0; kb < kblocks; ++kb, ++it) {
          const int s = it % ST;
          if (!mbar_wait_n(&full[s], (it / ST) & 1, stage_limit) || *abort_flag) {
            ok = false;
            break;
          }
          tc_fence_after();
          const uint32_t a = smem_u32(smem + s * G::kStageBytes);
          const uint32_t b = a + kTcBM * kTcBK * 2;
#pragma unroll
          for (int kk = 0; kk < kTcBK / 16; ++kk) {
            if constexpr (PAIR) tc_mma_pair(d, sdesc(a + kk * 32), sdesc(b + kk * 32), idesc, (kb > 0 || kk > 0) ? 1u : 0u);
            else tc_mma(d, sdesc(a + kk * 32), sdesc(b + kk * 32), idesc, (kb > 0 || kk > 0) ? 1u : 0u);
          }
          commit(&empty[s]);  // stage s is free once these MMAs have read it
        }
        if (!ok) {
          fail();
          break;
        }
        commit(&tfull[acc]);  // the tile's accumulator is complete
      }
      // every MMA issued has completed before TMEM is released
      commit(&mma_done);
      mbar_wait(&mma_done, 0);
    }
  } else {
    // ---------------- epilogue: warp w reads TMEM lanes 32 (w % 4) .. +31
    const int q = warp & 3;
    int lt = 0;
    for (int t = blockIdx.x / CG; t < ntiles; t += gridDim.x / CG, ++lt) {
      const int acc = lt & 1;
      int m0, n0;
      tile_origin(t, m0, n0);
      const bool ok = mbar_wait(&tfull[acc], (lt >> 1) & 1);
      if (!ok || *abort_flag) {
        fail();
        break;
      }
      tc_fence_after();
      const int row = m0 + q * 32 + lane;
      const uint32_t tl = tmem + (uint32_t)acc * kTcBN + ((uint32_t)(q * 32) << 16);
#pragma unroll 1
      for (int c0 = 0; c0 < BNout; c0 += 32) {
        float v[32], u[32];
        tc_ld32(tl + c0, v);
        if (NR == 2) tc_ld32(tl + 128 + c0, u);
        if (row >= M) continue;
        const int n = n0 + c0;
        if (n >= Nout) continue;
        const int cnt = min(32, Nout - n);
        if constexpr (SCALE) {
#pragma unroll
          for (int i = 0; i < 32; ++i) {
            if (i < cnt) {
              v[i] *= bf2f(scales[n + i]);
              if (NR == 2) u[i] *= bf2f(scales[up_off + n + i]);
            }
          }
        }
        const long long o = (long long)row * ldy + n;
        if constexpr (EPI == FP_EPI_F32) {
          float* y = (float*)Y + o;
          if (cnt == 32 && (o & 3) == 0) {
#pragma unroll
            for (int i = 0; i < 32; i += 4) *reinterpret_cast<float4*>(y + i) = make_float4(v[i], v[i + 1], v[i + 2], v[i + 3]);
          } else {
            for (int i = 0; i < cnt; ++i) y[i] = v[i];
          }
        } else {
          uint16_t* y = (uint16_t*)Y + o;
          float r[32];
#pragma unroll
          for (int i = 0; i < 32; ++i) {
            if constexpr (EPI == FP_EPI_SWIGLU) r[i] = silu(v[i]) * u[i];
            else r[i] = v[i];
          }
          if constexpr (EPI == FP_EPI_RESID) {
            const uint16_t* rr = R + o;
            for (int i = 0; i < cnt; ++i) r[i] += bf2f(rr[i]);
          }
          if (cnt == 32 && (o & 7) == 0) {
#pragma unroll
            for (int i = 0; i < 32; i += 8)
              *reinterpret_cast<uint4*>(y + i) = make_uint4(pack_bf2(r[i], r[i + 1]), pack_bf2(r[i + 2], r[i + 3]),
                                                            pack_bf2(r[i + 4], r[i + 5]), pack_bf2(r[i + 6], r[i + 7]));
          } else {
            for (int i = 0; i < cnt; ++i) y[i] = f2bf(r[i]);
          }
        }
      }
      // this warp's reads of the accumulator are done: hand the buffer back to the MMA thread
      tc_fence_before();
      __syncwarp();
      if (lane == 0) {
        if constexpr (PAIR) mbar_arrive_cluster(cluster_addr(&tempty[acc], 0));
        else mbar_arrive(&tempty[acc]);
      }
    }
  }
  tc_fence_before();
  __syncthreads();
  if constexpr (PAIR) cluster_sync();  // neither CTA leaves while the other's MMAs, copies or arrivals may touch it
  if (warp == 1) {
    tc_fence_after();
    if constexpr (PAIR)
      asm volatile("tcgen05.dealloc.cta_group::2.sync.aligned.b32 %0, %1;" ::"r"(tmem), "r"(kTcTmemCols) : "memory");
    else
      asm volatile("tcgen05.dealloc.cta_group::1.sync.aligned.b32 %0, %1;" ::"r"(tmem), "r"(kTcTmemCols) : "memory");
  }
}

// ------------------------------------------------------------------ dequant to bf16
// int8: w = q (exact; the row scale is applied by the GEMM epilogue).
// int4: w = bf16((q - z) * s), 8 elements (one packed word) at a time.
// GPTQ4: the same expansion back into channel order: output channel k is
// act-order column j = inv[k] (inv the inverse of the act order), with the
// scale and zero of group j / 128; 8 consecutive channels at a time.
// Output row r is row r0 + r of the matrix for r < cols, row up0 + r - cols
// after (SwiGLU: the band's gate rows, then its up rows).  A thread takes four
// words its row's threads apart, so that its loads are in flight together and
// every access of a warp is contiguous (one word a thread at a time, its row found
// by a division, took 35 us more on 22016 x 4096 int4).  Rows of up to 2048
// elements share a block: a block for each left most of its threads idle (whole linears:
// int4 26288 x 256 at 88 rows 35.1 us, 12.1 so; int8 16304 x 768 at 154 35.2, 23.2).  Bound by memory, the
// codes read and the bf16 written.  Running the expansion of one band beside the
// GEMM of the band before, in more and smaller bands, lost more to the GEMMs'
// starts and last rounds than it hid (22016 x 4096 int8, 4096 rows: 518-548 us
// against 507).
constexpr int kDqThreads = 128, kDqWords = 4;

template <int WQ>
__global__ void __launch_bounds__(kDqThreads)
    dequant_kernel(const void* __restrict__ codes, const uint16_t* __restrict__ scales,
                   const uint16_t* __restrict__ zeros, long long r0, long long up0, int cols, int rows, int K,
                   uint16_t* __restrict__ out, const int32_t* __restrict__ inv) {
  pdl_trigger();
  pdl_wait();
  const int tx = blockDim.x;
  for (int r = blockIdx.y * blockDim.y + threadIdx.y; r < rows; r += gridDim.y * blockDim.y) {
    const long long row = r < cols ? r0 + r : up0 + (r - cols);
    const int w0 = blockIdx.x * (tx * kDqWords) + threadIdx.x, words = K / 8;
    uint16_t* o = out + (long long)r * K;
    if constexpr (WQ == FP_W_GPTQ4) {
      const uint32_t* cw = (const uint32_t*)codes + row * words;
      const uint16_t *sr = scales + row * (K / 128), *zr = zeros + row * (K / 128);
      for (int i = 0; i < kDqWords; ++i) {
        const int w = w0 + i * tx;
        if (w >= words) break;
        float f[8];
#pragma unroll
        for (int j = 0; j < 8; ++j) {
          const int a = min(max(inv[w * 8 + j], 0), K - 1);  // the inverse comes from the act order, in range
          const int e = a & 7, nib = (e >> 1) + 4 * (e & 1);  // element e of a word sits in this nibble
          const float q = (float)((cw[a >> 3] >> (4 * nib)) & 0xF);
          f[j] = (q - bf2f(zr[a >> 7])) * bf2f(sr[a >> 7]);
        }
        *reinterpret_cast<uint4*>(o + (long long)w * 8) =
            make_uint4(pack_bf2(f[0], f[1]), pack_bf2(f[2], f[3]), pack_bf2(f[4], f[5]), pack_bf2(f[6], f[7]));
      }
    } else if constexpr (WQ == FP_W_INT8) {
      const uint2* cr = (const uint2*)codes + row * words;
      uint2 c[kDqWords];
#pragma unroll
      for (int i = 0; i < kDqWords; ++i)
        c[i] = w0 + i * tx < words ? __ldg(cr + w0 + i * tx) : make_uint2(0u, 0u);
#pragma unroll
      for (int i = 0; i < kDqWords; ++i) {
        const uint32_t w[2] = {c[i].x, c[i].y};
        float f[8];
#pragma unroll
        for (int j = 0; j < 8; ++j) f[j] = (float)(int8_t)((w[j >> 2] >> (8 * (j & 3))) & 0xFF);
        if (w0 + i * tx < words)
          *reinterpret_cast<uint4*>(o + (long long)(w0 + i * tx) * 8) =
              make_uint4(pack_bf2(f[0], f[1]), pack_bf2(f[2], f[3]), pack_bf2(f[4], f[5]), pack_bf2(f[6], f[7]));
      }
    } else {
      const uint32_t* cr = (const uint32_t*)codes + row * words;
      const uint16_t *sr = scales + row * (K / 128), *zr = zeros + row * (K / 128);
      uint32_t c[kDqWords];
      float s[kDqWords], z[kDqWords];
#pragma unroll
      for (int i = 0; i < kDqWords; ++i) {
        const int w = w0 + i * tx;
        const bool in = w < words;
        c[i] = in ? __ldg(cr + w) : 0u;
        s[i] = in ? bf2f(__ldg(sr + w / 16)) : 0.f;  // 16 words per group
        z[i] = in ? bf2f(__ldg(zr + w / 16)) : 0.f;
      }
#pragma unroll
      for (int i = 0; i < kDqWords; ++i) {
        float f[8];
        // nibbles i and i + 4 hold elements 2i and 2i + 1
#pragma unroll
        for (int j = 0; j < 4; ++j) {
          f[2 * j] = ((float)((c[i] >> (4 * j)) & 0xF) - z[i]) * s[i];
          f[2 * j + 1] = ((float)((c[i] >> (4 * j + 16)) & 0xF) - z[i]) * s[i];
        }
        if (w0 + i * tx < words)
          *reinterpret_cast<uint4*>(o + (long long)(w0 + i * tx) * 8) =
              make_uint4(pack_bf2(f[0], f[1]), pack_bf2(f[2], f[3]), pack_bf2(f[4], f[5]), pack_bf2(f[6], f[7]));
      }
    }
  }
}

// ------------------------------------------------------------------ host side
typedef CUresult (*EncodeTiledFn)(CUtensorMap*, CUtensorMapDataType, cuuint32_t, void*, const cuuint64_t*,
                                  const cuuint64_t*, const cuuint32_t*, const cuuint32_t*, CUtensorMapInterleave,
                                  CUtensorMapSwizzle, CUtensorMapL2promotion, CUtensorMapFloatOOBfill);

static EncodeTiledFn encode_fn() {
  static EncodeTiledFn fn = nullptr;
  if (!fn) {
    cudaDriverEntryPointQueryResult q;
    void* p = nullptr;
    if (cudaGetDriverEntryPoint("cuTensorMapEncodeTiled", &p, cudaEnableDefault, &q) == cudaSuccess &&
        q == cudaDriverEntryPointSuccess)
      fn = (EncodeTiledFn)p;
  }
  return fn;
}

bool make_tensor_map(CUtensorMap* map, const void* base, long long rows, long long cols, int elem_bytes,
                     int box_rows, int box_cols, int swizzle_bytes) {
  EncodeTiledFn fn = encode_fn();
  if (!fn || (elem_bytes != 1 && elem_bytes != 2 && elem_bytes != 4) || (swizzle_bytes != 64 && swizzle_bytes != 128))
    return false;
  cuuint64_t dims[2] = {(cuuint64_t)cols, (cuuint64_t)rows};
  cuuint64_t strides[1] = {(cuuint64_t)cols * elem_bytes};
  cuuint32_t box[2] = {(cuuint32_t)box_cols, (cuuint32_t)box_rows};
  cuuint32_t estr[2] = {1, 1};
  const CUtensorMapDataType dt = elem_bytes == 4   ? CU_TENSOR_MAP_DATA_TYPE_UINT32
                                 : elem_bytes == 2 ? CU_TENSOR_MAP_DATA_TYPE_BFLOAT16
                                                   : CU_TENSOR_MAP_DATA_TYPE_UINT8;
  return fn(map, dt, 2,
            const_cast<void*>(base), dims, strides, box, estr, CU_TENSOR_MAP_INTERLEAVE_NONE,
            swizzle_bytes == 128 ? CU_TENSOR_MAP_SWIZZLE_128B : CU_TENSOR_MAP_SWIZZLE_64B,
            CU_TENSOR_MAP_L2_PROMOTION_L2_256B, CU_TENSOR_MAP_FLOAT_OOB_FILL_NONE) == CUDA_SUCCESS;
}

bool tensor_maps_available() { return encode_fn() != nullptr; }

// bf16 [rows][cols] row-major, box [box_rows][64] with 128-byte swizzle.
static bool make_map(CUtensorMap* map, const void* base, long long rows, long long cols, int box_rows) {
  return make_tensor_map(map, base, rows, cols, 2, box_rows, kTcBK, 128);
}

// Quantised weights are expanded to bf16 band by band of output columns, so
// the scratch holds at most kTcScratchBytes (or one band of 256 columns).
constexpr size_t kTcScratchBytes = 128u << 20;

// Output columns per band: a multiple of the tile's (256, SwiGLU 128), all of them if they fit.
static int band_cols(int epi, int N, int K) {
  const int nr = epi == FP_EPI_SWIGLU ? 2 : 1;
  const int nout = nr == 2 ? N / 2 : N;
  const int unit = kTcBN / nr;
  const long long fit = (long long)(kTcScratchBytes / ((size_t)nr * K * 2)) / unit * unit;
  return (int)std::min<long long>(nout, std::max<long long>(unit, fit));
}

size_t gemm_tc_ws_bytes(int wquant, int N, int K) {
  if (wquant == FP_W_BF16) return 0;
  // the largest band over the epilogues (a SwiGLU band holds its gate and its up rows)
  const size_t plain = (size_t)band_cols(FP_EPI_STORE, N, K) * K * 2;
  const size_t swiglu = N % 2 == 0 ? (size_t)2 * band_cols(FP_EPI_SWIGLU, N, K) * K * 2 : 0;
  return std::max(plain, swiglu);
}

bool gemm_tc_ok(int M, int N, int K) { return M > 64 && K % 8 == 0 && N >= 1 && encode_fn() != nullptr; }

static int tc_sms() {
  static int sms = 0;
  if (!sms) {
    int dev = 0;
    if (cudaGetDevice(&dev) != cudaSuccess || cudaDeviceGetAttribute(&sms, cudaDevAttrMultiProcessorCount, dev) != cudaSuccess ||
        sms <= 0)
      sms = 152;
  }
  return sms;
}

static long long tc_tiles(int epi, int M, int N, int cg) {
  const int nout = epi == FP_EPI_SWIGLU ? N / 2 : N, bn = kTcBN / (epi == FP_EPI_SWIGLU ? 2 : 1);
  return (long long)((nout + bn - 1) / bn) * ((M + cg * kTcBM - 1) / (cg * kTcBM));
}

// A pair works through its 256 x 256 tile in 0.93 of the time that a CTA takes for
// its 128 x 256 (8192^3: 653 against 700 us; half of the weight rows' copies and
// reads leave shared memory, whose bandwidth bounds the single CTA), so it is taken
// unless its coarser tiles cost more rounds than that saves.  Starting and ending a
// pair's tile takes about 0.8 us longer, which a short K does not bring back.  In a
// single round shared memory is not the bound: there a pair gains, by reading the
// weights once for two row tiles, where they come from memory, as a forward pass's
// bf16 weights of some size do, and loses where they lie in L2, as a small expansion
// does and the weights of a small model.  Rows that a pair computes beyond M cost
// nothing then.  One CTA a tile / pairs, us (weights from memory but where said; one
// round: alike from 65 to 512 rows):
//   bf16, M 300       4096 x 1024 13.8 / 14.6   2048 20.2 / 20.2   3072 26.2 / 25.5   4096 32.3 / 31.0   8192 56.1 / 52.5
//                     1024 x 4096 31.1 / 30.6   8192 54.9 / 51.9
//     in L2           4096 x 1024 12.8 / 14.1   4096 28.9 / 30.3   11008 72.5 / 67.0
//                     1024 x 4096 28.6 / 30.0   8192 49.8 / 51.2
//   int4 expanded     4096 x 4096 36.8 / 37.5   8192 x 4096 45.4 / 45.0   4096 x 8192 67.5 / 64.9
//   bf16, 2048 x 8192 K 512 33.6 / 34.1   768 37.3 / 37.4   1024 43.0 / 40.5   2048 66.0 / 60.9
//     with SwiGLU     K 1024 44.6 / 46.6   1536 51.2 / 50.9   2048 62.9 / 59.2
// So in one round from 2^24 bf16 weights (a quarter of L2; a matrix of 4096 x 4096 that a
// loop leaves there loses 1.4 us) and from 2^25 expanded ones.
static bool tc_pair(int wquant, int epi, int M, int N, int K) {
  const long long sms = tc_sms();
  const long long r1 = (tc_tiles(epi, M, N, 1) + sms - 1) / sms, r2 = (tc_tiles(epi, M, N, 2) + sms / 2 - 1) / (sms / 2);
  if (r2 * 93 > r1 * 100) return false;
  if (r1 == 1) return K >= 3072 && (long long)N * K >= (wquant == FP_W_BF16 ? 1LL << 24 : 1LL << 25);
  return K >= (epi == FP_EPI_SWIGLU ? 1536 : 1024);
}

template <int EPI, bool SCALE>
static cudaError_t launch_tc_t(bool pair, const CUtensorMap& mx, const CUtensorMap& mw, int M, int N, int K,
                               const uint16_t* scales, long long up_off, const uint16_t* R, void* Y, int ldy,
                               int32_t* err, cudaStream_t s) {
  // persistent: one CTA per SM (its shared ring and 512 TMEM columns fill the SM)
  if (pair) {
    auto kern = gemm_tc_kernel<EPI, SCALE, true>;
    static std::atomic<unsigned long long> attr{0};
    FP_CUDA_TRY(smem_limit_once(kern, TcGeom<true>::kSmem, &attr));
    const long long pairs = std::min<long long>(tc_tiles(EPI, M, N, 2), tc_sms() / 2);
    cudaLaunchConfig_t cfg = {};
    cfg.gridDim = dim3((unsigned)(2 * pairs));
    cfg.blockDim = dim3(kTcThreads);
    cfg.dynamicSmemBytes = TcGeom<true>::kSmem;
    cfg.stream = s;
    cudaLaunchAttribute at[2];
    at[0].id = cudaLaunchAttributeProgrammaticStreamSerialization;
    at[0].val.programmaticStreamSerializationAllowed = g_pdl ? 1 : 0;
    at[1].id = cudaLaunchAttributeClusterDimension;
    at[1].val.clusterDim.x = 2, at[1].val.clusterDim.y = 1, at[1].val.clusterDim.z = 1;
    cfg.attrs = at;
    cfg.numAttrs = 2;
    return cudaLaunchKernelEx(&cfg, kern, mx, mw, M, N, K, scales, up_off, R, Y, ldy, err);
  }
  auto kern = gemm_tc_kernel<EPI, SCALE, false>;
  static std::atomic<unsigned long long> attr{0};
  FP_CUDA_TRY(smem_limit_once(kern, TcGeom<false>::kSmem, &attr));
  return launch(kern, dim3((unsigned)std::min<long long>(tc_tiles(EPI, M, N, 1), tc_sms())), dim3(kTcThreads),
                (size_t)TcGeom<false>::kSmem, s, mx, mw, M, N, K, scales, up_off, R, Y, ldy, err);
}

template <int EPI>
static cudaError_t launch_tc_e(bool sc, bool pair, const CUtensorMap& mx, const CUtensorMap& mw, int M, int N, int K,
                               const uint16_t* scales, long long up_off, const uint16_t* R, void* Y, int ldy,
                               int32_t* err, cudaStream_t s) {
  return sc ? launch_tc_t<EPI, true>(pair, mx, mw, M, N, K, scales, up_off, R, Y, ldy, err, s)
            : launch_tc_t<EPI, false>(pair, mx, mw, M, N, K, scales, up_off, R, Y, ldy, err, s);
}

static cudaError_t launch_tc_any(int epi, bool sc, bool pair, const CUtensorMap& mx, const CUtensorMap& mw, int M, int N,
                                 int K, const uint16_t* scales, long long up_off, const uint16_t* R, void* Y, int ldy,
                                 int32_t* err, cudaStream_t s) {
  switch (epi) {
    case FP_EPI_STORE: return launch_tc_e<FP_EPI_STORE>(sc, pair, mx, mw, M, N, K, scales, up_off, R, Y, ldy, err, s);
    case FP_EPI_RESID: return launch_tc_e<FP_EPI_RESID>(sc, pair, mx, mw, M, N, K, scales, up_off, R, Y, ldy, err, s);
    case FP_EPI_SWIGLU: return launch_tc_e<FP_EPI_SWIGLU>(sc, pair, mx, mw, M, N, K, scales, up_off, R, Y, ldy, err, s);
    default: return launch_tc_e<FP_EPI_F32>(sc, pair, mx, mw, M, N, K, scales, up_off, R, Y, ldy, err, s);
  }
}

// Expands a band into out [nr * cols][K] bf16: rows c0 .. of the matrix and, with
// SwiGLU (nr 2), rows Nout + c0 .. behind them.
template <int WQ>
static cudaError_t dequant_band(const void* codes, const uint16_t* scales, const uint16_t* zeros, int nr, int Nout, int c0,
                                int cols, int K, uint16_t* out, const int32_t* inv, cudaStream_t s) {
  int tx = kDqThreads;  // threads along a row: the fewest that take it in one block
  while (tx > 8 && tx / 2 * kDqWords * 8 >= K) tx /= 2;
  const int per = tx * kDqWords * 8, ty = kDqThreads / tx;  // elements of a row, rows per block
  return launch(dequant_kernel<WQ>, dim3((K + per - 1) / per, std::min((nr * cols + ty - 1) / ty, 65535)), dim3(tx, ty), 0,
                s, codes, scales, zeros, (long long)c0, (long long)Nout + c0, cols, nr * cols, K, out, inv);
}

cudaError_t launch_gemm_tc(int wquant, int epi, const uint16_t* x, int M, int N, int K, const void* codes,
                           const uint16_t* scales, const uint16_t* zeros, const uint16_t* residual, void* y,
                           void* ws, size_t ws_bytes, int32_t* err, cudaStream_t s, const int32_t* inv) {
  const int nr = epi == FP_EPI_SWIGLU ? 2 : 1;
  const int Nout = nr == 2 ? N / 2 : N;
  // rows of a weight box, per band: half a tile where a pair shares it or the gate and the up rows do
  auto wbox = [&](bool pair) { return epi == FP_EPI_SWIGLU || pair ? 128 : 256; };
  const bool sc = wquant == FP_W_INT8;
  CUtensorMap mx, mw;
  if (!make_map(&mx, x, M, K, kTcBM)) return cudaErrorInvalidValue;
  if (wquant == FP_W_BF16) {
    const bool pair = tc_pair(wquant, epi, M, N, K);
    if (!make_map(&mw, codes, N, K, wbox(pair))) return cudaErrorInvalidValue;
    return launch_tc_any(epi, sc, pair, mx, mw, M, N, K, scales, Nout, residual, y, Nout, err, s);
  }
  if (!ws || ws_bytes < gemm_tc_ws_bytes(wquant, N, K)) return cudaErrorInvalidValue;
  // band by band of output columns: expand the band's rows (SwiGLU: its gate
  // rows, then its up rows) into the scratch, then multiply
  uint16_t* w = (uint16_t*)ws;
  const int band = band_cols(epi, N, K);
  for (int c0 = 0; c0 < Nout; c0 += band) {
    const int cols = std::min(band, Nout - c0);
    switch (wquant) {
      case FP_W_INT8:
        FP_CUDA_TRY(dequant_band<FP_W_INT8>(codes, scales, zeros, nr, Nout, c0, cols, K, w, inv, s));
        break;
      case FP_W_GPTQ4:
        FP_CUDA_TRY(dequant_band<FP_W_GPTQ4>(codes, scales, zeros, nr, Nout, c0, cols, K, w, inv, s));
        break;
      default:
        FP_CUDA_TRY(dequant_band<FP_W_INT4_G128>(codes, scales, zeros, nr, Nout, c0, cols, K, w, inv, s));
    }
    const bool pair = tc_pair(wquant, epi, M, nr * cols, K);
    if (!make_map(&mw, w, (long long)nr * cols, K, wbox(pair))) return cudaErrorInvalidValue;
    const uint16_t* r = residual ? residual + c0 : nullptr;
    void* yb = epi == FP_EPI_F32 ? (void*)((float*)y + c0) : (void*)((uint16_t*)y + c0);
    const bool was = g_pdl;
    g_pdl = true;  // the GEMM's set-up overlaps the expansion
    const cudaError_t e =
        launch_tc_any(epi, sc, pair, mx, mw, M, nr * cols, K, sc ? scales + c0 : scales, Nout, r, yb, Nout, err, s);
    g_pdl = was;
    FP_CUDA_TRY(e);
  }
  return cudaSuccess;
}

}  // namespace fpk

extern "C" int fp_debug_set_wait_limit(long long rounds) {
  const long long v = rounds < 0 ? fpk::kTcSpinLimit : std::min(rounds, fpk::kTcSpinLimit);
  return cudaMemcpyToSymbol(g_stage_wait_limit, &v, sizeof v) == cudaSuccess ? FP_OK : FP_ERR_CUDA;
}
