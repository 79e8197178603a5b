// PTX wrappers for the 5th-generation tensor core path (tcgen05, TMEM, TMA,
// mbarrier) shared by the prefill GEMM and the quantised decode linear.
// sm_103a only.
#pragma once

#include <cuda.h>

#include "common.cuh"

namespace fpk {

constexpr long long kTcSpinLimit = 1LL << 20;  // try_wait rounds; legit waits here are < 1 ms

FP_DEV uint32_t smem_u32(const void* p) { return (uint32_t)__cvta_generic_to_shared(p); }

FP_DEV void mbar_init(uint64_t* bar, uint32_t count) {
  asm volatile("mbarrier.init.shared::cta.b64 [%0], %1;" ::"r"(smem_u32(bar)), "r"(count) : "memory");
}
FP_DEV void mbar_expect_tx(uint64_t* bar, uint32_t bytes) {
  asm volatile("mbarrier.arrive.expect_tx.shared::cta.b64 _, [%0], %1;" ::"r"(smem_u32(bar)), "r"(bytes) : "memory");
}
FP_DEV void mbar_arrive(uint64_t* bar) {
  asm volatile("mbarrier.arrive.shared::cta.b64 _, [%0];" ::"r"(smem_u32(bar)) : "memory");
}
// Bounded wait for the completion of phase `parity`; false after the limit.
FP_DEV bool mbar_wait(uint64_t* bar, uint32_t parity) {
  const uint32_t a = smem_u32(bar);
  for (long long it = 0; it < kTcSpinLimit; ++it) {
    uint32_t done;
    asm volatile(
        "{\n .reg .pred p;\n mbarrier.try_wait.parity.shared::cta.b64 p, [%1], %2;\n selp.u32 %0, 1, 0, p;\n}\n"
        : "=r"(done)
        : "r"(a), "r"(parity)
        : "memory");
    if (done) return true;
  }
  return false;
}

// As mbar_wait, giving up after `limit` rounds (at most kTcSpinLimit); limit
// 0 gives up at once.
FP_DEV bool mbar_wait_n(uint64_t* bar, uint32_t parity, long long limit) {
  const uint32_t a = smem_u32(bar);
  for (long long it = 0; it < kTcSpinLimit; ++it) {
    if (it >= limit) return false;
    uint32_t done;
    asm volatile(
        "{\n .reg .pred p;\n mbarrier.try_wait.parity.shared::cta.b64 p, [%1], %2;\n selp.u32 %0, 1, 0, p;\n}\n"
        : "=r"(done)
        : "r"(a), "r"(parity)
        : "memory");
    if (done) return true;
  }
  return false;
}

// As mbar_wait, but a thread that finds the phase still open sleeps a little
// before it polls again, so many waiting warps leave the issue slots to the
// warps that have work.
FP_DEV bool mbar_wait_sleep(uint64_t* bar, uint32_t parity) {
  const uint32_t a = smem_u32(bar);
  for (long long it = 0; it < kTcSpinLimit; ++it) {
    uint32_t done;
    asm volatile(
        "{\n .reg .pred p;\n mbarrier.try_wait.parity.shared::cta.b64 p, [%1], %2;\n selp.u32 %0, 1, 0, p;\n}\n"
        : "=r"(done)
        : "r"(a), "r"(parity)
        : "memory");
    if (done) return true;
    __nanosleep(32);
  }
  return false;
}

FP_DEV void tma_load_2d(void* dst, const CUtensorMap* map, int x, int y, uint64_t* bar) {
  asm volatile(
      "cp.async.bulk.tensor.2d.shared::cluster.global.mbarrier::complete_tx::bytes [%0], [%1, {%2, %3}], [%4];" ::"r"(
          smem_u32(dst)),
      "l"(map), "r"(x), "r"(y), "r"(smem_u32(bar))
      : "memory");
}

// One lane of a converged warp (always the same one).  A warp whose lanes all
// run the issuing loop, with only the MMAs and commits behind this, keeps their
// descriptors in uniform registers; a loop that one lane runs alone moves every
// operand of every MMA there first, which took longer than the MMA.
FP_DEV bool elect_one() {
  uint32_t p;
  asm volatile("{\n .reg .pred q;\n elect.sync _|q, 0xffffffff;\n selp.u32 %0, 1, 0, q;\n}\n" : "=r"(p));
  return p != 0;
}

// 1-D bulk copy: bytes a multiple of 16, both addresses 16-byte aligned.
FP_DEV void bulk_load(void* dst, const void* src, uint32_t bytes, uint64_t* bar) {
  asm volatile("cp.async.bulk.shared::cluster.global.mbarrier::complete_tx::bytes [%0], [%1], %2, [%3];" ::"r"(
                   smem_u32(dst)),
               "l"(src), "r"(bytes), "r"(smem_u32(bar))
               : "memory");
}

// Shared-memory matrix descriptor: K-major, 128-byte swizzle, 8-row groups
// 1024 bytes apart (stride byte offset), fixed field 0b001 at bit 46.
FP_DEV uint64_t sdesc(uint32_t saddr) {
  uint64_t d = 0;
  d |= (uint64_t)((saddr & 0x3FFFF) >> 4);
  d |= (uint64_t)1 << 16;              // leading byte offset (unused for swizzled K-major)
  d |= (uint64_t)(1024 >> 4) << 32;    // stride byte offset
  d |= (uint64_t)1 << 46;              // fixed 0b001
  d |= (uint64_t)2 << 61;              // 128-byte swizzle
  return d;
}

// Instruction descriptor, kind::f16: fp32 accumulator, bf16 A and B, both
// K-major, N >> 3 at bit 17, M >> 4 at bit 24.
constexpr uint32_t tc_idesc(int m, int n) {
  return (1u << 4) | (1u << 7) | (1u << 10) | ((uint32_t)(n >> 3) << 17) | ((uint32_t)(m >> 4) << 24);
}

// D (TMEM) (+)= A (shared, descriptor) x B (shared, descriptor).
FP_DEV void tc_mma(uint32_t tmem_d, uint64_t adesc, uint64_t bdesc, uint32_t idesc, uint32_t accumulate) {
  asm volatile(
      "{\n .reg .pred p;\n setp.ne.b32 p, %4, 0;\n"
      " tcgen05.mma.cta_group::1.kind::f16 [%0], %1, %2, %3, p;\n}\n" ::"r"(tmem_d),
      "l"(adesc), "l"(bdesc), "r"(idesc), "r"(accumulate)
      : "memory");
}
// D (TMEM) (+)= A (TMEM: row i in lane i, two K elements per 32-bit column)
// x B (shared, descriptor).
FP_DEV void tc_mma_ts(uint32_t tmem_d, uint32_t tmem_a, uint64_t bdesc, uint32_t idesc, uint32_t accumulate) {
  asm volatile(
      "{\n .reg .pred p;\n setp.ne.b32 p, %4, 0;\n"
      " tcgen05.mma.cta_group::1.kind::f16 [%0], [%1], %2, %3, p;\n}\n" ::"r"(tmem_d),
      "r"(tmem_a), "l"(bdesc), "r"(idesc), "r"(accumulate)
      : "memory");
}
// As tc_mma_ts for 8-bit operands (kind::f8f6f4, K 32 per instruction): A
// four K elements per 32-bit TMEM column.
FP_DEV void tc_mma_ts_f8(uint32_t tmem_d, uint32_t tmem_a, uint64_t bdesc, uint32_t idesc, uint32_t accumulate) {
  asm volatile(
      "{\n .reg .pred p;\n setp.ne.b32 p, %4, 0;\n"
      " tcgen05.mma.cta_group::1.kind::f8f6f4 [%0], [%1], %2, %3, p;\n}\n" ::"r"(tmem_d),
      "r"(tmem_a), "l"(bdesc), "r"(idesc), "r"(accumulate)
      : "memory");
}
// Instruction descriptor, kind::f8f6f4: fp32 accumulator, e4m3 A and B, both K-major.
constexpr uint32_t tc_idesc_e4m3(int m, int n) {
  return (1u << 4) | ((uint32_t)(n >> 3) << 17) | ((uint32_t)(m >> 4) << 24);
}
FP_DEV void tc_commit(uint64_t* bar) {
  asm volatile("tcgen05.commit.cta_group::1.mbarrier::arrive::one.shared::cluster.b64 [%0];" ::"r"(smem_u32(bar))
               : "memory");
}
// ---- CTA pairs (clusters of two, cta_group::2): the even CTA issues one MMA for
// both; its A rows and D rows are split between the two CTAs' shared and tensor
// memories (rows 0-127 and 128-255), its B rows (N) likewise.
FP_DEV uint32_t cluster_rank() {
  uint32_t r;
  asm volatile("mov.u32 %0, %%cluster_ctarank;" : "=r"(r));
  return r;
}
// The cluster address of this shared-memory location in CTA `rank` of the cluster.
FP_DEV uint32_t cluster_addr(const void* p, uint32_t rank) {
  uint32_t a;
  asm volatile("mapa.shared::cluster.u32 %0, %1, %2;" : "=r"(a) : "r"(smem_u32(p)), "r"(rank));
  return a;
}
FP_DEV void cluster_sync() {
  asm volatile("barrier.cluster.arrive.release;\nbarrier.cluster.wait.acquire;" ::: "memory");
}
FP_DEV void mbar_arrive_cluster(uint32_t bar) {
  asm volatile("mbarrier.arrive.release.cluster.shared::cluster.b64 _, [%0];" ::"r"(bar) : "memory");
}
// TMA into this CTA's shared memory, its bytes counted on a barrier of either CTA.
FP_DEV void tma_load_2d_pair(void* dst, const CUtensorMap* map, int x, int y, uint32_t bar) {
  asm volatile(
      "cp.async.bulk.tensor.2d.cta_group::2.shared::cluster.global.mbarrier::complete_tx::bytes [%0], [%1, {%2, %3}], "
      "[%4];" ::"r"(smem_u32(dst)),
      "l"(map), "r"(x), "r"(y), "r"(bar)
      : "memory");
}
FP_DEV void tc_mma_pair(uint32_t tmem_d, uint64_t adesc, uint64_t bdesc, uint32_t idesc, uint32_t accumulate) {
  asm volatile(
      "{\n .reg .pred p;\n setp.ne.b32 p, %4, 0;\n"
      " tcgen05.mma.cta_group::2.kind::f16 [%0], %1, %2, %3, p;\n}\n" ::"r"(tmem_d),
      "l"(adesc), "l"(bdesc), "r"(idesc), "r"(accumulate)
      : "memory");
}
// Arrives on this barrier in both CTAs once the MMAs issued so far have completed.
FP_DEV void tc_commit_pair(uint64_t* bar) {
  asm volatile(
      "tcgen05.commit.cta_group::2.mbarrier::arrive::one.shared::cluster.multicast::cluster.b64 [%0], %1;" ::"r"(
          smem_u32(bar)),
      "h"((uint16_t)3)
      : "memory");
}

// Orders this thread's generic-proxy shared-memory writes before later
// async-proxy reads (tcgen05.mma operands, TMA stores) of the same bytes.
FP_DEV void fence_proxy_async() { asm volatile("fence.proxy.async.shared::cta;" ::: "memory"); }
FP_DEV void tc_fence_after() { asm volatile("tcgen05.fence::after_thread_sync;" ::: "memory"); }
FP_DEV void tc_fence_before() { asm volatile("tcgen05.fence::before_thread_sync;" ::: "memory"); }

#define FP_R8(b) "=r"(r[b]), "=r"(r[b + 1]), "=r"(r[b + 2]), "=r"(r[b + 3]), "=r"(r[b + 4]), "=r"(r[b + 5]), \
                 "=r"(r[b + 6]), "=r"(r[b + 7])
#define FP_E8(b) "=&r"(r[b]), "=&r"(r[b + 1]), "=&r"(r[b + 2]), "=&r"(r[b + 3]), "=&r"(r[b + 4]), "=&r"(r[b + 5]), \
                 "=&r"(r[b + 6]), "=&r"(r[b + 7])
#define FP_Q8(b) "=r"(q[b]), "=r"(q[b + 1]), "=r"(q[b + 2]), "=r"(q[b + 3]), "=r"(q[b + 4]), "=r"(q[b + 5]), \
                 "=r"(q[b + 6]), "=r"(q[b + 7])
#define FP_W8(b) "r"(r[b]), "r"(r[b + 1]), "r"(r[b + 2]), "r"(r[b + 3]), "r"(r[b + 4]), "r"(r[b + 5]), \
                 "r"(r[b + 6]), "r"(r[b + 7])

// N consecutive 32-bit columns of this thread's TMEM lane (warp-wide).  The
// wait for the load sits in the same asm statement as the load: the
// destination registers are undefined until tcgen05.wait::ld, and a separate
// statement would not stop the compiler from reading them before it.
// N = 4, 8, 16, 32 or 64.
template <int N>
FP_DEV void tc_ld(uint32_t taddr, uint32_t* r) {
  if constexpr (N == 4) {
    asm volatile(
        "tcgen05.ld.sync.aligned.32x32b.x4.b32 {%0,%1,%2,%3}, [%4];\n"
        "tcgen05.wait::ld.sync.aligned;"
        : "=r"(r[0]), "=r"(r[1]), "=r"(r[2]), "=r"(r[3])
        : "r"(taddr)
        : "memory");
  } else if constexpr (N == 8) {
    asm volatile(
        "tcgen05.ld.sync.aligned.32x32b.x8.b32 {%0,%1,%2,%3,%4,%5,%6,%7}, [%8];\n"
        "tcgen05.wait::ld.sync.aligned;"
        : FP_R8(0)
        : "r"(taddr)
        : "memory");
  } else if constexpr (N == 16) {
    asm volatile(
        "tcgen05.ld.sync.aligned.32x32b.x16.b32 {%0,%1,%2,%3,%4,%5,%6,%7,%8,%9,%10,%11,%12,%13,%14,%15}, [%16];\n"
        "tcgen05.wait::ld.sync.aligned;"
        : FP_R8(0), FP_R8(8)
        : "r"(taddr)
        : "memory");
  } else if constexpr (N == 64) {
    asm volatile(
        "tcgen05.ld.sync.aligned.32x32b.x64.b32 {%0,%1,%2,%3,%4,%5,%6,%7,%8,%9,%10,%11,%12,%13,%14,%15,%16,%17,%18,"
        "%19,%20,%21,%22,%23,%24,%25,%26,%27,%28,%29,%30,%31,%32,%33,%34,%35,%36,%37,%38,%39,%40,%41,%42,%43,%44,"
        "%45,%46,%47,%48,%49,%50,%51,%52,%53,%54,%55,%56,%57,%58,%59,%60,%61,%62,%63}, [%64];\n"
        "tcgen05.wait::ld.sync.aligned;"
        : FP_R8(0), FP_R8(8), FP_R8(16), FP_R8(24), FP_R8(32), FP_R8(40), FP_R8(48), FP_R8(56)
        : "r"(taddr)
        : "memory");
  } else {
    static_assert(N == 32, "tc_ld: 4, 8, 16, 32 or 64 columns");
    asm volatile(
        "tcgen05.ld.sync.aligned.32x32b.x32.b32 {%0,%1,%2,%3,%4,%5,%6,%7,%8,%9,%10,%11,%12,%13,%14,%15,%16,%17,%18,"
        "%19,%20,%21,%22,%23,%24,%25,%26,%27,%28,%29,%30,%31}, [%32];\n"
        "tcgen05.wait::ld.sync.aligned;"
        : FP_R8(0), FP_R8(8), FP_R8(16), FP_R8(24)
        : "r"(taddr)
        : "memory");
  }
}

// tc_ld of N columns from two places with one wait (N = 8 or 16).  The first load's
// results are there before the second load's address is read, hence the early clobbers.
template <int N>
FP_DEV void tc_ld_pair(uint32_t ta, uint32_t tb, uint32_t* r, uint32_t* q) {
  if constexpr (N == 8) {
    asm volatile(
        "tcgen05.ld.sync.aligned.32x32b.x8.b32 {%0,%1,%2,%3,%4,%5,%6,%7}, [%16];\n"
        "tcgen05.ld.sync.aligned.32x32b.x8.b32 {%8,%9,%10,%11,%12,%13,%14,%15}, [%17];\n"
        "tcgen05.wait::ld.sync.aligned;"
        : FP_E8(0), FP_Q8(0)
        : "r"(ta), "r"(tb)
        : "memory");
  } else {
    static_assert(N == 16, "tc_ld_pair: 8 or 16 columns");
    asm volatile(
        "tcgen05.ld.sync.aligned.32x32b.x16.b32 {%0,%1,%2,%3,%4,%5,%6,%7,%8,%9,%10,%11,%12,%13,%14,%15}, [%32];\n"
        "tcgen05.ld.sync.aligned.32x32b.x16.b32 {%16,%17,%18,%19,%20,%21,%22,%23,%24,%25,%26,%27,%28,%29,%30,%31}, "
        "[%33];\n"
        "tcgen05.wait::ld.sync.aligned;"
        : FP_E8(0), FP_E8(8), FP_Q8(0), FP_Q8(8)
        : "r"(ta), "r"(tb)
        : "memory");
  }
}

FP_DEV void tc_ld32(uint32_t taddr, float* v) {
  uint32_t r[32];
  tc_ld<32>(taddr, r);
#pragma unroll
  for (int i = 0; i < 32; ++i) v[i] = __uint_as_float(r[i]);
}

// 32 consecutive 32-bit columns into this thread's TMEM lane (warp-wide; the
// caller issues tcgen05.wait::st before the columns are consumed).
FP_DEV void tc_st32(uint32_t taddr, const uint32_t* r) {
  asm volatile(
      "tcgen05.st.sync.aligned.32x32b.x32.b32 [%0], {%1,%2,%3,%4,%5,%6,%7,%8,%9,%10,%11,%12,%13,%14,%15,%16,%17,%18,"
      "%19,%20,%21,%22,%23,%24,%25,%26,%27,%28,%29,%30,%31,%32};" ::"r"(taddr),
      FP_W8(0), FP_W8(8), FP_W8(16), FP_W8(24)
      : "memory");
}
// 16 consecutive 32-bit columns into this thread's TMEM lane.
FP_DEV void tc_st16(uint32_t taddr, const uint32_t* r) {
  asm volatile(
      "tcgen05.st.sync.aligned.32x32b.x16.b32 [%0], {%1,%2,%3,%4,%5,%6,%7,%8,%9,%10,%11,%12,%13,%14,%15,%16};" ::"r"(
          taddr),
      FP_W8(0), FP_W8(8)
      : "memory");
}
FP_DEV void tc_wait_st() { asm volatile("tcgen05.wait::st.sync.aligned;" ::: "memory"); }

#undef FP_R8
#undef FP_E8
#undef FP_Q8
#undef FP_W8

// ---- host: tensor maps (fp_gemm_tc.cu)
// Row-major [rows][cols] matrix of elem_bytes-sized elements (2: bf16; 1 and
// 4: raw bytes and words), box [box_rows][box_cols], with swizzle_bytes 64
// or 128.
bool make_tensor_map(CUtensorMap* map, const void* base, long long rows, long long cols, int elem_bytes,
                     int box_rows, int box_cols, int swizzle_bytes);
bool tensor_maps_available();

// The sums of a row tile that several CTAs share: v[i] += sum over CTAs of the
// partials of token i at p0 + CTA * slot + i * NR * ROWS (u: the second row set of
// SwiGLU), in CTA order, for the first `m` of TB tokens.  The loads of UC CTAs are in
// flight together: one CTA after another, a tile shared by five waited out an L2
// latency five times per eight tokens.
template <int TB, int NR, int ROWS, int UC>
FP_DEV void sum_partials(const float* p0, size_t slot, int cnt, int m, float* v, float* u) {
#pragma unroll 1
  for (int cc = 0; cc < cnt; cc += UC) {
    float t[NR][UC][TB];
#pragma unroll
    for (int k = 0; k < UC; ++k)
#pragma unroll
      for (int r = 0; r < NR; ++r)
#pragma unroll
        for (int i = 0; i < TB; ++i)
          t[r][k][i] = cc + k < cnt && i < m ? __ldcg(p0 + (size_t)(cc + k) * slot + (size_t)(i * NR + r) * ROWS) : 0.f;
#pragma unroll
    for (int k = 0; k < UC; ++k)
#pragma unroll
      for (int i = 0; i < TB; ++i) {
        v[i] += t[0][k][i];
        if (NR == 2) u[i] += t[NR - 1][k][i];
      }
  }
}

}  // namespace fpk
