// Helpers of the tensor-core contractions (as_gemm_tc.cu, as_gemm_split.cu): mbarriers with bounded waits, TMA, tcgen05
// descriptors and instructions, staging tiles.
#pragma once

#include <cuda.h>

#include "as_internal.cuh"

namespace as {
namespace {

constexpr uint32_t WAIT_LIMIT = 1u << 22;
enum { MAJ_K = 0, MAJ_MN = 1 };

__device__ __forceinline__ uint32_t smem_u32(const void* p) { return (uint32_t)__cvta_generic_to_shared(p); }

__device__ __forceinline__ void mbar_init(uint64_t* bar, uint32_t count) {
  asm volatile("mbarrier.init.shared::cta.b64 [%0], %1;" ::"r"(smem_u32(bar)), "r"(count));
}
__device__ __forceinline__ void mbar_expect_tx(uint64_t* bar, uint32_t bytes) {
  asm volatile("mbarrier.arrive.expect_tx.shared::cta.b64 _, [%0], %1;" ::"r"(smem_u32(bar)), "r"(bytes) : "memory");
}
// bounded wait: returns false if the phase did not complete within WAIT_LIMIT polls
__device__ __forceinline__ bool mbar_wait(uint64_t* bar, uint32_t parity, volatile int* abort_flag = nullptr) {
  const uint32_t addr = smem_u32(bar);
  for (uint32_t it = 0; it < WAIT_LIMIT; ++it) {
    uint32_t ok;
    asm volatile(
        "{\n\t.reg .pred p;\n\t"
        "mbarrier.try_wait.parity.shared::cta.b64 p, [%1], %2;\n\t"
        "selp.u32 %0, 1, 0, p;\n\t}"
        : "=r"(ok)
        : "r"(addr), "r"(parity)
        : "memory");
    if (ok) return true;
    if (abort_flag && *abort_flag) return false;
  }
  return false;
}
// One lane of a converged warp.  The warps that issue TMA and MMA instructions run their loops as a whole and elect the lane
// around the instructions alone: their operands then are warp-uniform to the compiler.  (With the whole loop inside a
// lane-0 branch every block of the contraction took some 750 cycles whatever its size.)
__device__ __forceinline__ bool elect_one() {
  uint32_t p;
  asm volatile("{\n\t.reg .pred p;\n\telect.sync _|p, 0xffffffff;\n\tselp.u32 %0, 1, 0, p;\n\t}" : "=r"(p));
  return p != 0;
}
__device__ __forceinline__ void tma_load_3d(void* dst, const CUtensorMap* tm, int c0, int c1, int c2, uint64_t* bar) {
  asm volatile(
      "cp.async.bulk.tensor.3d.shared::cluster.global.mbarrier::complete_tx::bytes [%0], [%1, {%2, %3, %4}], [%5];"
      ::"r"(smem_u32(dst)), "l"(tm), "r"(c0), "r"(c1), "r"(c2), "r"(smem_u32(bar)) : "memory");
}

// shared-memory matrix descriptor, 128-byte swizzle, descriptor version 1
__device__ __forceinline__ uint64_t make_desc(uint32_t saddr, uint32_t lbo_bytes, uint32_t sbo_bytes) {
  uint64_t d = 0;
  d |= (uint64_t)((saddr >> 4) & 0x3FFF);
  d |= (uint64_t)((lbo_bytes >> 4) & 0x3FFF) << 16;
  d |= (uint64_t)((sbo_bytes >> 4) & 0x3FFF) << 32;
  d |= (uint64_t)1 << 46;
  d |= (uint64_t)2 << 61;
  return d;
}

__device__ __forceinline__ void umma_bf16(uint32_t d_tmem, uint64_t adesc, uint64_t bdesc, uint32_t idesc, uint32_t acc) {
  asm volatile(
      "{\n\t.reg .pred p;\n\tsetp.ne.b32 p, %4, 0;\n\t"
      "tcgen05.mma.cta_group::1.kind::f16 [%0], %1, %2, %3, p;\n\t}"
      ::"r"(d_tmem), "l"(adesc), "l"(bdesc), "r"(idesc), "r"(acc)
      : "memory");
}
__device__ __forceinline__ void umma_commit(uint64_t* bar) {
  asm volatile("tcgen05.commit.cta_group::1.mbarrier::arrive::one.shared::cluster.b64 [%0];" ::"r"(smem_u32(bar))
               : "memory");
}
__device__ __forceinline__ void tmem_ld16(uint32_t taddr, uint32_t (&r)[16]) {
  asm volatile(
      "tcgen05.ld.sync.aligned.32x32b.x16.b32 {%0,%1,%2,%3,%4,%5,%6,%7,%8,%9,%10,%11,%12,%13,%14,%15}, [%16];"
      : "=r"(r[0]), "=r"(r[1]), "=r"(r[2]), "=r"(r[3]), "=r"(r[4]), "=r"(r[5]), "=r"(r[6]), "=r"(r[7]), "=r"(r[8]),
        "=r"(r[9]), "=r"(r[10]), "=r"(r[11]), "=r"(r[12]), "=r"(r[13]), "=r"(r[14]), "=r"(r[15])
      : "r"(taddr));
  asm volatile("tcgen05.wait::ld.sync.aligned;" ::: "memory");
}

// softplus(u) = max(u, 0) + log(1 + z), z = exp(-|u|) in (0, 1].  SP_LOG: two MUFU ops (ex2, lg2) and a short series for small z,
// where forming 1 + z would lose z's low bits (relative error of the result < 1e-5 from Delta = 0.02 on, 2e-5 below); kept for
// the calls that make up a step of a bf16 stack (Plan.ordered), which turns a change of Delta's last bits into some per cent of its outputs.
__device__ __forceinline__ float softplus_log(float u) {
  const float z = ex2_approx(-fabsf(u) * LOG2E);
  float l;
  asm("lg2.approx.ftz.f32 %0, %1;" : "=f"(l) : "f"(1.f + z));
  const float big = l * LN2;
  const float small = z * fmaf(z, fmaf(z, 1.f / 3.f, -0.5f), 1.f);   // z - z^2/2 + z^3/3
  return fmaxf(u, 0.f) + (z < 0.0078125f ? small : big);
}
// SP_POLY, SP_FINE, of a packed pair: log(1 + z) is z Q(z) with the polynomial Q of least relative error on [0, 1] (Remez exchange;
// degree 7: 1.9e-7, degree 9: 4.7e-9): packed multiply-adds, where the logarithm takes a second MUFU operation and the series beside it.
// SP_POLY, degree 7: with fp32 rounding and an exact exp2 the relative error is 3.9e-7 for u in [-2, 10], 5.4e-7 in [-10, -2], 8.1e-7 in
// [-20, -10] and 3.6e-6 in [-80, -60], for the product -|u| log2 e is rounded.  SP_FINE, degree 9, puts that rounding back as a factor of z:
// 2.1e-7 for all u.  ex2.approx adds up to 2.4e-7 to either.
// The projections of 131,072 x 768: 174 us with SP_LOG, 166 with SP_POLY.
enum { SP_LOG = 0, SP_POLY = 1, SP_FINE = 2 };
template <int SP> __device__ __forceinline__ f2 softplus2(f2 u) {
  constexpr bool FINE = SP == SP_FINE;
  float u0, u1;
  upk(u, u0, u1);
  if (SP == SP_LOG) return pk(softplus_log(u0), softplus_log(u1));
  auto expm = [](float v) {
    const float a = -fabsf(v), t = __fmul_rn(a, LOG2E), z = ex2_approx(t);
    if (!FINE) return z;
    const float back = fmaf(a, 1.925963e-8f, fmaf(a, LOG2E, -t));   // log2 e = LOG2E + 1.925963e-8
    return fmaf(z, back * LN2, z);
  };
  const f2 z = pk(expm(u0), expm(u1));
  constexpr int N = FINE ? 10 : 8;
  constexpr float c7[8] = {9.999998212e-01f, -4.999740422e-01f, 3.327547908e-01f, -2.449546307e-01f,
                           1.774524152e-01f, -1.076817140e-01f, 4.408963397e-02f, -8.539208211e-03f};
  constexpr float c9[10] = {1.0f, -4.999990165e-01f, 3.332996368e-01f, -2.495413423e-01f, 1.967593879e-01f,
                            -1.530559212e-01f, 1.060365513e-01f, -5.695953593e-02f, 1.985146292e-02f, -3.244025167e-03f};
  auto coef = [&](int i) { const float c = FINE ? c9[i] : c7[i < 8 ? i : 7]; return pk(c, c); };
  f2 q = coef(N - 1);
#pragma unroll
  for (int i = N - 2; i >= 0; --i) q = fma2(q, z, coef(i));
  return fma2(z, q, pk(fmaxf(u0, 0.f), fmaxf(u1, 0.f)));
}

// ---- TMA stores out of the staging tile (bulk async-groups are tracked per issuing thread) ----
__device__ __forceinline__ void fence_async_smem() { asm volatile("fence.proxy.async.shared::cta;" ::: "memory"); }
__device__ __forceinline__ void tma_store_3d(const CUtensorMap* tm, const void* src, int c0, int c1, int c2) {
  asm volatile("cp.async.bulk.tensor.3d.global.shared::cta.bulk_group [%0, {%1, %2, %3}], [%4];"
               ::"l"(tm), "r"(c0), "r"(c1), "r"(c2), "r"(smem_u32(src)) : "memory");
}
__device__ __forceinline__ void tma_reduce_add_3d(const CUtensorMap* tm, const void* src, int c0, int c1, int c2) {
  asm volatile("cp.reduce.async.bulk.tensor.3d.global.shared::cta.add.tile.bulk_group [%0, {%1, %2, %3}], [%4];"
               ::"l"(tm), "r"(c0), "r"(c1), "r"(c2), "r"(smem_u32(src)) : "memory");
}
__device__ __forceinline__ void bulk_commit() { asm volatile("cp.async.bulk.commit_group;" ::: "memory"); }
template <int N> __device__ __forceinline__ void bulk_wait_read() {
  asm volatile("cp.async.bulk.wait_group.read %0;" ::"n"(N) : "memory");
}
// byte offset of 16-byte piece q of row r in a [rows][64 B] tile under the 64-byte swizzle
__device__ __forceinline__ uint32_t swz64(int r, int q) { return (uint32_t)(r * 64 + ((q ^ ((r >> 1) & 3)) << 4)); }

__device__ __forceinline__ void mbar_arrive(uint64_t* bar) {
  asm volatile("mbarrier.arrive.shared::cta.b64 _, [%0];" ::"r"(smem_u32(bar)) : "memory");
}


}  // namespace
}  // namespace as
