// nbm_tc_ptx.cuh -- inline-PTX wrappers for the Blackwell (sm_100 family)
// tensor-core path: tcgen05 MMA with TMEM accumulators, TMEM loads, bulk
// (TMA) copies and bounded mbarrier waits.
//
// Shared-memory operand image used everywhere in this library: a 128 x 128
// 16-bit matrix X[row][col] is stored as 8-row x 64-column atoms of 1024
// bytes with the 128-byte XOR swizzle (16-byte chunk index ^= row % 8):
//   byte(row, col) = (cb*16 + row/8)*1024 + (row%8)*128
//                    + (((col%64)/8 ^ row%8) * 16) + (col%8)*2,   cb = col/64.
// The same image is read by the MMA as a K-major operand (K = col) or as an
// MN-major operand (MN = col, K = row), which is what lets the forward,
// input-gradient and weight-gradient GEMMs share buffers without transposes.
#pragma once

#include <stdint.h>

namespace nbm {
namespace tc {

__device__ __forceinline__ uint32_t smem_u32(const void* p) {
  return (uint32_t)__cvta_generic_to_shared(p);
}

// First 1024-byte boundary of a dynamic shared array.  By pointer arithmetic: through
// an integer and back the compiler loses the shared address space, and every access
// becomes a generic one with 64-bit addresses (training step C2 2007 -> 1905 us per two
// steps, four layers 6.48 -> 6.10 ms, 513^3 evaluation 29.9 -> 28.3 ms without that).
__device__ __forceinline__ unsigned char* align1024(unsigned char* p) {
  return p + ((0u - smem_u32(p)) & 1023u);
}

// byte offset of element (row, col) in the swizzled 128x128 image
__host__ __device__ __forceinline__ uint32_t img_off(int row, int col) {
  const int cb = col >> 6, cc = col & 63;
  return (uint32_t)((cb * 16 + (row >> 3)) * 1024 + (row & 7) * 128 +
                    ((((cc >> 3) ^ row) & 7) << 4) + (cc & 7) * 2);
}

// ---- shared-memory matrix descriptors (tcgen05 format, SWIZZLE_128B) ----
// 64 bits: address >> 4 | leading offset >> 4 in the low word; stride offset (8-row
// groups, 1024 bytes) >> 4, the tcgen05 version and the swizzle mode in the high word,
// the same for every operand here.  The low word of K-step 0 is made once per operand and
// the K-steps are additions to it (an address stays below 2^18, so none carries into the
// offset): one thread issues the 8 MMAs of a GEMM, and building 16 descriptors from
// addresses held it up (training step C2 949 -> 932 us, four layers 6.06 -> 5.94 ms).
constexpr uint32_t kDescHi = (1024u >> 4) | (1u << 14) | (2u << 29);
// K-major operand (K = image column, 16 columns per K-step): rows at 128 B inside an
// atom, 8-row groups 1024 B apart.
__device__ __forceinline__ uint32_t desc_kmajor(uint32_t base) { return (base >> 4) | (1u << 16); }
__device__ __forceinline__ constexpr uint32_t kstep_kmajor(int k) {
  return (uint32_t)(k >> 2) * (16384u >> 4) + (uint32_t)(k & 3) * (32u >> 4);
}
// MN-major operand (MN = image column, K = image row, 16 rows per K-step): 64-column
// blocks 16384 B apart (LBO), 8-row groups 1024 B apart.
__device__ __forceinline__ uint32_t desc_mnmajor(uint32_t base) {
  return (base >> 4) | ((16384u >> 4) << 16);
}
__device__ __forceinline__ constexpr uint32_t kstep_mnmajor(int k) {
  return (uint32_t)k * (2048u >> 4);
}

// Instruction descriptor of kind::f16, M = 128, N a multiple of 16 up to 256, FP32
// accumulate.  is_bf16: both operands BF16 (else both FP16).  a_mn / b_mn: MN-major.
__host__ __device__ __forceinline__ uint32_t idesc_f16_n(bool is_bf16, bool a_mn, bool b_mn,
                                                         uint32_t n) {
  const uint32_t fmt = is_bf16 ? 1u : 0u;
  return (1u << 4) | (fmt << 7) | (fmt << 10) | ((a_mn ? 1u : 0u) << 15) |
         ((b_mn ? 1u : 0u) << 16) | ((n >> 3) << 17) | ((128u >> 4) << 24);
}

// ---- named barriers (ids 1..15; id 0 is __syncthreads) over `n` threads ----
__device__ __forceinline__ void named_sync(uint32_t id, uint32_t n) {
  asm volatile("bar.sync %0, %1;" ::"r"(id), "r"(n) : "memory");
}
// Named barrier that also returns whether `pred` held in any participating thread.
__device__ __forceinline__ bool named_sync_or(uint32_t id, uint32_t n, bool pred) {
  uint32_t r;
  asm volatile(
      "{\n\t.reg .pred p, q;\n\tsetp.ne.u32 p, %1, 0;\n\t"
      "bar.red.or.pred q, %2, %3, p;\n\tselp.u32 %0, 1, 0, q;\n\t}\n"
      : "=r"(r)
      : "r"((uint32_t)pred), "r"(id), "r"(n)
      : "memory");
  return r != 0;
}

// Release store / acquire load of a shared-memory flag (CTA scope).
__device__ __forceinline__ void st_release_s32(int* p, int v) {
  asm volatile("st.release.cta.shared::cta.b32 [%0], %1;" ::"r"(smem_u32(p)), "r"(v) : "memory");
}
__device__ __forceinline__ int ld_acquire_s32(const int* p) {
  int v;
  asm volatile("ld.acquire.cta.shared::cta.b32 %0, [%1];" : "=r"(v) : "r"(smem_u32(p)) : "memory");
  return v;
}

// Asynchronous 4-byte global -> shared copy (LDGSTS) and its completion wait.
__device__ __forceinline__ void cp_async4(uint32_t dst_smem, const void* src) {
  asm volatile("cp.async.ca.shared.global [%0], [%1], 4;" ::"r"(dst_smem), "l"(src) : "memory");
}
__device__ __forceinline__ void cp_async_wait_all() {
  asm volatile("cp.async.wait_all;" ::: "memory");
}

// ---- tcgen05 ----
__device__ __forceinline__ void tmem_alloc(uint32_t dst_smem, uint32_t ncols) {
  asm volatile("tcgen05.alloc.cta_group::1.sync.aligned.shared::cta.b32 [%0], %1;" ::"r"(dst_smem),
               "r"(ncols));
  asm volatile("tcgen05.relinquish_alloc_permit.cta_group::1.sync.aligned;");
}
__device__ __forceinline__ void tmem_dealloc(uint32_t taddr, uint32_t ncols) {
  asm volatile("tcgen05.dealloc.cta_group::1.sync.aligned.b32 %0, %1;" ::"r"(taddr), "r"(ncols));
}
// (adesc, bdesc: low descriptor words)
__device__ __forceinline__ void mma_f16(uint32_t d_tmem, uint32_t adesc, uint32_t bdesc,
                                        uint32_t idesc, uint32_t accumulate) {
  asm volatile(
      "{\n\t.reg .pred p;\n\t.reg .b64 da, db;\n\tsetp.ne.b32 p, %4, 0;\n\t"
      "mov.b64 da, {%1, %5};\n\tmov.b64 db, {%2, %5};\n\t"
      "tcgen05.mma.cta_group::1.kind::f16 [%0], da, db, %3, p;\n\t}\n" ::"r"(d_tmem),
      "r"(adesc), "r"(bdesc), "r"(idesc), "r"(accumulate), "r"(kDescHi));
}
// The same MMA with the A operand in TMEM: a_tmem addresses lane 0 and the
// first of the K/2 32-bit columns of this K-step (row m of A in lane m, two
// 16-bit elements per column, the lower K index in the lower half).
__device__ __forceinline__ void mma_f16_ta(uint32_t d_tmem, uint32_t a_tmem, uint32_t bdesc,
                                           uint32_t idesc, uint32_t accumulate) {
  asm volatile(
      "{\n\t.reg .pred p;\n\t.reg .b64 db;\n\tsetp.ne.b32 p, %4, 0;\n\t"
      "mov.b64 db, {%2, %5};\n\t"
      "tcgen05.mma.cta_group::1.kind::f16 [%0], [%1], db, %3, p;\n\t}\n" ::"r"(d_tmem),
      "r"(a_tmem), "r"(bdesc), "r"(idesc), "r"(accumulate), "r"(kDescHi));
}
// 16 consecutive 32-bit columns from each lane of the warp's quadrant
// (shape 32x32b: lane l of the warp writes TMEM lane base + l).
__device__ __forceinline__ void tmem_st16(uint32_t taddr, const uint32_t (&v)[16]) {
  asm volatile(
      "tcgen05.st.sync.aligned.32x32b.x16.b32 [%0], "
      "{%1,%2,%3,%4,%5,%6,%7,%8,%9,%10,%11,%12,%13,%14,%15,%16};" ::"r"(taddr),
      "r"(v[0]), "r"(v[1]), "r"(v[2]), "r"(v[3]), "r"(v[4]), "r"(v[5]), "r"(v[6]), "r"(v[7]),
      "r"(v[8]), "r"(v[9]), "r"(v[10]), "r"(v[11]), "r"(v[12]), "r"(v[13]), "r"(v[14]),
      "r"(v[15])
      : "memory");
}
__device__ __forceinline__ void tmem_wait_st() {
  asm volatile("tcgen05.wait::st.sync.aligned;" ::: "memory");
}
// Weights of hidden layers 1..nl from their shared-memory images (img_bytes
// apart) into TMEM as the A operand of GEMMs: layer l in the 64 columns from
// tw + 64 (l-1), row u of W in the calling lane (tw carries the warp's lane
// quadrant), W[u][2c] and W[u][2c+1] in column c.  Out of line: it runs once
// per network and keeps its registers out of the callers' hot loops.
static __device__ __noinline__ void stage_weights_tmem(const unsigned char* img0, int img_bytes,
                                                       uint32_t tw, int u, int nl) {
  for (int l = 0; l < nl; ++l) {
    const unsigned char* img = img0 + l * img_bytes;
#pragma unroll 1
    for (int j = 0; j < 4; ++j) {
      uint32_t v[16];
#pragma unroll
      for (int c = 0; c < 16; ++c)
        v[c] = *reinterpret_cast<const uint32_t*>(img + img_off(u, 2 * (16 * j + c)));
      tmem_st16(tw + 64u * (uint32_t)l + 16u * (uint32_t)j, v);
    }
  }
  tmem_wait_st();
}
__device__ __forceinline__ void mma_commit(uint32_t mbar) {
  asm volatile(
      "tcgen05.commit.cta_group::1.mbarrier::arrive::one.shared::cluster.b64 [%0];" ::"r"(mbar)
      : "memory");
}
__device__ __forceinline__ void fence_before_sync() {
  asm volatile("tcgen05.fence::before_thread_sync;" ::: "memory");
}
__device__ __forceinline__ void fence_after_sync() {
  asm volatile("tcgen05.fence::after_thread_sync;" ::: "memory");
}
__device__ __forceinline__ void fence_proxy_async() {
  asm volatile("fence.proxy.async.shared::cta;" ::: "memory");
}
// 32 consecutive TMEM columns of this warp's 32 lanes (one lane per thread)
__device__ __forceinline__ void tmem_ld32(uint32_t taddr, float* v) {
  uint32_t r[32];
  asm volatile(
      "tcgen05.ld.sync.aligned.32x32b.x32.b32 "
      "{%0,%1,%2,%3,%4,%5,%6,%7,%8,%9,%10,%11,%12,%13,%14,%15,"
      "%16,%17,%18,%19,%20,%21,%22,%23,%24,%25,%26,%27,%28,%29,%30,%31}, [%32];"
      : "=r"(r[0]), "=r"(r[1]), "=r"(r[2]), "=r"(r[3]), "=r"(r[4]), "=r"(r[5]), "=r"(r[6]),
        "=r"(r[7]), "=r"(r[8]), "=r"(r[9]), "=r"(r[10]), "=r"(r[11]), "=r"(r[12]), "=r"(r[13]),
        "=r"(r[14]), "=r"(r[15]), "=r"(r[16]), "=r"(r[17]), "=r"(r[18]), "=r"(r[19]),
        "=r"(r[20]), "=r"(r[21]), "=r"(r[22]), "=r"(r[23]), "=r"(r[24]), "=r"(r[25]),
        "=r"(r[26]), "=r"(r[27]), "=r"(r[28]), "=r"(r[29]), "=r"(r[30]), "=r"(r[31])
      : "r"(taddr));
  asm volatile("tcgen05.wait::ld.sync.aligned;" ::: "memory");
#pragma unroll
  for (int i = 0; i < 32; ++i) v[i] = __uint_as_float(r[i]);
}
// 16 consecutive TMEM columns of this warp's 32 lanes
__device__ __forceinline__ void tmem_ld16(uint32_t taddr, float* v) {
  uint32_t r[16];
  asm volatile(
      "tcgen05.ld.sync.aligned.32x32b.x16.b32 "
      "{%0,%1,%2,%3,%4,%5,%6,%7,%8,%9,%10,%11,%12,%13,%14,%15}, [%16];"
      : "=r"(r[0]), "=r"(r[1]), "=r"(r[2]), "=r"(r[3]), "=r"(r[4]), "=r"(r[5]), "=r"(r[6]),
        "=r"(r[7]), "=r"(r[8]), "=r"(r[9]), "=r"(r[10]), "=r"(r[11]), "=r"(r[12]), "=r"(r[13]),
        "=r"(r[14]), "=r"(r[15])
      : "r"(taddr));
  asm volatile("tcgen05.wait::ld.sync.aligned;" ::: "memory");
#pragma unroll
  for (int i = 0; i < 16; ++i) v[i] = __uint_as_float(r[i]);
}
// ---- mbarrier + bulk copy ----
__device__ __forceinline__ void mbar_init(uint32_t mbar, uint32_t count) {
  asm volatile("mbarrier.init.shared::cta.b64 [%0], %1;" ::"r"(mbar), "r"(count));
}
__device__ __forceinline__ void fence_mbar_init() {
  asm volatile("fence.mbarrier_init.release.cluster;" ::: "memory");
}
__device__ __forceinline__ void mbar_expect_tx(uint32_t mbar, uint32_t bytes) {
  asm volatile("mbarrier.arrive.expect_tx.shared::cta.b64 _, [%0], %1;" ::"r"(mbar), "r"(bytes)
               : "memory");
}
// Plain arrival (count 1) without a transaction: stands in for an MMA commit
// that is not issued, so that the waiters wake up.
__device__ __forceinline__ void mbar_arrive(uint32_t mbar) {
  asm volatile("mbarrier.arrive.shared::cta.b64 _, [%0];" ::"r"(mbar) : "memory");
}
__device__ __forceinline__ bool mbar_try_wait(uint32_t mbar, uint32_t parity) {
  uint32_t ok;
  asm volatile(
      "{\n\t.reg .pred p;\n\tmbarrier.try_wait.parity.shared::cta.b64 p, [%1], %2;\n\t"
      "selp.b32 %0, 1, 0, p;\n\t}\n"
      : "=r"(ok)
      : "r"(mbar), "r"(parity)
      : "memory");
  return ok != 0;
}
// The same with a suspend-time hint: the thread may sleep up to `hint_ns`
// nanoseconds and is woken when the phase completes, instead of spinning on
// issue slots that other warps could use.
__device__ __forceinline__ bool mbar_try_wait_sleep(uint32_t mbar, uint32_t parity,
                                                    uint32_t hint_ns) {
  uint32_t ok;
  asm volatile(
      "{\n\t.reg .pred p;\n\tmbarrier.try_wait.parity.shared::cta.b64 p, [%1], %2, %3;\n\t"
      "selp.b32 %0, 1, 0, p;\n\t}\n"
      : "=r"(ok)
      : "r"(mbar), "r"(parity), "r"(hint_ns)
      : "memory");
  return ok != 0;
}
// Bounded wait: gives up after ~`budget` clock cycles and returns false.
__device__ __forceinline__ bool mbar_wait_bounded(uint32_t mbar, uint32_t parity,
                                                  long long budget = 4000000000LL) {
  if (mbar_try_wait(mbar, parity)) return true;
  const long long t0 = clock64();
  while (true) {
    if (mbar_try_wait_sleep(mbar, parity, 20000u)) return true;
    if (clock64() - t0 > budget) return false;
  }
}
__device__ __forceinline__ void bulk_g2s(uint32_t dst_smem, const void* src, uint32_t bytes,
                                         uint32_t mbar) {
  asm volatile(
      "cp.async.bulk.shared::cluster.global.mbarrier::complete_tx::bytes [%0], [%1], %2, [%3];" ::"r"(
          dst_smem),
      "l"(src), "r"(bytes), "r"(mbar)
      : "memory");
}

}  // namespace tc
}  // namespace nbm
