// whtmix_fast.cuh -- register, tensor-memory and copy primitives shared by the kernels of whole planes (whtmix_tri.cuh and
// what builds on it, whtmix_x16.cuh).
//
// Butterflies run on register pairs with packed add/sub.f32x2 (half the instructions), and tensor memory serves as
// per-thread storage: a thread holds up to 512 fp32 in its TMEM lane.
#pragma once

#include "whtmix_kernels.cuh"

namespace whtmix {
namespace fast {

// ---------------------------------------------------------------------------------------------
// packed fp32 pairs
__device__ __forceinline__ float2 add2(float2 a, float2 b) {
  float2 r;
  asm("{.reg .b64 pa, pb, pd;\n\t"
      "mov.b64 pa, {%2, %3};\n\tmov.b64 pb, {%4, %5};\n\t"
      "add.rn.f32x2 pd, pa, pb;\n\tmov.b64 {%0, %1}, pd;}"
      : "=f"(r.x), "=f"(r.y) : "f"(a.x), "f"(a.y), "f"(b.x), "f"(b.y));
  return r;
}
__device__ __forceinline__ float2 sub2(float2 a, float2 b) {
  float2 r;
  asm("{.reg .b64 pa, pb, pd;\n\t"
      "mov.b64 pa, {%2, %3};\n\tmov.b64 pb, {%4, %5};\n\t"
      "sub.rn.f32x2 pd, pa, pb;\n\tmov.b64 {%0, %1}, pd;}"
      : "=f"(r.x), "=f"(r.y) : "f"(a.x), "f"(a.y), "f"(b.x), "f"(b.y));
  return r;
}
__device__ __forceinline__ float2 mul2(float2 a, float2 b) {
  float2 r;
  asm("{.reg .b64 pa, pb, pd;\n\t"
      "mov.b64 pa, {%2, %3};\n\tmov.b64 pb, {%4, %5};\n\t"
      "mul.rn.f32x2 pd, pa, pb;\n\tmov.b64 {%0, %1}, pd;}"
      : "=f"(r.x), "=f"(r.y) : "f"(a.x), "f"(a.y), "f"(b.x), "f"(b.y));
  return r;
}
// a * s + b with s = +-1 (exact)
__device__ __forceinline__ float2 fma2(float2 a, float2 s, float2 b) {
  float2 r;
  asm("{.reg .b64 pa, ps, pb, pd;\n\t"
      "mov.b64 pa, {%2, %3};\n\tmov.b64 ps, {%4, %5};\n\tmov.b64 pb, {%6, %7};\n\t"
      "fma.rn.f32x2 pd, pa, ps, pb;\n\tmov.b64 {%0, %1}, pd;}"
      : "=f"(r.x), "=f"(r.y) : "f"(a.x), "f"(a.y), "f"(s.x), "f"(s.y), "f"(b.x), "f"(b.y));
  return r;
}

// butterfly on two pairs: (a, b) -> (a + b, a - b), elementwise
__device__ __forceinline__ void bf2(float2& a, float2& b) {
  const float2 s = add2(a, b), d = sub2(a, b);
  a = s;
  b = d;
}
// butterfly inside one pair: (x, y) -> (x + y, x - y)
__device__ __forceinline__ void bf_in(float2& a) {
  const float s = a.x + a.y, d = a.x - a.y;
  a.x = s;
  a.y = d;
}

// Butterflies over the bits of an index into v[]: for every h = 1, 2, ..., N/2 pair (i, i + h).
template <int N>
__device__ __forceinline__ void bfly_all(float2 (&v)[N]) {
#pragma unroll
  for (int h = 1; h < N; h <<= 1)
#pragma unroll
    for (int i = 0; i < N; ++i)
      if ((i & h) == 0) bf2(v[i], v[i + h]);
}

// ---------------------------------------------------------------------------------------------
// TMEM (tensor memory) as per-thread storage: thread t of warp w owns lane 32*(w%4) + t.
__device__ __forceinline__ void tmem_alloc_512(uint32_t* smem_slot) {
  const uint32_t dst = static_cast<uint32_t>(__cvta_generic_to_shared(smem_slot));
  asm volatile("tcgen05.alloc.cta_group::1.sync.aligned.shared::cta.b32 [%0], 512;" ::"r"(dst) : "memory");
  asm volatile("tcgen05.relinquish_alloc_permit.cta_group::1.sync.aligned;" ::: "memory");
}
__device__ __forceinline__ void tmem_dealloc_512(uint32_t taddr) {
  asm volatile("tcgen05.dealloc.cta_group::1.sync.aligned.b32 %0, 512;" ::"r"(taddr) : "memory");
}
__device__ __forceinline__ void tmem_fence_before() { asm volatile("tcgen05.fence::before_thread_sync;" ::: "memory"); }
__device__ __forceinline__ void tmem_fence_after() { asm volatile("tcgen05.fence::after_thread_sync;" ::: "memory"); }
__device__ __forceinline__ void tmem_wait_ld() { asm volatile("tcgen05.wait::ld.sync.aligned;" ::: "memory"); }
__device__ __forceinline__ void tmem_wait_st() { asm volatile("tcgen05.wait::st.sync.aligned;" ::: "memory"); }

// 16 consecutive 32-bit columns of this thread's lane <-> registers
__device__ __forceinline__ void tmem_ld16(uint32_t ta, float (&r)[16]) {
  asm volatile("tcgen05.ld.sync.aligned.32x32b.x16.b32 {%0,%1,%2,%3,%4,%5,%6,%7,%8,%9,%10,%11,%12,%13,%14,%15}, [%16];"
               : "=f"(r[0]), "=f"(r[1]), "=f"(r[2]), "=f"(r[3]), "=f"(r[4]), "=f"(r[5]), "=f"(r[6]), "=f"(r[7]),
                 "=f"(r[8]), "=f"(r[9]), "=f"(r[10]), "=f"(r[11]), "=f"(r[12]), "=f"(r[13]), "=f"(r[14]), "=f"(r[15])
               : "r"(ta) : "memory");
}
__device__ __forceinline__ void tmem_st16(uint32_t ta, const float (&r)[16]) {
  asm volatile("tcgen05.st.sync.aligned.32x32b.x16.b32 [%0], {%1,%2,%3,%4,%5,%6,%7,%8,%9,%10,%11,%12,%13,%14,%15,%16};"
               ::"r"(ta), "f"(r[0]), "f"(r[1]), "f"(r[2]), "f"(r[3]), "f"(r[4]), "f"(r[5]), "f"(r[6]), "f"(r[7]),
                 "f"(r[8]), "f"(r[9]), "f"(r[10]), "f"(r[11]), "f"(r[12]), "f"(r[13]), "f"(r[14]), "f"(r[15])
               : "memory");
}

// ---------------------------------------------------------------------------------------------
// Asynchronous global -> shared copies (no registers held while in flight).
__device__ __forceinline__ void cp_async16(float* smem_dst, const void* gsrc) {
  const uint32_t s = static_cast<uint32_t>(__cvta_generic_to_shared(smem_dst));
  asm volatile("cp.async.cg.shared.global [%0], [%1], 16;" ::"r"(s), "l"(gsrc) : "memory");
}
__device__ __forceinline__ void cp_async_commit() { asm volatile("cp.async.commit_group;" ::: "memory"); }
// every copy this thread has issued, committed to a group or not (wait_group 0 passes over those that were not)
__device__ __forceinline__ void cp_async_wait_all() { asm volatile("cp.async.wait_all;" ::: "memory"); }

// Where row r of the plane group that starts at plane b0 lives in X / Y (planes of lv stored
// elements, back to back): its first element and how many of its 2^R elements are stored.
// Rows wholly in the padding get lim = 0 and the plane's first element (never accessed).
template <int R, int Q>
__device__ __forceinline__ void row_loc(long long b0, long long r, long long lv, long long* e0, int* lim) {
  const long long b = r >> Q, start = (r & ((1ll << Q) - 1)) << R;
  long long n = lv - start;
  n = n < 0 ? 0 : n > (1ll << R) ? (1ll << R) : n;
  *e0 = (b0 + b) * lv + (n > 0 ? start : 0);
  *lim = static_cast<int>(n);
}

// Issued before pdl_wait(): asks L2 for the X rows [rb, re) of the first plane group that this
// CTA's phase 1 reads, at most PREFETCH_BYTES of them, so that their HBM reads overlap the
// previous kernel's tail.  A cache hint only: L2 is the point of coherence, so a line fetched
// before the previous kernel's last writes to it still returns those writes.
constexpr long long PREFETCH_BYTES = 128 * 1024;
template <int D, int R, int Q>
__device__ __forceinline__ void l2_prefetch_first_rows(const void* src, long long rb, long long re, long long lv) {
  constexpr long long ES = D == DT_BF16 ? 2 : 4;
  const long long r = rb + threadIdx.x;
  if (r >= re || (r - rb) * (ES << R) >= PREFETCH_BYTES) return;
  long long e0;
  int lim;
  row_loc<R, Q>(0, r, lv, &e0, &lim);
  if (lim > 0)
    asm volatile("cp.async.bulk.prefetch.L2.global [%0], %1;" ::"l"(static_cast<const char*>(src) + e0 * ES),
                 "r"(static_cast<unsigned>(lim * ES))
                 : "memory");
}

}  // namespace fast
}  // namespace whtmix
