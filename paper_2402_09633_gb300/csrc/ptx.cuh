// Thin inline-PTX wrappers for sm_103a: mbarriers, bulk copies, tcgen05
// (TMEM allocation, MMA, commit, TMEM loads/stores, fences) and a bounded
// wait helper.  Every spin in this library goes through bounded_wait(), which
// gives up after a wall-clock limit, records an error code and lets the
// caller unwind instead of hanging the GPU.
#pragma once
#include <cstdint>
#include <cuda_bf16.h>

namespace gnn {

// Device-side error bits (OR-ed into the context's error word).
enum : uint32_t {
  DEV_ERR_INDEX_RANGE = 1u,   // an edge endpoint was outside [0, n_nodes)
  DEV_ERR_TIMEOUT     = 2u,   // a bounded wait expired (pipeline stalled)
  DEV_ERR_CAPACITY    = 4u,   // an output buffer was too small (graph building)
};

__device__ __forceinline__ uint32_t smem_u32(const void* p) {
  return static_cast<uint32_t>(__cvta_generic_to_shared(p));
}

__device__ __forceinline__ uint64_t global_timer_ns() {
  uint64_t t;
  asm volatile("mov.u64 %0, %%globaltimer;" : "=l"(t));
  return t;
}

// ---------------------------------------------------------------- mbarrier
__device__ __forceinline__ void mbar_init(uint64_t* bar, uint32_t count) {
  asm volatile("mbarrier.init.shared::cta.b64 [%0], %1;" ::"r"(smem_u32(bar)), "r"(count) : "memory");
}
__device__ __forceinline__ void fence_mbar_init() {
  asm volatile("fence.mbarrier_init.release.cluster;" ::: "memory");
}
__device__ __forceinline__ void mbar_arrive(uint64_t* bar) {
  asm volatile("mbarrier.arrive.release.cta.shared::cta.b64 _, [%0];" ::"r"(smem_u32(bar)) : "memory");
}
__device__ __forceinline__ void mbar_arrive_expect_tx(uint64_t* bar, uint32_t bytes) {
  asm volatile("mbarrier.arrive.expect_tx.release.cta.shared::cta.b64 _, [%0], %1;"
               ::"r"(smem_u32(bar)), "r"(bytes) : "memory");
}
__device__ __forceinline__ bool mbar_try_wait(uint64_t* bar, uint32_t parity) {
  uint32_t ok;
  asm volatile(
      "{\n\t.reg .pred p;\n\t"
      "mbarrier.try_wait.parity.acquire.cta.shared::cta.b64 p, [%1], %2;\n\t"
      "selp.u32 %0, 1, 0, p;\n\t}\n"
      : "=r"(ok) : "r"(smem_u32(bar)), "r"(parity) : "memory");
  return ok != 0;
}

// Non-blocking probe of the completion of the phase with `parity`.
__device__ __forceinline__ bool mbar_test_wait(uint64_t* bar, uint32_t parity) {
  uint32_t ok;
  asm volatile(
      "{\n\t.reg .pred p;\n\t"
      "mbarrier.test_wait.parity.acquire.cta.shared::cta.b64 p, [%1], %2;\n\t"
      "selp.u32 %0, 1, 0, p;\n\t}\n"
      : "=r"(ok) : "r"(smem_u32(bar)), "r"(parity) : "memory");
  return ok != 0;
}

// True on every lane when x is true on all of them (the result is uniform across the warp).
__device__ __forceinline__ bool warp_all(bool x) { return __all_sync(0xffffffffu, x); }
// A value that is the same on every lane, as one the compiler may keep in a uniform register.
__device__ __forceinline__ int uniform(int x) { return __shfl_sync(0xffffffffu, x, 0); }
// True on one lane of a converged warp.
__device__ __forceinline__ bool elect_one() {
  uint32_t ok;
  asm volatile(
      "{\n\t.reg .pred p;\n\t"
      "elect.sync _|p, 0xffffffff;\n\t"
      "selp.u32 %0, 1, 0, p;\n\t}\n"
      : "=r"(ok));
  return ok != 0;
}

// Wall-clock limit of every wait in the library (ns).
constexpr uint64_t kWaitLimitNs = 2000000000ull;   // 2 s

// Waits until the mbarrier phase with `parity` completed, or until `*abort`
// becomes non-zero, or until `limit_ns` expires (then records DEV_ERR_TIMEOUT
// in *err and sets *abort).  Returns true when the phase completed.
__device__ __forceinline__ bool bounded_wait(uint64_t* bar, uint32_t parity, volatile int* abort, uint32_t* err,
                                             uint64_t limit_ns = kWaitLimitNs) {
  if (mbar_try_wait(bar, parity)) return true;
  const uint64_t t0 = global_timer_ns();
  for (uint32_t it = 0;; ++it) {
    if (mbar_try_wait(bar, parity)) return true;
    if (*abort) return false;
    if ((it & 63u) == 63u && global_timer_ns() - t0 > limit_ns) {
      atomicOr(err, DEV_ERR_TIMEOUT);
      *abort = 1;
      return false;
    }
  }
}

// Teardown wait for this thread's own asynchronous work (a copy or an MMA commit) after the pipeline
// may have aborted: ignores the abort flag, records nothing, and gives up after `limit_ns`.
__device__ __forceinline__ void drain_wait(uint64_t* bar, uint32_t parity, uint64_t limit_ns = 20000000ull) {
  if (mbar_try_wait(bar, parity)) return;
  const uint64_t t0 = global_timer_ns();
  for (uint32_t it = 0;; ++it) {
    if (mbar_try_wait(bar, parity)) return;
    if ((it & 63u) == 63u && global_timer_ns() - t0 > limit_ns) return;
  }
}

// ------------------------------------------------------------- bulk copies
// global -> shared, completion counted in bytes on `bar`.
__device__ __forceinline__ void bulk_g2s(void* smem_dst, const void* gsrc, uint32_t bytes, uint64_t* bar) {
  asm volatile(
      "cp.async.bulk.shared::cluster.global.mbarrier::complete_tx::bytes [%0], [%1], %2, [%3];"
      ::"r"(smem_u32(smem_dst)), "l"(gsrc), "r"(bytes), "r"(smem_u32(bar)) : "memory");
}
__device__ __forceinline__ void prefetch_l2_bulk(const void* gsrc, uint32_t bytes) {
  asm volatile("cp.async.bulk.prefetch.L2.global [%0], %1;" ::"l"(gsrc), "r"(bytes) : "memory");
}

// ------------------------------------------------------------------ tcgen05
__device__ __forceinline__ void tmem_alloc(uint32_t* smem_dst, uint32_t ncols) {
  asm volatile("tcgen05.alloc.cta_group::1.sync.aligned.shared::cta.b32 [%0], %1;"
               ::"r"(smem_u32(smem_dst)), "r"(ncols) : "memory");
}
__device__ __forceinline__ void tmem_relinquish() {
  asm volatile("tcgen05.relinquish_alloc_permit.cta_group::1.sync.aligned;" ::: "memory");
}
__device__ __forceinline__ void tmem_dealloc(uint32_t taddr, uint32_t ncols) {
  asm volatile("tcgen05.dealloc.cta_group::1.sync.aligned.b32 %0, %1;" ::"r"(taddr), "r"(ncols) : "memory");
}
__device__ __forceinline__ void tc_fence_before() {
  asm volatile("tcgen05.fence::before_thread_sync;" ::: "memory");
}
__device__ __forceinline__ void tc_fence_after() {
  asm volatile("tcgen05.fence::after_thread_sync;" ::: "memory");
}

// D[tmem] (+)= A[tmem] * B[smem]^T, kind::f16 (bf16 inputs, fp32 accumulate).
__device__ __forceinline__ void mma_bf16_ts(uint32_t d_tmem, uint32_t a_tmem, uint64_t b_desc,
                                            uint32_t idesc, uint32_t accumulate) {
  asm volatile(
      "{\n\t.reg .pred p;\n\t"
      "setp.ne.b32 p, %4, 0;\n\t"
      "tcgen05.mma.cta_group::1.kind::f16 [%0], [%1], %2, %3, p;\n\t}\n"
      ::"r"(d_tmem), "r"(a_tmem), "l"(b_desc), "r"(idesc), "r"(accumulate) : "memory");
}
// The same with A in shared memory.
__device__ __forceinline__ void mma_bf16_ss(uint32_t d_tmem, uint64_t a_desc, uint64_t b_desc, uint32_t idesc,
                                            uint32_t accumulate) {
  asm volatile(
      "{\n\t.reg .pred p;\n\t"
      "setp.ne.b32 p, %4, 0;\n\t"
      "tcgen05.mma.cta_group::1.kind::f16 [%0], %1, %2, %3, p;\n\t}\n"
      ::"r"(d_tmem), "l"(a_desc), "l"(b_desc), "r"(idesc), "r"(accumulate) : "memory");
}
// Arrive once on `bar` when every tcgen05 op issued so far by this thread completed.
__device__ __forceinline__ void mma_commit(uint64_t* bar) {
  asm volatile("tcgen05.commit.cta_group::1.mbarrier::arrive::one.shared::cluster.b64 [%0];"
               ::"r"(smem_u32(bar)) : "memory");
}

// 16 lanes x 32 columns of 32-bit: thread t receives, for each 8-column block b, in v[2b] lane t/4's
// columns 8b + 2(t%4) and + 1, and in v[2b + 1] the same columns of lane t/4 + 8.  The values are
// defined only after tmem_ld_wait(v) on the same array.
__device__ __forceinline__ void tmem_ld_16x32(uint32_t taddr, float2* v) {
  asm volatile(
      "tcgen05.ld.sync.aligned.16x256b.x4.b32 "
      "{%0,%1,%2,%3,%4,%5,%6,%7,%8,%9,%10,%11,%12,%13,%14,%15}, [%16];"
      : "=f"(v[0].x), "=f"(v[0].y), "=f"(v[1].x), "=f"(v[1].y), "=f"(v[2].x), "=f"(v[2].y),
        "=f"(v[3].x), "=f"(v[3].y), "=f"(v[4].x), "=f"(v[4].y), "=f"(v[5].x), "=f"(v[5].y),
        "=f"(v[6].x), "=f"(v[6].y), "=f"(v[7].x), "=f"(v[7].y)
      : "r"(taddr));
}
// Waits for this thread's tensor-memory loads; the array's values depend on the wait.
__device__ __forceinline__ void tmem_ld_wait(float2* v) {
  asm volatile("tcgen05.wait::ld.sync.aligned;"
               : "+f"(v[0].x), "+f"(v[0].y), "+f"(v[1].x), "+f"(v[1].y), "+f"(v[2].x), "+f"(v[2].y),
                 "+f"(v[3].x), "+f"(v[3].y), "+f"(v[4].x), "+f"(v[4].y), "+f"(v[5].x), "+f"(v[5].y),
                 "+f"(v[6].x), "+f"(v[6].y), "+f"(v[7].x), "+f"(v[7].y)
               :
               : "memory");
}
// 16 lanes x 32 columns of 32-bit, in the layout of tmem_ld_16x32.
__device__ __forceinline__ void tmem_st_16x32(uint32_t taddr, const float2* v) {
  asm volatile(
      "tcgen05.st.sync.aligned.16x256b.x4.b32 "
      "[%0], {%1,%2,%3,%4,%5,%6,%7,%8,%9,%10,%11,%12,%13,%14,%15,%16};"
      ::"r"(taddr), "f"(v[0].x), "f"(v[0].y), "f"(v[1].x), "f"(v[1].y), "f"(v[2].x), "f"(v[2].y), "f"(v[3].x),
        "f"(v[3].y), "f"(v[4].x), "f"(v[4].y), "f"(v[5].x), "f"(v[5].y), "f"(v[6].x), "f"(v[6].y),
        "f"(v[7].x), "f"(v[7].y)
      : "memory");
}
// 16 lanes x 16 columns of packed words: thread t supplies, for each 4-column block b, in r[2b] lane
// t/4's column 4b + t%4 and in r[2b + 1] the same column of lane t/4 + 8.
__device__ __forceinline__ void tmem_st_16x16(uint32_t taddr, const uint32_t* r) {
  asm volatile(
      "tcgen05.st.sync.aligned.16x128b.x4.b32 [%0], {%1,%2,%3,%4,%5,%6,%7,%8};"
      ::"r"(taddr), "r"(r[0]), "r"(r[1]), "r"(r[2]), "r"(r[3]), "r"(r[4]), "r"(r[5]), "r"(r[6]), "r"(r[7])
      : "memory");
}
__device__ __forceinline__ void tmem_st_wait() {
  asm volatile("tcgen05.wait::st.sync.aligned;" ::: "memory");
}

// Programmatic dependent launch: the executing thread waits until every grid this one depends on has
// completed and its memory writes are visible (it returns at once when the kernel was not launched
// as a programmatic dependent).  Everything a kernel does before it may overlap the previous kernel,
// so it must touch no data that kernel writes or reads.  Without a trigger a dependent launches as its
// predecessor's CTAs exit, which hides the launch latency.
__device__ __forceinline__ void pdl_wait() { asm volatile("griddepcontrol.wait;" ::: "memory"); }
// Lets the next kernel's CTAs launch as soon as every CTA of this one has called it (after its own
// pdl_wait), where SMs are free; they set up (weights, tensor memory, barriers) and wait.  Worth it only
// when this grid leaves SMs idle: tiny event (57 CTAs) 120 -> 114 us, 3,000 hits / 9,000 edges 195 -> 188; with
// tile kernels that fill every SM it made the full event's step slower (6.51 -> 6.83 ms, an earlier form of
// the kernels) and the mid event's (716 -> 726 us).
__device__ __forceinline__ void pdl_trigger() { asm volatile("griddepcontrol.launch_dependents;" ::: "memory"); }
__device__ __forceinline__ void pdl_trigger_small() {
  if (gridDim.x <= 64) pdl_trigger();
}

// ------------------------------------------------- 32-byte global accesses
// One 32-byte sector per thread (256-bit accesses, sm_100 and later; the address is 32-byte aligned).
// KEEP false: the line will not be wanted in L1 again.
template <bool KEEP = true>
__device__ __forceinline__ void ld_global_32b(const void* p, uint32_t* r) {
  if constexpr (KEEP)
    asm volatile("ld.global.v8.b32 {%0,%1,%2,%3,%4,%5,%6,%7}, [%8];"
                 : "=r"(r[0]), "=r"(r[1]), "=r"(r[2]), "=r"(r[3]), "=r"(r[4]), "=r"(r[5]), "=r"(r[6]), "=r"(r[7])
                 : "l"(p)
                 : "memory");
  else
    asm volatile("ld.global.L1::no_allocate.v8.b32 {%0,%1,%2,%3,%4,%5,%6,%7}, [%8];"
                 : "=r"(r[0]), "=r"(r[1]), "=r"(r[2]), "=r"(r[3]), "=r"(r[4]), "=r"(r[5]), "=r"(r[6]), "=r"(r[7])
                 : "l"(p)
                 : "memory");
}
__device__ __forceinline__ void st_global_32b(void* p, const uint32_t* r) {
  asm volatile("st.global.v8.b32 [%0], {%1,%2,%3,%4,%5,%6,%7,%8};"
               ::"l"(p), "r"(r[0]), "r"(r[1]), "r"(r[2]), "r"(r[3]), "r"(r[4]), "r"(r[5]), "r"(r[6]), "r"(r[7])
               : "memory");
}

// ------------------------------------------------------- operand encodings
// Shared-memory matrix descriptor (tcgen05 format): K-major, 128-byte swizzle,
// 8-row core groups 1024 bytes apart.  `saddr` must lie in a 1024-byte aligned
// swizzle atom (it may be offset by a multiple of 32 bytes inside the 128-byte
// row to select a K step).
__device__ __forceinline__ uint64_t sdesc_kmajor_sw128(uint32_t saddr) {
  uint64_t d = 0;
  d |= (uint64_t)((saddr >> 4) & 0x3FFFu);          // start address
  d |= (uint64_t)(1u) << 16;                         // leading byte offset (unused for SW128 K-major)
  d |= (uint64_t)(1024u >> 4) << 32;                 // stride byte offset: 8 rows x 128 B
  d |= (uint64_t)1u << 46;                           // descriptor version for tcgen05
  d |= (uint64_t)2u << 61;                           // layout: 128-byte swizzle
  return d;
}

// The same without a swizzle, for a tile of 16 K elements (one K step): 8-row x 16-byte core matrices,
// the two of a row group 128 bytes apart (leading byte offset, along K), row groups 256 bytes apart
// (stride byte offset).
__device__ __forceinline__ uint64_t sdesc_kmajor_plain(uint32_t saddr) {
  return (uint64_t)((saddr >> 4) & 0x3FFFu) | (uint64_t)(128u >> 4) << 16 | (uint64_t)(256u >> 4) << 32 |
         (uint64_t)1u << 46;
}

// Instruction descriptor, kind::f16: A = B = bf16, D = f32, both K-major, M x N.
__host__ __device__ constexpr uint32_t idesc_bf16_f32(uint32_t M, uint32_t N) {
  return (1u << 4)            // D format f32
       | (1u << 7)            // A format bf16
       | (1u << 10)           // B format bf16
       | ((N >> 3) << 17)     // N / 8
       | ((M >> 4) << 24);    // M / 16
}

// fp32 pair -> (hi, lo) bf16x2 words with hi + lo ~= v to ~16 mantissa bits.
__device__ __forceinline__ void split_bf16x2(float2 v, uint32_t& hi, uint32_t& lo) {
  const __nv_bfloat162 h = __floats2bfloat162_rn(v.x, v.y);
  hi = *reinterpret_cast<const uint32_t*>(&h);
  const float2 r = __fadd2_rn(v, make_float2(-__uint_as_float(hi << 16), -__uint_as_float(hi & 0xffff0000u)));
  const __nv_bfloat162 l = __floats2bfloat162_rn(r.x, r.y);
  lo = *reinterpret_cast<const uint32_t*>(&l);
}
__device__ __forceinline__ uint32_t pack_bf16x2(float a, float b) {
  __nv_bfloat162 h = __floats2bfloat162_rn(a, b);
  return *reinterpret_cast<uint32_t*>(&h);
}

}  // namespace gnn
