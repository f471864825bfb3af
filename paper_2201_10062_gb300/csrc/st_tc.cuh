// Building blocks of the tensor-core (tcgen05) kernels: shared-memory matrix descriptors, MMA issue,
// bounded mbarrier waits, tensor-memory loads and stores, bulk copies, the fp16 hi + lo split and
// the float32 symbol of the preconditioner.
#pragma once

#include <cuda_fp16.h>

#include "st_internal.cuh"
#include "st_symbol.cuh"

namespace st {
namespace {

constexpr int kTN = 32;          // spatial columns per tile (MMA N)
constexpr int kM = 128;          // MMA M (rows of S of one parity, zero padded)
constexpr float kSScale = 8.0f;  // S is stored times 8
constexpr int kSpinLimit = 1 << 20;  // bounded mbarrier wait

__device__ __forceinline__ uint32_t smem_u32(const void *p) {
  return (uint32_t)__cvta_generic_to_shared(p);
}

// byte offset of element (row, k) in a K-major, no-swizzle canonical operand with K columns
__host__ __device__ __forceinline__ uint32_t canon_off(int row, int k, int K) {
  return (uint32_t)((((row >> 3) * (K >> 3) + (k >> 3)) << 7) + ((row & 7) << 4) + ((k & 7) << 1));
}

// shared-memory matrix descriptor: start address, leading-dimension byte offset (between
// core matrices along K) = 128, stride byte offset (between 8-row groups) = 16 K bytes,
// descriptor version 1, no swizzle
__device__ __forceinline__ uint64_t make_desc(uint32_t saddr, int K) {
  const uint64_t lbo = 128, sbo = (uint64_t)K * 16;
  uint64_t d = 0;
  d |= (uint64_t)((saddr >> 4) & 0x3FFF);
  d |= (uint64_t)((lbo >> 4) & 0x3FFF) << 16;
  d |= (uint64_t)((sbo >> 4) & 0x3FFF) << 32;
  d |= (uint64_t)1 << 46;
  return d;
}

// kind::f16, D f32, A (tensor memory) and B (shared memory) f16, both K-major, M = 128
template <int N>
__device__ __forceinline__ void mma_ta(uint32_t dtmem, uint32_t atmem, uint64_t bd, uint32_t acc) {
  constexpr uint32_t idesc = (1u << 4) | ((uint32_t)(N >> 3) << 17) | ((uint32_t)(kM >> 4) << 24);
  asm volatile(
      "{\n\t.reg .pred p;\n\t"
      "setp.ne.b32 p, %4, 0;\n\t"
      "tcgen05.mma.cta_group::1.kind::f16 [%0], [%1], %2, %3, p;\n\t}\n" ::"r"(dtmem),
      "r"(atmem), "l"(bd), "r"(idesc), "r"(acc));
}

__device__ __forceinline__ void mma_commit(uint32_t mbar) {
  asm volatile("tcgen05.commit.cta_group::1.mbarrier::arrive::one.shared::cluster.b64 [%0];" ::"r"(
                   mbar)
               : "memory");
}

// one lane of a converged warp.  The compiler knows a region under elect.sync to run in a single
// thread, and a tcgen05.mma then takes fewer instructions to issue than under `lane == 0`
// (k_time_tcd at 255^2 x 256: 763 against 617 us a time stage).
__device__ __forceinline__ bool elect_one() {
  uint32_t p;
  asm volatile(
      "{\n\t.reg .pred P;\n\t"
      "elect.sync _|P, 0xffffffff;\n\t"
      "selp.u32 %0, 1, 0, P;\n\t}"
      : "=r"(p));
  return p != 0;
}

// bounded wait for a phase; each try may suspend the thread for up to a microsecond, so that a warp
// that waits for another role does not take its issue slots
__device__ __forceinline__ bool mbar_wait(uint32_t mbar, uint32_t phase) {
  for (int it = 0; it < kSpinLimit; ++it) {
    uint32_t done;
    asm volatile(
        "{\n\t.reg .pred p;\n\t"
        "mbarrier.try_wait.parity.shared::cta.b64 p, [%1], %2, %3;\n\t"
        "selp.u32 %0, 1, 0, p;\n\t}\n"
        : "=r"(done)
        : "r"(mbar), "r"(phase), "r"(1000u)
        : "memory");
    if (done) return true;
  }
  return false;
}

__device__ __forceinline__ void mbar_arrive(uint32_t mbar) {
  asm volatile("mbarrier.arrive.shared::cta.b64 _, [%0];" ::"r"(mbar) : "memory");
}

// 16 columns of this warp's 32 lanes into registers; the values are valid only after
// tmem_wait_ld (several loads may be in flight)
__device__ __forceinline__ void tmem_ld16_async(uint32_t taddr, uint32_t (&r)[16]) {
  asm volatile(
      "tcgen05.ld.sync.aligned.32x32b.x16.b32 {%0,%1,%2,%3,%4,%5,%6,%7,%8,%9,%10,%11,%12,%13,%14,"
      "%15}, [%16];"
      : "=r"(r[0]), "=r"(r[1]), "=r"(r[2]), "=r"(r[3]), "=r"(r[4]), "=r"(r[5]), "=r"(r[6]),
        "=r"(r[7]), "=r"(r[8]), "=r"(r[9]), "=r"(r[10]), "=r"(r[11]), "=r"(r[12]), "=r"(r[13]),
        "=r"(r[14]), "=r"(r[15])
      : "r"(taddr));
}
__device__ __forceinline__ void tmem_wait_ld() {
  asm volatile("tcgen05.wait::ld.sync.aligned;" ::: "memory");
}

__device__ __forceinline__ void tmem_ld16(uint32_t taddr, float *v) {
  uint32_t r[16];
  asm volatile(
      "tcgen05.ld.sync.aligned.32x32b.x16.b32 {%0,%1,%2,%3,%4,%5,%6,%7,%8,%9,%10,%11,%12,%13,%14,"
      "%15}, [%16];"
      : "=r"(r[0]), "=r"(r[1]), "=r"(r[2]), "=r"(r[3]), "=r"(r[4]), "=r"(r[5]), "=r"(r[6]),
        "=r"(r[7]), "=r"(r[8]), "=r"(r[9]), "=r"(r[10]), "=r"(r[11]), "=r"(r[12]), "=r"(r[13]),
        "=r"(r[14]), "=r"(r[15])
      : "r"(taddr));
  asm volatile("tcgen05.wait::ld.sync.aligned;" ::: "memory");
#pragma unroll
  for (int i = 0; i < 16; ++i) v[i] = __uint_as_float(r[i]);
}

__device__ __forceinline__ void fence_before() {
  asm volatile("tcgen05.fence::before_thread_sync;" ::: "memory");
}
__device__ __forceinline__ void fence_after() {
  asm volatile("tcgen05.fence::after_thread_sync;" ::: "memory");
}
__device__ __forceinline__ void fence_async_smem() {
  asm volatile("fence.proxy.async.shared::cta;" ::: "memory");
}


// End of a tensor-core block: after a timeout (ok false), one more bounded wait on each commit
// barrier whose last wait ran out (pendN, waited with phase phN).  Tensor memory is released only
// when every MMA batch has completed and no other asynchronous copy is left in flight
// (copies_done, uniform); otherwise the block records that it keeps it.  The decision is uniform
// across the block (one __syncthreads_and); warp 0 releases COLS columns at tmem.
template <int COLS>
__device__ __forceinline__ void tc_release_cols(bool ok, bool pend1, uint32_t mbar1, uint32_t ph1,
                                                bool pend2, uint32_t mbar2, uint32_t ph2,
                                                uint32_t tmem, State *S, bool copies_done = true) {
  // every thread that saw a timeout waits (bounded) on the barriers that still owe a completion;
  // the results are combined over the whole block (ok may differ between the tile pipelines of
  // one block), so that every thread takes the same decision
  bool d = true;
  if (!ok) {
    d = copies_done;
    if (pend1) d = mbar_wait(mbar1, ph1) && d;
    if (pend2) d = mbar_wait(mbar2, ph2) && d;
  }
  const bool drained = __syncthreads_and(d ? 1 : 0) != 0;
  const bool failed = __syncthreads_or(ok ? 0 : 1) != 0;
  if (failed && threadIdx.x == 0) {
    S->status = ST_ERR_TIMEOUT;
    if (!drained) atomicExch(&S->tmem_held, 1);
  }
  fence_before();
  __syncthreads();
  if (drained && (threadIdx.x >> 5) == 0) {
    fence_after();
    asm volatile("tcgen05.dealloc.cta_group::1.sync.aligned.b32 %0, %1;" ::"r"(tmem), "n"(COLS)
                 : "memory");
  }
}

// fp16 (hi, lo) pieces of two floats, packed as half2 words
__device__ __forceinline__ void split_h2(float a, float b, uint32_t &hi, uint32_t &lo) {
  const __half2 h = __floats2half2_rn(a, b);
  const float2 f = __half22float2(h);
  const __half2 l = __floats2half2_rn(a - f.x, b - f.y);
  hi = *reinterpret_cast<const uint32_t *>(&h);
  lo = *reinterpret_cast<const uint32_t *>(&l);
}

// Per-row (time frequency k) constants of 1/p(k, tau mu), hoisted out of the column loop.
struct SymRow {
  float a, b, c;
};

__device__ __forceinline__ SymRow sym_row(const Spec<float> &sp, int k) {
  SymRow r;
  const float hk = sp.hk[k - 1], ck = sp.ck[k - 1], sk = sp.sk[k - 1];
  if (sp.prec == ST_PREC_PTHETA) {
    r.a = sp.lh[k - 1];
    r.b = sp.lht[k - 1];
    r.c = 0.f;
  } else if (sp.scheme == ST_THETA) {
    r.a = hk;
    r.b = sp.theta + (1.0f - sp.theta) * ck;
    r.c = sk;
  } else {
    r.a = hk * hk;
    r.b = 1.0f;
    r.c = -sk * (1.0f + hk);
  }
  return r;
}

__device__ __forceinline__ void tmem_st8(uint32_t taddr, const uint32_t (&r)[8]) {
  asm volatile(
      "tcgen05.st.sync.aligned.32x32b.x8.b32 [%0], {%1,%2,%3,%4,%5,%6,%7,%8};" ::"r"(taddr),
      "r"(r[0]), "r"(r[1]), "r"(r[2]), "r"(r[3]), "r"(r[4]), "r"(r[5]), "r"(r[6]), "r"(r[7])
      : "memory");
}

// barrier of the `nthreads` threads of named barrier `id`
__device__ __forceinline__ void group_sync(int id, int nthreads) {
  asm volatile("bar.sync %0, %1;" ::"r"(id), "r"(nthreads) : "memory");
}

// barrier that also returns whether v holds in every participating thread
__device__ __forceinline__ bool group_sync_and(bool v, int id, int nthreads) {
  uint32_t out;
  asm volatile(
      "{\n\t.reg .pred p, q;\n\t"
      "setp.ne.b32 q, %1, 0;\n\t"
      "bar.red.and.pred p, %2, %3, q;\n\t"
      "selp.u32 %0, 1, 0, p;\n\t}"
      : "=r"(out)
      : "r"((uint32_t)v), "r"(id), "r"(nthreads)
      : "memory");
  return out != 0;
}

__device__ __forceinline__ void mbar_expect_tx(uint32_t mbar, uint32_t bytes) {
  asm volatile("mbarrier.arrive.expect_tx.shared::cta.b64 _, [%0], %1;" ::"r"(mbar), "r"(bytes)
               : "memory");
}

// tau mu_j of padded column j (x fastest, px = mx + 1 slots a row, m columns in all): the padding
// slots hold zeros, and get a factor that keeps them zero
__device__ __forceinline__ float tmu_col(const Spec<float> &sp, long long j, int mx, int px,
                                         long long m) {
  const unsigned row = (unsigned)j / (unsigned)px, jx = (unsigned)j - row * (unsigned)px;
  return (j < m && (int)jx < mx) ? sp.mux[jx] + sp.muy[row] : 1.0f;
}

}  // namespace
}  // namespace st
