// What the TMA-fed tensor-core transforms share (st_dst_tma.cu, st_dst_long.cu): tensor copies and
// their maps, the operand split, MMA issue, the copy of A into tensor memory, the symbol.
#pragma once

#include <cuda.h>

#include <cmath>

#include "st_tc.cuh"

namespace st {
namespace {

__device__ __forceinline__ uint64_t make_desc_sbo(uint32_t saddr, uint32_t sbo) {
  uint64_t d = 0;
  d |= (uint64_t)((saddr >> 4) & 0x3FFF);
  d |= (uint64_t)(128u >> 4) << 16;
  d |= (uint64_t)((sbo >> 4) & 0x3FFF) << 32;
  d |= (uint64_t)1 << 46;
  return d;
}

// MMAs of one operand pair over KS (at most MAXK) K steps, into two accumulators of N columns at d and
// d + N, which the epilogue adds: A_hi at a in tensor memory, A_lo vc columns further; B_hi at
// descriptor b, B_lo (adjacent along N) at b + lo.
// An MMA adds its K step to the accumulator with the sum cut off, not rounded, at float32's last bit,
// and so takes half an ulp off it on average: one accumulator for all K steps left the two transforms
// of a time stage short by 1e-6 (n = 256) to 2e-6 (n = 500) of the result, up to four times the error
// of the float32 kernels.  So the K steps go half and half to the two accumulators, whose sum is
// rounded, and the small products (A_hi B_lo, A_lo B_hi: 2^-11 of the large ones, and cut off that much
// lower) come before the large ones of the second; axes beyond 256 take two pairs.  Against float64 the
// root mean square and the largest error are then 0.95 of the float32 kernels' in the geometric mean
// over 510 sizes, schemes and inputs.  In the first half A_hi meets B_hi and B_lo in one MMA of twice the width.
// What this costs is the issue of the further MMAs (time stage at 255^2 x 256: 53.4 us with one
// accumulator and 55.4 now; 511 x 127 x 365: 80.7 and 84.3 a launch; y at 511^2 x 128: 77 and 80), so the
// conditions and operands of a step are shared where two pairs go together (pair after pair, the time
// stage took 57 and 90 us).  keep: 0 overwrites the accumulators, 1 adds to them.
template <int N, int MAXK>
__device__ __forceinline__ void issue_pair(uint32_t d, uint32_t a, uint32_t vc, uint64_t b, uint64_t lo,
                                           int KS, uint32_t keep) {
  const int K2 = (KS + 1) >> 1;
#pragma unroll
  for (int ks = 0; ks < (MAXK + 1) / 2; ++ks)
    if (ks < K2) mma_ta<2 * N>(d, a + 8u * ks, b + 16u * (uint64_t)ks, ks > 0 ? 1u : keep);
#pragma unroll
  for (int ks = 0; ks < MAXK; ++ks) {
    if (ks < KS) mma_ta<N>(d + N, a + vc + 8u * ks, b + 16u * (uint64_t)ks, 1u);
    if (ks >= K2 && ks < KS) mma_ta<N>(d + N, a + 8u * ks, b + lo + 16u * (uint64_t)ks, 1u);
  }
#pragma unroll
  for (int ks = 1; ks < MAXK; ++ks)
    if (ks >= K2 && ks < KS) mma_ta<N>(d + N, a + 8u * ks, b + 16u * (uint64_t)ks, 1u);
}
// Two such pairs in turns, of KS and KS1 (KS, or one less) steps.
template <int N, int MAXK>
__device__ __forceinline__ void issue_two_pairs(uint32_t d0, uint32_t d1, uint32_t a0, uint32_t a1,
                                                uint32_t vc, uint64_t b0, uint64_t b1, uint64_t lo,
                                                int KS, int KS1) {
  const int K2 = (KS + 1) >> 1;
#pragma unroll
  for (int ks = 0; ks < (MAXK + 1) / 2; ++ks)
    if (ks < K2) {
      mma_ta<2 * N>(d0, a0 + 8u * ks, b0 + 16u * (uint64_t)ks, ks > 0 ? 1u : 0u);
      mma_ta<2 * N>(d1, a1 + 8u * ks, b1 + 16u * (uint64_t)ks, ks > 0 ? 1u : 0u);
    }
#pragma unroll
  for (int ks = 0; ks < MAXK; ++ks) {
    if (ks < KS) {
      mma_ta<N>(d0 + N, a0 + vc + 8u * ks, b0 + 16u * (uint64_t)ks, 1u);
      if (ks < KS1) mma_ta<N>(d1 + N, a1 + vc + 8u * ks, b1 + 16u * (uint64_t)ks, 1u);
    }
    if (ks >= K2 && ks < KS) {
      mma_ta<N>(d0 + N, a0 + 8u * ks, b0 + lo + 16u * (uint64_t)ks, 1u);
      if (ks < KS1) mma_ta<N>(d1 + N, a1 + 8u * ks, b1 + lo + 16u * (uint64_t)ks, 1u);
    }
  }
#pragma unroll
  for (int ks = 1; ks < MAXK; ++ks)
    if (ks >= K2 && ks < KS) {
      mma_ta<N>(d0 + N, a0 + 8u * ks, b0 + 16u * (uint64_t)ks, 1u);
      if (ks < KS1) mma_ta<N>(d1 + N, a1 + 8u * ks, b1 + 16u * (uint64_t)ks, 1u);
    }
}

// A into tensor memory: variant (slot or block's own rows, piece) at columns variant * hK / 2, from the host image
// [variant][hK / 16][128 rows][16 halves]; `nw` warps of the block share the work
__device__ __forceinline__ void load_a_variants(const uint4 *img, int nv, int hK, uint32_t a_base,
                                                int warp, int nw, int lane) {
  const int q = warp & 3, nq = (nw - q + 3) / 4, KS = hK >> 4, cnt = nv * KS;
  const uint32_t lanes = (uint32_t)(q * 32) << 16;
  // four pieces' loads in flight before the first store: one at a time, the latency of eight loads in
  // a row was 4 of a 30 us launch
  for (int i0 = warp >> 2; i0 < cnt; i0 += 4 * nq) {
    uint4 c[4][2];
#pragma unroll
    for (int k = 0; k < 4; ++k) {
      const int i = i0 + k * nq;
      if (i < cnt) {
        const uint4 *p = img + ((size_t)i * kM + (size_t)(q * 32 + lane)) * 2;
        c[k][0] = __ldg(p);
        c[k][1] = __ldg(p + 1);
      }
    }
#pragma unroll
    for (int k = 0; k < 4; ++k) {
      const int i = i0 + k * nq;
      if (i < cnt) {
        const uint32_t w[8] = {c[k][0].x, c[k][0].y, c[k][0].z, c[k][0].w,
                               c[k][1].x, c[k][1].y, c[k][1].z, c[k][1].w};
        const int v = i / KS, ks = i - v * KS;
        tmem_st8(a_base + lanes + (uint32_t)(v * (hK >> 1) + ks * 8), w);
      }
    }
  }
  asm volatile("tcgen05.wait::st.sync.aligned;" ::: "memory");
}

// ---------------------------------------------------------------- tensor copies
__device__ __forceinline__ void tma_load3(uint32_t dst, const CUtensorMap *map, int x, int y, int z,
                                          uint32_t mbar) {
  asm volatile(
      "cp.async.bulk.tensor.3d.shared::cluster.global.mbarrier::complete_tx::bytes [%0], [%1, {%2, "
      "%3, %4}], [%5];" ::"r"(dst),
      "l"(map), "r"(x), "r"(y), "r"(z), "r"(mbar)
      : "memory");
}
__device__ __forceinline__ void tma_store3(const CUtensorMap *map, uint32_t src, int x, int y,
                                           int z) {
  asm volatile(
      "cp.async.bulk.tensor.3d.global.shared::cta.bulk_group [%0, {%1, %2, %3}], [%4];" ::"l"(map),
      "r"(x), "r"(y), "r"(z), "r"(src)
      : "memory");
}
__device__ __forceinline__ void bulk_commit() {
  asm volatile("cp.async.bulk.commit_group;" ::: "memory");
}
// this thread's stores have read their shared memory / are complete
__device__ __forceinline__ void bulk_wait_read() {
  asm volatile("cp.async.bulk.wait_group.read 0;" ::: "memory");
}
__device__ __forceinline__ void bulk_wait_done() {
  asm volatile("cp.async.bulk.wait_group 0;" ::: "memory");
}

__device__ __forceinline__ float4 lds4(uint32_t a) {
  float4 v;
  asm volatile("ld.shared.v4.f32 {%0, %1, %2, %3}, [%4];"
               : "=f"(v.x), "=f"(v.y), "=f"(v.z), "=f"(v.w)
               : "r"(a));
  return v;
}
__device__ __forceinline__ float lds1(uint32_t a) {
  float v;
  asm volatile("ld.shared.f32 %0, [%1];" : "=f"(v) : "r"(a));
  return v;
}
__device__ __forceinline__ void sts4(uint32_t a, uint32_t x, uint32_t y, uint32_t z, uint32_t w) {
  asm volatile("st.shared.v4.b32 [%0], {%1, %2, %3, %4};" ::"r"(a), "r"(x), "r"(y), "r"(z), "r"(w)
               : "memory");
}
__device__ __forceinline__ void sts4f(uint32_t a, float x, float y, float z, float w) {
  asm volatile("st.shared.v4.f32 [%0], {%1, %2, %3, %4};" ::"r"(a), "f"(x), "f"(y), "f"(z), "f"(w)
               : "memory");
}
__device__ __forceinline__ void sts2f(uint32_t a, float x, float y) {
  asm volatile("st.shared.v2.f32 [%0], {%1, %2};" ::"r"(a), "f"(x), "f"(y) : "memory");
}
__device__ __forceinline__ void sts1f(uint32_t a, float x) {
  asm volatile("st.shared.f32 [%0], %1;" ::"r"(a), "f"(x) : "memory");
}

// Column scale: the power of two that brings the column's largest folded value m into [2^13, 2^14)
// (1 for m = 0 or not finite), and 1 / (8 scale).
__device__ __forceinline__ float scale_of(float m) {
  const int E = (int)((__float_as_uint(m) >> 23) & 255u);  // m in [2^(E-127), 2^(E-126))
  if (m == 0.f || E == 255) return 1.0f;
  const int s = 267 - E;  // biased exponent of 2^(14 - (E - 126))
  return __uint_as_float((uint32_t)(s > 254 ? 254 : s) << 23);
}
__device__ __forceinline__ float inv_scale(float s) {
  return (1.0f / s) * (1.0f / kSScale);
}

// eight folded rows of one column and parity, times the scale, as the hi and lo pieces
__device__ __forceinline__ void put_piece(uint32_t a, uint32_t ph, const float (&v)[8], float sc) {
  uint32_t hi[4], lo[4];
#pragma unroll
  for (int q = 0; q < 4; ++q) split_h2(v[2 * q] * sc, v[2 * q + 1] * sc, hi[q], lo[q]);
  sts4(a, hi[0], hi[1], hi[2], hi[3]);
  sts4(a + ph, lo[0], lo[1], lo[2], lo[3]);
}

// 16 columns of one accumulator plus those of the one `off` columns further
__device__ __forceinline__ void tmem_sum16(uint32_t acc, uint32_t off, float (&v)[16]) {
  uint32_t a[16], b[16];
  tmem_ld16_async(acc, a);
  tmem_ld16_async(acc + off, b);
  tmem_wait_ld();
#pragma unroll
  for (int c = 0; c < 16; ++c) v[c] = __uint_as_float(a[c]) + __uint_as_float(b[c]);
}

// 1/p of row r and column factor tmu for one kind of symbol; the kinds are compiled apart so that the
// unrolled epilogue stays small.
// 0, theta:  re = (1 - cos x) + tmu (th + (1-th) cos x), im = (-1 + (1-th) tmu) sin x;
// 1, BDF2:   re = (1 - cos x)^2 + tmu, im = -sin x (2 - cos x);
// 2, P_theta: 1/(lam_H + lam_Htheta tmu)
template <int KIND>
__device__ __forceinline__ float inv_sym_k(const SymRow &r, float omth, float tmu) {
  if (KIND == 2) return 1.0f / (r.a + r.b * tmu);
  float re, im;
  if (KIND == 0) {
    re = r.a + tmu * r.b;
    im = (-1.0f + omth * tmu) * r.c;
  } else {
    re = r.a + tmu;
    im = r.c;
  }
  float y;  // p is far from the subnormal range
  asm("rsqrt.approx.ftz.f32 %0, %1;" : "=f"(y) : "f"(re * re + im * im));
  return y;
}

// ---------------------------------------------------------------- host
// The hi (low half) and lo fp16 pieces of 8 sqrt(2/(len+1)) sin(pi a/(len+1)) for a = 0 .. len: every
// entry of the operand images is one of these or its negative (S_{k,t} has a = k t mod 2 (len+1)).  They
// go to the kernels that fill the images as an argument: filled by the host and copied, the images of
// a handle took 0.1 to 0.3 ms of its set-up.
struct SinePieces {
  uint32_t v[513];
  explicit SinePieces(int len) {
    const double PI = 3.14159265358979323846, sn = std::sqrt(2.0 / (len + 1));
    for (int a = 0; a <= len; ++a) {
      const double x = kSScale * sn * std::sin(PI * (double)a / (len + 1));
      const __half h = __float2half_rn((float)x);
      const __half l = __float2half_rn((float)(x - (double)__half2float(h)));
      const __half_raw rh = h, rl = l;
      v[a] = (uint32_t)rh.x | (uint32_t)rl.x << 16;
    }
  }
};

// Pieces of row k, folded columns t0 .. t0 + 15 (0-based; zeros from h on, and for k past len): the 16
// halves of hi and of lo as they stand in an image.
__device__ __forceinline__ void image_row(const SinePieces &S, int len, int h, int k, int t0, uint4 (&hi)[2],
                                          uint4 (&lo)[2]) {
  uint32_t w[16];
#pragma unroll
  for (int j = 0; j < 16; ++j) {
    const int t = t0 + j;
    int a = (int)((unsigned)(k * (t + 1)) % (unsigned)(2 * (len + 1)));
    uint32_t flip = 0u;
    if (a > len) {
      a -= len + 1;
      flip = 0x80008000u;
    }
    w[j] = k <= len && t < h ? S.v[a] ^ flip : 0u;
  }
  auto lo2 = [&](int j) { return __byte_perm(w[j], w[j + 1], 0x5410); };
  auto hi2 = [&](int j) { return __byte_perm(w[j], w[j + 1], 0x7632); };
#pragma unroll
  for (int q = 0; q < 2; ++q) {
    hi[q] = make_uint4(lo2(8 * q), lo2(8 * q + 2), lo2(8 * q + 4), lo2(8 * q + 6));
    lo[q] = make_uint4(hi2(8 * q), hi2(8 * q + 2), hi2(8 * q + 4), hi2(8 * q + 6));
  }
}

typedef CUresult (*EncodeFn)(CUtensorMap *, CUtensorMapDataType, cuuint32_t, void *,
                             const cuuint64_t *, const cuuint64_t *, const cuuint32_t *,
                             const cuuint32_t *, CUtensorMapInterleave, CUtensorMapSwizzle,
                             CUtensorMapL2promotion, CUtensorMapFloatOOBfill);

inline EncodeFn encode_fn() {
  static const EncodeFn f = [] {
    void *p = nullptr;
    cudaDriverEntryPointQueryResult q;
    if (cudaGetDriverEntryPointByVersion("cuTensorMapEncodeTiled", &p, 12000, cudaEnableDefault,
                                         &q) != cudaSuccess ||
        q != cudaDriverEntryPointSuccess)
      p = nullptr;
    return reinterpret_cast<EncodeFn>(p);
  }();
  return f;
}

// float32 tensor [d2][d1][d0], rows s1 floats apart, planes s2 floats apart; boxes of 32 x b1 x 1
// in 128-byte-swizzled rows.  Bases and strides are multiples of 16 bytes in the padded layout,
// and every copy starts at a multiple of 32 columns.
inline cudaError_t tma_encode(CUtensorMap *m, const float *base, long long d0, long long d1, long long d2,
                   long long s1, long long s2, int b1) {
  const EncodeFn f = encode_fn();
  if (!f) return cudaErrorNotSupported;
  const cuuint64_t dims[3] = {(cuuint64_t)d0, (cuuint64_t)d1, (cuuint64_t)d2};
  const cuuint64_t str[2] = {(cuuint64_t)s1 * 4u, (cuuint64_t)s2 * 4u};
  const cuuint32_t box[3] = {32u, (cuuint32_t)b1, 1u}, es[3] = {1u, 1u, 1u};
  const CUresult r = f(m, CU_TENSOR_MAP_DATA_TYPE_FLOAT32, 3, const_cast<float *>(base), dims, str,
                       box, es, CU_TENSOR_MAP_INTERLEAVE_NONE, CU_TENSOR_MAP_SWIZZLE_128B,
                       CU_TENSOR_MAP_L2_PROMOTION_L2_256B, CU_TENSOR_MAP_FLOAT_OOB_FILL_NONE);
  return r == CUDA_SUCCESS ? cudaSuccess : cudaErrorInvalidValue;
}

}  // namespace
}  // namespace st
