// Sine transforms of the mixed path on the tensor cores for axes of 257 to 512 points (y and z passes,
// and the time stage), fed and drained by tensor copies.  Float32 data in the padded layout.
//
// One parity of the folded transform (see st_dst_tma.cu) is a matrix A_P of up to 256 x 256 in two
// fp16 pieces: 256 KB, all of one SM's tensor memory.  So the rows are cut in halves as well: a block
// keeps the 128 rows mt 128 .. of one parity P (256 columns of tensor memory) for the whole launch, and
// the four blocks (P, mt) of a tile of 32 columns each load it, fold it for their parity, multiply and
// store their quarter of the rows.  The tile comes from memory once and from L2 three times more; the
// fold is done twice, which is cheap beside streaming A: the kernel this one replaced for the time
// stage (n <= 512, multiples of 32) streamed 512 KB of A through shared memory for every tile.
//   - a quarter's rows are written while other blocks may still read the tile, so the transform
//     goes from one vector to another (the stencil-output vector is free during a preconditioner
//     pass); the time stage is two launches, there (scaled by 1/p, with <v, P^-1 v>) and back;
//   - warps 0..3: epilogue (one per lane quadrant); 4..11 and 12..19: two build sets that take
//     alternate tiles, each with its own B buffer; 20: MMAs, 21: loads, 22: stores.  The staging
//     buffer of a tile (64 KB, two of them) is free as soon as its build has read it.
// Bound by latency like the kernels of st_dst_tma.cu (ncu, y at 511^2 x 32: issue slots 40% busy, tensor
// pipe 22%, DRAM 15%).  80 registers a thread is what 23 warps leave; 44 to 88 bytes of them spill.
// Every wait is bounded, as in st_dst_tma.cu.
#include "st_tma.cuh"

namespace st {
namespace {

constexpr int kNTL = 23 * 32;
constexpr uint32_t kSlotL = 65536u;  // 512 rows of 32 floats

struct LongDim {
  int len, h, hK;
  uint32_t sbo, ph;  // B operand: bytes between 8-column groups, of one piece (32 columns)
};
__host__ __device__ inline LongDim long_dim(int len) {
  LongDim d;
  d.len = len;
  d.h = (len + 1) >> 1;
  d.hK = (d.h + 15) & ~15;
  d.sbo = 16u * (uint32_t)d.hK + 16u;
  d.ph = 4u * d.sbo;
  return d;
}

struct LongSmem {
  // full[2], inempty[2], bfull[2], bempty[2], afull[2], aempty[2], ofull, oempty, done
  static constexpr uint32_t mbar = 0, tmem = 15u * 8u, zero = 128u, colinv = 160u,
                            tmu = colinv + 256u, part = tmu + 256u, ring = 3072u,
                            out = ring + 2u * kSlotL, bop = out + 16384u;
  static_assert(part + 2u * 1024u <= ring, "small arrays");
  static __host__ __device__ uint32_t total(const LongDim &D) { return bop + 4u * D.ph + 1008u; }
};

// KIND: -1 the transform alone; 0, 1, 2: scaled by 1/p (theta, BDF2, P_theta) with <v, P^-1 v>
template <int KIND>
__global__ void __launch_bounds__(kNTL, 1)
    k_dst_long(const __grid_constant__ CUtensorMap in0, const __grid_constant__ CUtensorMap out0,
               const __grid_constant__ CUtensorMap out1, int len, int chunks, unsigned groups,
               const uint4 *img, long long m, int mx, int px, Spec<float> sp, State *S, int tmode,
               double *__restrict__ partials, int gk) {
  __shared__ double red[32];
  if (gate_closed(S, gk)) return;
  extern __shared__ unsigned char smem_raw[];
  using L = LongSmem;
  const LongDim D = long_dim(len);
  const uint32_t sm = (smem_u32(smem_raw) + 1023u) & ~1023u;
  const int tid = threadIdx.x, warp = tid >> 5, lane = tid & 31;
  const int P = (blockIdx.x >> 1) & 1, mt = blockIdx.x & 1;
  const uint32_t full = sm + L::mbar, inempty = full + 16u, bfull = full + 32u, bempty = full + 48u,
                 afull = full + 64u, aempty = full + 80u, ofull = full + 96u, oempty = full + 104u,
                 done = full + 112u, tslot = sm + L::tmem;
  const unsigned first = blockIdx.x >> 2, step = gridDim.x >> 2;
  if (tid == 0) {
    for (int i = 0; i < 15; ++i) {
      uint32_t cnt = 1u;
      if (i == 6 || i == 7) cnt = 5u;                // bempty: MMA commit + epilogue warps
      if (i == 10 || i == 11 || i == 12) cnt = 4u;   // aempty, ofull: epilogue warps
      asm volatile("mbarrier.init.shared::cta.b64 [%0], %1;" ::"r"(full + 8u * i), "r"(cnt)
                   : "memory");
    }
    sts4(sm + L::zero, 0u, 0u, 0u, 0u);
    asm volatile("fence.mbarrier_init.release.cluster;" ::: "memory");
  }
  if (warp == 0) {
    asm volatile("tcgen05.alloc.cta_group::1.sync.aligned.shared::cta.b32 [%0], 512;" ::"r"(tslot)
                 : "memory");
    asm volatile("tcgen05.relinquish_alloc_permit.cta_group::1.sync.aligned;" ::: "memory");
  }
  fence_before();
  __syncthreads();
  fence_after();
  const uint32_t tmem = __float_as_uint(lds1(tslot));
  const uint32_t dcol = tmem + 256u;  // after A: [buffer][four accumulators][32 columns]
  auto load = [&](unsigned tile, int s) {
    const uint32_t mb = full + 8u * s, dst = sm + L::ring + (uint32_t)s * kSlotL;
    const unsigned pl = tile / (unsigned)chunks;
    const int x = (int)(tile - pl * chunks) * 32;
    mbar_expect_tx(mb, kSlotL);  // rows past the axis arrive as zeros
    tma_load3(dst, &in0, x, 0, (int)pl, mb);
    tma_load3(dst + kSlotL / 2, &in0, x, 256, (int)pl, mb);
  };
  // the first two loads fly while A is copied
  uint32_t preloaded = 0;
  if (warp == 21 && elect_one())
    for (unsigned tile = first; tile < groups && preloaded < 2u; tile += step)
      load(tile, (int)preloaded++);
  __syncwarp();
  load_a_variants(img + (size_t)(2 * P + mt) * (size_t)(2 * (D.hK >> 4)) * kM * 2, 2, D.hK, tmem,
                  warp, kNTL / 32, lane);
  fence_before();
  __syncthreads();
  fence_after();
  bool ok = true, drained = true;
  float esum = 0.f, ecomp = 0.f;
  if (warp == 21) {
    // ------------------------------------------------------------------ loads
    if (elect_one()) {
      uint32_t n = preloaded;
      for (unsigned tile = first + preloaded * step; tile < groups; tile += step, ++n) {
        if (!mbar_wait(inempty + 8u * (n & 1u), ((n >> 1) & 1u) ^ 1u)) {
          ok = false;
          break;
        }
        load(tile, (int)(n & 1u));
      }
      for (uint32_t i = n > 2u ? n - 2u : 0u; i < n; ++i)
        if (!mbar_wait(full + 8u * (i & 1u), (i >> 1) & 1u)) drained = false;
    }
    __syncwarp();
  } else if (warp == 22) {
    // ------------------------------------------------------------------ stores
    if (elect_one()) {
      uint32_t n = 0;
      for (unsigned tile = first; tile < groups; tile += step, ++n) {
        if (!mbar_wait(ofull, n & 1u)) {
          ok = false;
          break;
        }
        const unsigned pl = tile / (unsigned)chunks;
        tma_store3(P ? &out1 : &out0, sm + L::out, (int)(tile - pl * chunks) * 32, mt * 128, (int)pl);
        bulk_commit();
        bulk_wait_read();
        mbar_arrive(oempty);
      }
      bulk_wait_done();
    }
    __syncwarp();
  } else if (warp == 20) {
    // ------------------------------------------------------------------ MMA thread
    if (elect_one()) {
      // two pairs of accumulators, each for half of the 9 to 16 K steps (see issue_pair)
      const int KS = D.hK >> 4, KA = (KS + 1) >> 1;
      uint32_t n = 0;
      for (unsigned tile = first; tile < groups; tile += step, ++n) {
        const uint32_t b = n & 1u, ph = (n >> 1) & 1u, d = dcol + 128u * b;
        if (!mbar_wait(bfull + 8u * b, ph) || !mbar_wait(aempty + 8u * b, ph ^ 1u)) {
          ok = false;
          break;
        }
        fence_after();
        const uint64_t bd = make_desc_sbo(sm + L::bop + b * 2u * D.ph, D.sbo);
        issue_two_pairs<32, 8>(d, d + 64u, tmem, tmem + 8u * KA, (uint32_t)(D.hK >> 1), bd,
                               bd + 16u * (uint64_t)KA, D.ph >> 4, KA, KS - KA);
        mma_commit(afull + 8u * b);
        mma_commit(bempty + 8u * b);
      }
      mma_commit(done);
    }
    __syncwarp();
  } else if (warp >= 4) {
    // ------------------------------------------------------------------ build sets
    // thread: four adjacent columns of one t-block of eight folded rows
    const uint32_t k = (uint32_t)(warp - 4) >> 3;
    const int bt = tid - 128 - 256 * (int)k, w = bt >> 5, bar = 1 + (int)k;
    const int cq = lane & 7, tb = w * 4 + (lane >> 3);
    const uint32_t part = sm + L::part + k * 1024u, ci = sm + L::colinv + k * 128u;
    const uint32_t bo = sm + L::bop + k * 2u * D.ph, zero = sm + L::zero;
    const float sg = P ? -1.f : 1.f;
    uint32_t n = 0;
    for (unsigned tile = first; tile < groups; tile += step, ++n) {
      if ((n & 1u) != k) continue;
      const uint32_t ph = (n >> 1) & 1u, buf = sm + L::ring + k * kSlotL;
      float tv = 0.f;
      if (KIND >= 0 && bt < 32) {
        const unsigned pl = tile / (unsigned)chunks;
        tv = tmu_col(sp, (long long)(tile - pl * chunks) * 32 + bt, mx, px, m);
      }
      ok = mbar_wait(full + 8u * k, ph);
      float v[4][8];
      float4 mxv = make_float4(0.f, 0.f, 0.f, 0.f);
      if (ok) {
#pragma unroll
        for (int q = 0; q < 8; ++q) {
          const int t = tb * 8 + q, tm = len - 1 - t;
          auto row = [&](int r) { return buf + (uint32_t)(r * 128) + (uint32_t)((cq ^ (r & 7)) << 4); };
          // rows past the fold read zeros; the middle row of an odd length folds with nothing
          const float4 a = lds4(t < D.h ? row(t) : zero);
          const float4 b = lds4(t < D.h && tm != t ? row(tm) : zero);
          v[0][q] = fmaf(sg, b.x, a.x);
          v[1][q] = fmaf(sg, b.y, a.y);
          v[2][q] = fmaf(sg, b.z, a.z);
          v[3][q] = fmaf(sg, b.w, a.w);
          mxv.x = fmaxf(mxv.x, fabsf(v[0][q]));
          mxv.y = fmaxf(mxv.y, fabsf(v[1][q]));
          mxv.z = fmaxf(mxv.z, fabsf(v[2][q]));
          mxv.w = fmaxf(mxv.w, fabsf(v[3][q]));
        }
      }
#pragma unroll
      for (int o = 8; o <= 16; o <<= 1) {
        mxv.x = fmaxf(mxv.x, __shfl_xor_sync(0xffffffffu, mxv.x, o));
        mxv.y = fmaxf(mxv.y, __shfl_xor_sync(0xffffffffu, mxv.y, o));
        mxv.z = fmaxf(mxv.z, __shfl_xor_sync(0xffffffffu, mxv.z, o));
        mxv.w = fmaxf(mxv.w, __shfl_xor_sync(0xffffffffu, mxv.w, o));
      }
      if (lane < 8) sts4f(part + (uint32_t)(w * 128 + cq * 16), mxv.x, mxv.y, mxv.z, mxv.w);
      if (ok) ok = mbar_wait(bempty + 8u * k, ph ^ 1u);
      ok = group_sync_and(ok, bar, 256);
      if (!ok) break;
      if (bt == 0) mbar_arrive(inempty + 8u * k);  // every thread has its rows: the slot is free
      if (KIND >= 0 && bt < 32) sts1f(sm + L::tmu + k * 128u + (uint32_t)bt * 4u, tv);
#pragma unroll
      for (int i = 0; i < 8; ++i) {
        const float4 x = lds4(part + (uint32_t)(i * 128 + cq * 16));
        mxv.x = fmaxf(mxv.x, x.x);
        mxv.y = fmaxf(mxv.y, x.y);
        mxv.z = fmaxf(mxv.z, x.z);
        mxv.w = fmaxf(mxv.w, x.w);
      }
      const float sc[4] = {scale_of(mxv.x), scale_of(mxv.y), scale_of(mxv.z), scale_of(mxv.w)};
      if (tb == 0)
        sts4f(ci + (uint32_t)(cq * 16), inv_scale(sc[0]), inv_scale(sc[1]), inv_scale(sc[2]),
              inv_scale(sc[3]));
      if (tb * 8 < D.hK) {
#pragma unroll
        for (int j = 0; j < 4; ++j) {
          const int c = 4 * cq + j;
          put_piece(bo + (uint32_t)(c >> 3) * D.sbo + (uint32_t)(tb * 128 + (c & 7) * 16), D.ph, v[j],
                    sc[j]);
        }
      }
      fence_async_smem();
      group_sync(bar, 256);
      if (bt == 0) mbar_arrive(bfull + 8u * k);
    }
  } else {
    // ------------------------------------------------------------------ epilogue
    const int R = warp * 32 + lane, r = mt * 128 + R;
    const uint32_t lanes = (uint32_t)(warp * 32) << 16;
    const int kf = 2 * r + 1 + P;  // a row past len holds zeros and is not stored
    SymRow sr{};
    float omth = 0.f;
    if (KIND >= 0) {
      sr = sym_row(sp, kf <= len ? kf : len);
      omth = 1.0f - sp.theta;
    }
    const uint32_t a = sm + L::out + (uint32_t)(R * 128), sw = (uint32_t)(R & 7) << 4;
    uint32_t n = 0;
    for (unsigned tile = first; tile < groups; tile += step, ++n) {
      const uint32_t b = n & 1u, ph = (n >> 1) & 1u;
      ok = __all_sync(0xffffffffu, mbar_wait(bfull + 8u * b, ph) ? 1 : 0) != 0;
      if (ok) ok = __all_sync(0xffffffffu, mbar_wait(afull + 8u * b, ph) ? 1 : 0) != 0;
      if (ok) ok = __all_sync(0xffffffffu, mbar_wait(oempty, (n & 1u) ^ 1u) ? 1 : 0) != 0;
      if (!ok) break;
      fence_after();
      const uint32_t ci = sm + L::colinv + b * 128u, tm = sm + L::tmu + b * 128u;
      float rs = 0.f;
#pragma unroll
      for (int hf = 0; hf < 2; ++hf) {
        float v[16];
        {
          float w[16];
          const uint32_t acc = dcol + 128u * b + lanes + 16u * hf;
          tmem_sum16(acc, 32u, v);
          tmem_sum16(acc + 64u, 32u, w);
#pragma unroll
          for (int c = 0; c < 16; ++c) v[c] += w[c];
        }
        if (hf == 1) {
          fence_before();
          __syncwarp();
          if (lane == 0) mbar_arrive(aempty + 8u * b);  // the accumulator is free
        }
#pragma unroll
        for (int c = 0; c < 4; ++c) {
          const uint32_t co = 64u * (uint32_t)hf + 16u * c;
          const float4 f4 = lds4(ci + co);
          float o[4] = {v[4 * c] * f4.x, v[4 * c + 1] * f4.y, v[4 * c + 2] * f4.z,
                        v[4 * c + 3] * f4.w};
          if (KIND >= 0) {
            const float4 t4 = lds4(tm + co);
            const float t[4] = {t4.x, t4.y, t4.z, t4.w};
#pragma unroll
            for (int e = 0; e < 4; ++e) {
              const float y = o[e];
              o[e] = y * inv_sym_k<KIND < 0 ? 0 : KIND>(sr, omth, t[e]);
              rs = fmaf(y, o[e], rs);
            }
          }
          sts4f(a + (co ^ sw), o[0], o[1], o[2], o[3]);
        }
      }
      if (KIND >= 0) {
        const float term = rs - ecomp;
        const float t = esum + term;
        ecomp = (t - esum) - term;
        esum = t;
      }
      fence_async_smem();
      __syncwarp();
      if (lane == 0) {
        mbar_arrive(bempty + 8u * b);  // the column factors are read
        mbar_arrive(ofull);
      }
    }
  }
  fence_before();
  const bool all_ok = __syncthreads_and(ok ? 1 : 0) != 0;
  const bool copies = __syncthreads_and(drained ? 1 : 0) != 0;
  tc_release_cols<512>(all_ok, true, done, 0u, false, 0u, 0u, tmem, S, copies);
  if (KIND >= 0 && tmode != TM_NONE) {
    const double e = (double)esum - (double)ecomp;
    double tot;
    if (last_block_reduce<kNTL>(e, partials, &S->counter[CNT_TIME], gridDim.x, blockIdx.x, red,
                                &tot) &&
        tid == 0) {
      if (tmode == TM_INIT || tmode == TM_RESTART)
        minres_init_scalars_dev(S, tot);
      else
        minres_givens_dev(S, tot);
    }
  }
}

// Operand image of 8 S_len: [parity][half of the rows][hi, lo][K step][128 rows][16], zeros past the axis.  A
// block per K step and quarter, a thread per row.
__global__ void __launch_bounds__(kM) k_image_long(const __grid_constant__ SinePieces S, int len, uint4 *img) {
  const int KS = gridDim.x, ks = blockIdx.x, p = blockIdx.y, row = threadIdx.x;
  const int h = (len + 1) >> 1, r = (p & 1) * 128 + row;
  uint4 hi[2], lo[2];
  image_row(S, len, h, r < h ? 2 * r + 1 + (p >> 1) : len + 1, ks * 16, hi, lo);
  uint4 *q = img + ((size_t)(2 * p * KS + ks) * kM + row) * 2;
  q[0] = hi[0];
  q[1] = hi[1];
  q += (size_t)KS * kM * 2;
  q[0] = lo[0];
  q[1] = lo[1];
}

template <int KIND>
cudaError_t launch_long(const float *in, float *out, int len, long long cols, long long planes,
                        long long rs, long long ps, const unsigned short *img, const Geom &g,
                        const Spec<float> &sp, State *S, int tmode, double *partials, int gk, int kc,
                        cudaStream_t st) {
  const LongDim D = long_dim(len);
  const uint32_t smem = LongSmem::total(D);
  const int chunks = (int)((cols + 31) / 32);
  const unsigned groups = (unsigned)(planes * chunks);
  CUtensorMap mi, m0, m1;
  cudaError_t e = tma_encode(&mi, in, cols, len, planes, rs, ps, 256);
  if (e == cudaSuccess) e = tma_encode(&m0, out, cols, (len + 1) / 2, planes, 2 * rs, ps, 128);
  if (e == cudaSuccess) e = tma_encode(&m1, out + rs, cols, len / 2, planes, 2 * rs, ps, 128);
  if (e != cudaSuccess) return e;
  auto kern = k_dst_long<KIND>;
  e = cudaFuncSetAttribute(kern, cudaFuncAttributeMaxDynamicSharedMemorySize, (int)smem);
  if (e != cudaSuccess) return e;
  unsigned quads = (unsigned)time_tc_grid() / 4u;
  if (groups < quads) quads = groups;
  prof_begin(kc, st);
  kern<<<4u * quads, kNTL, smem, st>>>(mi, m0, m1, len, chunks, groups,
                                       reinterpret_cast<const uint4 *>(img), g.mp, g.mx, g.px, sp, S,
                                       tmode, partials, gk);
  prof_end(st);
  return cudaGetLastError();
}

}  // namespace

bool dst_long_supported(int len) { return len > 256 && len <= 512; }

size_t dst_long_image_halves(int len) {
  return (size_t)4 * 2 * kM * (((len + 1) / 2 + 15) & ~15);
}

cudaError_t dst_long_build_image(int len, unsigned short *img) {
  k_image_long<<<dim3(long_dim(len).hK >> 4, 4), kM>>>(SinePieces(len), len, (uint4 *)img);
  return cudaGetLastError();
}

cudaError_t launch_dst_long_y(const float *in, float *out, const Geom &g, const unsigned short *img,
                              State *S, int gk, cudaStream_t st) {
  return launch_long<-1>(in, out, g.my, g.px, (long long)g.n * g.mz, g.px, (long long)g.px * g.my, img,
                         g, Spec<float>{}, S, TM_NONE, nullptr, gk, KC_DSTY, st);
}

cudaError_t launch_dst_long_z(const float *in, float *out, const Geom &g, const unsigned short *img,
                              State *S, int gk, cudaStream_t st) {
  const long long pl = (long long)g.px * g.my;
  return launch_long<-1>(in, out, g.mz, pl, g.n, pl, g.mp, img, g, Spec<float>{}, S, TM_NONE, nullptr,
                         gk, KC_DSTY, st);
}

cudaError_t launch_time_long(float *data, float *scratch, const Geom &g, const Spec<float> &sp,
                             const unsigned short *img, State *S, int tmode, double *partials, int gk,
                             cudaStream_t st) {
  cudaError_t e;
  if (sp.prec == ST_PREC_PTHETA)
    e = launch_long<2>(data, scratch, g.n, g.mp, 1, g.mp, g.Np, img, g, sp, S, tmode, partials, gk,
                       KC_TIME, st);
  else if (sp.scheme == ST_THETA)
    e = launch_long<0>(data, scratch, g.n, g.mp, 1, g.mp, g.Np, img, g, sp, S, tmode, partials, gk,
                       KC_TIME, st);
  else
    e = launch_long<1>(data, scratch, g.n, g.mp, 1, g.mp, g.Np, img, g, sp, S, tmode, partials, gk,
                       KC_TIME, st);
  if (e != cudaSuccess) return e;
  return launch_long<-1>(scratch, data, g.n, g.mp, 1, g.mp, g.Np, img, g, sp, S, TM_NONE, partials, gk,
                         KC_TIME, st);
}

}  // namespace st
