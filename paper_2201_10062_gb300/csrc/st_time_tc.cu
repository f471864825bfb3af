// Float64-accurate time-axis DST-I on the 5th-generation tensor cores (tcgen05) with integer digits, for
// the float64 path (k_time_tcd).
//
// The folded transform is two dense products per parity of the output index k:
//   odd  k = 2r+1:  Y_k = sum_{t=1..h} S_{k,t} (x_t + x_{n+1-t})
//   even k = 2r+2:  Y_k = sum_{t=1..h} S_{k,t} (x_t - x_{n+1-t}),     h = ceil(n/2),
// i.e. D_P[r][j] = sum_t A_P[r][t] B_P[t][j] with A_P fixed and B_P the folded data of a tile of 32
// spatial columns.  Every wait on an mbarrier is bounded; on timeout the block records
// ST_ERR_TIMEOUT in the MINRES state and stops.  Before it releases its tensor memory it gives every MMA
// batch whose commit it has not seen complete one more bounded wait: MMAs still in flight may be
// writing that memory.  If that wait runs out as well, the block keeps it (it must not be given to
// another block while an MMA may write it) and sets State::tmem_held, which closes the device to
// further calls on the host side.
#include <cmath>
#include <vector>
#include <cstdlib>

#include "st_tc.cuh"

namespace st {
namespace {

constexpr int kYS = kTN + 1;  // padded row of the parity-split Y tile (conflict-free row writes)

}  // namespace

int time_tc_grid() {
  static int sms = 0;
  if (!sms) {
    int dev = 0;
    cudaGetDevice(&dev);
    cudaDeviceGetAttribute(&sms, cudaDevAttrMultiProcessorCount, dev);
    if (sms <= 0) sms = 152;
  }
  return sms;
}

// ------------------------------------------------------------------ float64-accurate time DST
// The time stage of the float64 preconditioner (Sec. 3.1.1, steps 1-3 along time) on the tensor
// cores, for double-float data.  An fp16 MMA with float32 accumulation is exact on integers as
// long as every partial sum stays below 2^24, so both operands are cut into integer digits:
//   S^ = S 2^eS = sum_i S_i 2^-7i,   X^ = X 2^ec = sum_j B_j 2^-7j,   i, j = 0..6,
// with |S_i|, |B_j| <= 2^7 (one scale for S, one per column c of X and parity).  S's digits are
// rounded ones taken in float64 on the host; X's are those of the folded double-float value as a
// 64-bit fixed-point integer (2^42 X^, rounded), in -64..63 below the top one.  One product
// S_i B_j over K = h <= 128 folded rows is at most 2^21 in magnitude, and the at most seven
// products of a digit group g = i + j sum below 2^24, so each group accumulates exactly in
// float32.  The groups g <= 6 are kept (28 products per parity); the dropped ones and the
// digits' remainders are below 2^-41 of the column's largest entry, and of no sign: measured against
// float64 the stage is the more accurate one.  The groups are summed in
// double-float (sum_g acc_g 2^-7g, TwoSum) and unscaled by 2^-(eS + ec).
//
// With S's digits read from shared memory each MMA (M = 128, N = 32) costs about ten times one
// that reads A from tensor memory, so the seven digits of one parity (448 tensor-memory columns)
// stay resident for a whole phase: a block takes its tiles of 32 spatial columns once for each
// parity.  Within a phase three roles work on different tiles at once, handing off through
// mbarriers (every wait bounded):
//   - eight build warps fold a tile's rows for the parity (x_t + x_{n+1-t}, or the difference),
//     choose each column's scale from its largest folded entry and write the seven digits as fp16
//     B operands (canonical K-major, [digit][32][h]) into one of two buffers;
//   - one thread issues the digit groups g = 0..6 of a tile in order, alternating between two
//     32-column accumulators, and frees the B buffer after the tile's last group;
//   - eight drain warps take each group out of tensor memory (tcgen05.ld; one row, 16 columns
//     per thread), add it into double-float sums, release the accumulator, and after group 6
//     unscale the tile's rows (and in the first launch multiply by 1/p and accumulate
//     <v, P^-1 v>), stage them in shared memory and write them out row by row.
// A row of output depends on every input row, so the transform cannot run in place: the first
// launch reads the data and writes the scaled transform into a scratch vector, the second
// transforms the scratch vector back into the data.
namespace {

constexpr int kDg = 7;                                   // digits per operand
constexpr int kDgW = 7;                                  // bits per digit
constexpr int kDrainW = 8;                               // warps 0..7: drain and epilogue
constexpr int kBuildW = 8;                               // warps 8..15: digits of the next tile
constexpr int kNTG = (kDrainW + kBuildW + 1) * 32;       // and warp 16: the MMA thread
constexpr int kBarD = 1, kBarB = 2;                      // named barriers of the two groups

struct TcdSmem {
  uint32_t bdig, ytile, part, cdown, tmu, mbar, tmem, total;
};

// folded rows padded to the MMA's K step (rows past the fold are zero digits)
__host__ __device__ inline int tcd_hk(int n) { return ((n + 1) / 2 + 15) & ~15; }

__host__ __device__ inline TcdSmem tcd_layout(int n) {
  const int h = (n + 1) / 2, hK = tcd_hk(n);
  TcdSmem L{};
  uint32_t o = 0;
  L.bdig = o;  // two buffers of [digit][32][hK] fp16
  o += 2u * kDg * kTN * (uint32_t)hK * 2u;
  L.ytile = o;  // the drain warps' staged rows: hi floats then lo floats, [h][kYS]
  o += 2u * (uint32_t)h * kYS * 4u;
  L.part = o;  // 8 build warps x 32 per-column partial maxima
  o += (uint32_t)kBuildW * kTN * 4u;
  L.cdown = o;  // per buffer and column: 2^-(eS + e_c), the factor that undoes both scales
  o += 2u * kTN * 4u;
  L.tmu = o;  // per column: tau mu_j and the symbol's column factor w_j, double-float
  o += 2u * kTN * 8u;
  L.mbar = o;  // bfull[2], bempty[2], afull[2], aempty[2], done
  o += 9u * 8u;
  L.tmem = o;
  o += 8u;
  L.total = o;
  return L;
}

__device__ __forceinline__ dd ld_dd(const dd *p) {
  const float2 v = *reinterpret_cast<const float2 *>(p);
  return dd(v.x, v.y);
}
__device__ __forceinline__ void st_dd(dd *p, dd v) {
  *reinterpret_cast<float2 *>(p) = make_float2(v.hi, v.lo);
}

// 2^e as a float (exact; e outside the normal range through ldexpf)
__device__ __forceinline__ float pow2f(int e) {
  return (e >= -126 && e <= 127) ? __int_as_float((e + 127) << 23) : ldexpf(1.0f, e);
}

// 1/p in double-float with the per-row parts hoisted (the double-float form of inv_symbol):
// theta and BDF2 take 1/sqrt((a + tmu b)^2 + (w c)^2) with a, b, c per time frequency and
// w per column (w = -1 + (1 - theta) tmu for theta, 1 for BDF2); P_theta takes 1/(a + b tmu).
struct SymRowDD {
  dd a, b, c;
};
__device__ __forceinline__ SymRowDD sym_row_dd(const Spec<dd> &sp, int k) {
  SymRowDD r;
  const dd hk = sp.hk[k - 1], ck = sp.ck[k - 1], sk = sp.sk[k - 1];
  if (sp.prec == ST_PREC_PTHETA) {
    r.a = sp.lh[k - 1];
    r.b = sp.lht[k - 1];
    r.c = dd(0.f, 0.f);
  } else if (sp.scheme == ST_THETA) {
    r.a = hk;
    r.b = sp.theta + (dd(1) - sp.theta) * ck;
    r.c = sk;
  } else {
    r.a = hk * hk;
    r.b = dd(1);
    r.c = -(sk * (dd(1) + hk));
  }
  return r;
}
__device__ __forceinline__ dd sym_col_w(const Spec<dd> &sp, dd tmu) {
  if (sp.prec != ST_PREC_PTHETA && sp.scheme == ST_THETA)
    return dd(-1) + (dd(1) - sp.theta) * tmu;
  return dd(1);
}
__device__ __forceinline__ dd inv_sym_dd(const Spec<dd> &sp, const SymRowDD &r, dd tmu, dd w) {
  if (sp.prec == ST_PREC_PTHETA) return dd(1) / (r.a + r.b * tmu);
  const dd re = dd_fma(tmu, r.b, r.a), im = w * r.c;
  return rsqrt_dd(dd_fma(re, re, im * im));
}

// max(a, b), NaN if either is one
__device__ __forceinline__ float max_nan(float a, float b) {
  float r;
  asm("max.NaN.f32 %0, %1, %2;" : "=f"(r) : "f"(a), "f"(b));
  return r;
}

// The seven 7-bit digits of x 2^e (|x 2^e| < 2^7, double-float): X = 2^42 x 2^e rounded to an
// integer, held as H 2^21 + Lo with 0 <= Lo < 2^21 (32-bit parts: no float64 conversion), is
// sum_k d_k 2^(42-7k) with d_0 signed and -64 <= d_k < 64 below it: half of every lower digit's
// range is added to X first, and the 7-bit fields of the sum are d_k + 64.  Balanced, the products that
// the digit groups leave out have no mean.  (With d_k in 0..127 they left the same error in every
// column, which the transforms along space gather in a few nodes: at 127 x 63 x 191 a largest error
// of 5.2e-13 of the largest entry, now 2.0e-14; the double-float kernel's is 5.9e-14.)
// Returned are the fields d_0 + 128 and d_k + 64: 0..256 and 0..127.
__device__ __forceinline__ void digits7(dd x, float up21, uint32_t (&d)[kDg]) {
  constexpr int kMid = (64 << 14) | (64 << 7) | 64;
  const float xh = x.hi * up21, xl = x.lo * up21;  // exact: powers of two
  int H = __float2int_rn(xh);                      // |H| <= 2^28; exact when |xh| >= 2^24
  const float r = xh - (float)H;                   // exact, |r| <= 1/2
  int Lo = __float2int_rn((r + xl) * 2097152.0f);  // (r + xl) 2^21; the rounding is below 1
  Lo += kMid;
  const int carry = Lo >> 21;                      // floor(Lo / 2^21)
  const uint32_t L = (uint32_t)Lo;
  const uint32_t U = (uint32_t)H + (uint32_t)carry + (uint32_t)kMid + (128u << 21);
  d[0] = (U >> 21) & 511u;  // 9 bits: a column that is not finite stays within half's integers too
  d[1] = (U >> 14) & 127u;
  d[2] = (U >> 7) & 127u;
  d[3] = U & 127u;
  d[4] = (L >> 14) & 127u;
  d[5] = (L >> 7) & 127u;
  d[6] = L & 127u;
}

// two fields as halves, their offset taken off: half 0x6400 | f is 1024 + f for f < 1024
__device__ __forceinline__ uint32_t digit_pair(uint32_t f0, uint32_t f1, bool top) {
  const uint32_t v = f0 | (f1 << 16) | 0x64006400u;
  const uint32_t o = top ? 0x64806480u : 0x64406440u;  // 1024 + 128, 1024 + 64
  const __half2 r = __hsub2(*reinterpret_cast<const __half2 *>(&v),
                            *reinterpret_cast<const __half2 *>(&o));
  return *reinterpret_cast<const uint32_t *>(&r);
}

// scaled: out = (S_n x)/p per column with <in, P^-1 in> into the MINRES state (tmode);
// otherwise out = S_n x.  in and out do not overlap.
__global__ void __launch_bounds__(kNTG, 1)
    k_time_tcd(const dd *__restrict__ in, dd *__restrict__ out, int n, long long m, int mx,
               Spec<dd> sp, const unsigned char *A_g, int eS, int scaled, State *S, int tmode,
               double *__restrict__ partials, int gk) {
  __shared__ double red[32];
  if (gate_closed(S, gk)) return;
  extern __shared__ __align__(1024) unsigned char smem[];
  const int h = (n + 1) >> 1, hK = tcd_hk(n), hb = hK >> 3;
  const TcdSmem L = tcd_layout(n);
  const int tid = threadIdx.x, warp = tid >> 5, lane = tid & 31;
  const uint32_t bop = (uint32_t)kTN * hK * 2u;  // one digit's B operand
  const uint32_t bbytes = (uint32_t)kDg * bop;   // one B buffer
  uint32_t *tmem_slot = reinterpret_cast<uint32_t *>(smem + L.tmem);
  float *yhi = reinterpret_cast<float *>(smem + L.ytile);
  float *ylo = yhi + (size_t)h * kYS;
  float *part = reinterpret_cast<float *>(smem + L.part);
  float *cdown = reinterpret_cast<float *>(smem + L.cdown);
  dd *tmus = reinterpret_cast<dd *>(smem + L.tmu);
  const uint32_t mb = smem_u32(smem + L.mbar);
  const uint32_t bfull = mb, bempty = mb + 16u, afull = mb + 32u, aempty = mb + 48u,
                 done = mb + 64u;
  const long long ntiles = (m + kTN - 1) / kTN;
  if (tid == 0) {
    for (int i = 0; i < 9; ++i) {
      const uint32_t cnt = (i == 6 || i == 7) ? (uint32_t)kDrainW : 1u;  // aempty: every drain warp
      asm volatile("mbarrier.init.shared::cta.b64 [%0], %1;" ::"r"(mb + 8u * i), "r"(cnt)
                   : "memory");
    }
    asm volatile("fence.mbarrier_init.release.cluster;" ::: "memory");
  }
  if (warp == 0) {
    asm volatile("tcgen05.alloc.cta_group::1.sync.aligned.shared::cta.b32 [%0], 512;" ::"r"(
                     smem_u32(tmem_slot))
                 : "memory");
    asm volatile("tcgen05.relinquish_alloc_permit.cta_group::1.sync.aligned;" ::: "memory");
  }
  fence_before();
  __syncthreads();
  fence_after();
  if (tid == 0) {  // both B buffers and both accumulators start free
    mbar_arrive(bempty);
    mbar_arrive(bempty + 8u);
    for (int k = 0; k < kDrainW; ++k) {
      mbar_arrive(aempty);
      mbar_arrive(aempty + 8u);
    }
  }
  const uint32_t tmem = *tmem_slot;
  const uint32_t acol = (uint32_t)(hK / 2);           // tensor-memory columns of one S digit
  const uint32_t dcol = tmem + (uint32_t)kDg * acol;  // the two accumulators follow S
  bool ok = true;
  // phases of bfull, bempty, afull and aempty as this thread's role waits on them
  // mbarrier phases, one bit per buffer (registers; an indexed array would live in local memory)
  uint32_t pbf = 0u, pbe = 0u, paf = 0u, pae = 0u;
  uint32_t G = 0;  // digit groups this thread's role has handled (accumulator G & 1)
  MacAcc<dd> en;   // drain threads: their part of <v, P^-1 v>
  en.zero();
  __syncthreads();

  for (int P = 0; P < 2 && ok; ++P) {
    // this parity's seven S digits into tensor memory: warp w writes lanes 32 (w % 4).., pieces
    // split among the warps of that quadrant
    {
      const int q = warp & 3, nq = (kNTG / 32 - q + 3) / 4, r = (q << 5) + lane;
      const uint32_t tl = (uint32_t)(q * 32) << 16;
      for (int pc = warp >> 2; pc < kDg; pc += nq) {
        const unsigned char *img = A_g + (size_t)(P * kDg + pc) * kM * hK * 2u;
        for (int ks = 0; ks < hK / 16; ++ks) {
          uint32_t w[8];
          const uint4 a0 = *reinterpret_cast<const uint4 *>(img + canon_off(r, ks * 16, hK));
          const uint4 a1 = *reinterpret_cast<const uint4 *>(img + canon_off(r, ks * 16 + 8, hK));
          w[0] = a0.x; w[1] = a0.y; w[2] = a0.z; w[3] = a0.w;
          w[4] = a1.x; w[5] = a1.y; w[6] = a1.z; w[7] = a1.w;
          tmem_st8(tmem + tl + (uint32_t)pc * acol + (uint32_t)ks * 8u, w);
        }
      }
      asm volatile("tcgen05.wait::st.sync.aligned;" ::: "memory");
    }
    fence_before();
    __syncthreads();
    fence_after();
    if (warp == kDrainW + kBuildW) {
      // ---------------------------------------------------------------- MMA thread (the same elected
      // lane in every phase)
      if (elect_one()) {
        int u = 0;
        for (long long tile = blockIdx.x; tile < ntiles && ok; tile += gridDim.x, ++u) {
          const int b = u & 1;
          if (!mbar_wait(bfull + 8u * b, ((pbf >> b) & 1u))) {
            ok = false;
            break;
          }
          pbf ^= 1u << b;
          // descriptors differ only in their start-address field (address / 16), so each MMA
          // takes one add on a descriptor built once per tile
          const uint64_t bdesc = make_desc(smem_u32(smem + L.bdig) + (uint32_t)b * bbytes, hK);
          const int ksteps = hK / 16;
          for (int g = 0; g < kDg; ++g) {
            const int a = (int)(G & 1u);
            if (!mbar_wait(aempty + 8u * a, ((pae >> a) & 1u))) {
              ok = false;
              break;
            }
            pae ^= 1u << a;
            fence_after();
            const uint32_t d = dcol + (uint32_t)(kTN * a);
            uint32_t acc = 0u;
            for (int i = 0; i <= g; ++i) {
              const uint32_t at = tmem + (uint32_t)i * acol;
              const uint64_t bd = bdesc + (uint64_t)(((uint32_t)(g - i) * bop) >> 4);
#pragma unroll 8
              for (int ks = 0; ks < ksteps; ++ks) {
                mma_ta<kTN>(d, at + (uint32_t)ks * 8u, bd + (uint64_t)(16 * ks), acc);
                acc = 1u;
              }
            }
            mma_commit(afull + 8u * a);
            ++G;
          }
          if (!ok) break;
          mma_commit(bempty + 8u * b);  // the buffer is free once this tile's MMAs are done
        }
      }
      __syncwarp();
    } else if (warp >= kDrainW) {
      // ---------------------------------------------------------------- build warps
      const int bw = warp - kDrainW, bc = lane;
      int u = 0;
      for (long long tile = blockIdx.x; tile < ntiles; tile += gridDim.x, ++u) {
        const int b = u & 1;
        const long long j0 = tile * kTN;
        const int je = (int)min((long long)kTN, m - j0);
        ok = group_sync_and(mbar_wait(bempty + 8u * b, ((pbe >> b) & 1u)), kBarB, kBuildW * 32);
        if (!ok) break;
        pbe ^= 1u << b;
        dd f[2][8];
        float mxv = 0.f;
#pragma unroll
        for (int it = 0; it < 2; ++it) {
          const int tb = bw + kBuildW * it;
#pragma unroll
          for (int q = 0; q < 8; ++q) {
            f[it][q] = dd(0.f, 0.f);
            const int t = tb * 8 + q, tm = n - 1 - t;
            if (t <= tm && bc < je) {
              const dd x1 = ld_dd(in + (long long)t * m + j0 + bc);
              if (t == tm) {
                // the middle row of an odd n: only odd k see it
                if (P == 0) f[it][q] = x1;
              } else {
                const dd x2 = ld_dd(in + (long long)tm * m + j0 + bc);
                f[it][q] = P == 0 ? x1 + x2 : x1 - x2;
              }
              mxv = max_nan(mxv, fabsf(f[it][q].hi));
            }
          }
        }
        part[bw * kTN + bc] = mxv;
        group_sync(kBarB, kBuildW * 32);
        float cm = 0.f;
#pragma unroll
        for (int k = 0; k < kBuildW; ++k) cm = max_nan(cm, part[k * kTN + bc]);
        // digits hold no NaN or infinity: a column with one gets the factor NaN, which the drain
        // multiplies the whole column of the result by
        const bool fin = isfinite(cm);
        int e = 0;
        if (cm > 0.f && fin) {
          int E;
          frexpf(cm, &E);
          // cm 2^e in [2^6, 2^7); below 2^-100 the digits end at 2^-148, where float32 itself does,
          // and 2^(e + 21) stays finite
          e = min(7 - E, 106);
        }
        if (bw == 0) cdown[b * kTN + bc] = fin ? pow2f(-(eS + e)) : __int_as_float(0x7fc00000);
        const float up21 = pow2f(e + 21);
        unsigned char *bb = smem + L.bdig + (uint32_t)b * bbytes;
#pragma unroll
        for (int it = 0; it < 2; ++it) {
          const int tb = bw + kBuildW * it;
          if (tb >= hb) continue;
          uint32_t dq[8][kDg];
#pragma unroll
          for (int q = 0; q < 8; ++q) digits7(f[it][q], up21, dq[q]);
          const uint32_t off = canon_off(bc, tb * 8, hK);
#pragma unroll
          for (int dg = 0; dg < kDg; ++dg) {
            uint32_t pk[4];
#pragma unroll
            for (int q2 = 0; q2 < 4; ++q2)
              pk[q2] = digit_pair(dq[2 * q2][dg], dq[2 * q2 + 1][dg], dg == 0);
            *reinterpret_cast<uint4 *>(bb + (uint32_t)dg * bop + off) =
                make_uint4(pk[0], pk[1], pk[2], pk[3]);
          }
        }
        fence_async_smem();
        group_sync(kBarB, kBuildW * 32);  // the buffer is written (and `part` read)
        if (bw == 0 && lane == 0) mbar_arrive(bfull + 8u * b);
      }
    } else {
      // ---------------------------------------------------------------- drain warps
      const int q4 = warp & 3, c0 = (warp >> 2) * 16;
      const int r = (q4 << 5) + lane;
      const int krow = (P == 0) ? 2 * r + 1 : 2 * r + 2;  // time frequency of row r (1-based)
      const bool row_ok = r < h && krow <= n;
      const SymRowDD srow = sym_row_dd(sp, row_ok ? krow : 1);
      const uint32_t lanes = (uint32_t)(q4 * 32) << 16;
      int u = 0;
      for (long long tile = blockIdx.x; tile < ntiles; tile += gridDim.x, ++u) {
        const int b = u & 1;
        const long long j0 = tile * kTN;
        const int je = (int)min((long long)kTN, m - j0);
        // each warp waits on its own (warp-uniform result); the drain group combines the results
        // once per tile, before its first named barrier, so that no warp leaves a barrier early
        if (ok) {
          ok = __all_sync(0xffffffffu, mbar_wait(bfull + 8u * b, ((pbf >> b) & 1u)) ? 1 : 0) != 0;
          if (ok) pbf ^= 1u << b;
        }
        float cd[16];
#pragma unroll
        for (int c = 0; c < 16; ++c) cd[c] = cdown[b * kTN + c0 + c];
        if (scaled && warp == 0) {
          dd tv(0.f, 0.f);
          if (lane < je) {
            const long long jj = j0 + lane;
            const long long jy = jj / mx, jx = jj - jy * mx;
            tv = sp.mux[jx] + sp.muy[jy];
          }
          tmus[lane] = tv;
          tmus[kTN + lane] = sym_col_w(sp, tv);
        }
        float s[16], t[16];
        for (int g = 0; g < kDg; ++g) {
          const int a = (int)(G & 1u);
          ++G;
          if (!ok) continue;
          ok = __all_sync(0xffffffffu, mbar_wait(afull + 8u * a, ((paf >> a) & 1u)) ? 1 : 0) != 0;
          if (!ok) continue;
          paf ^= 1u << a;
          fence_after();
          float v[16];
          tmem_ld16(dcol + lanes + (uint32_t)(kTN * a + c0), v);
          // the values are in registers: the accumulator is free for group g + 2
          fence_before();
          __syncwarp();
          if (lane == 0) mbar_arrive(aempty + 8u * a);
          const float sc = pow2f(-kDgW * g);
#pragma unroll
          for (int c = 0; c < 16; ++c) {
            const float x = v[c] * sc;
            if (g == 0) {
              s[c] = x;
              t[c] = 0.f;
            } else {
              float ss, er;
              two_sum(s[c], x, ss, er);
              s[c] = ss;
              t[c] += er;
            }
          }
        }
        ok = group_sync_and(ok, kBarD, kDrainW * 32);
        if (!ok) break;
        if (row_ok) {
#pragma unroll
          for (int c = 0; c < 16; ++c) {
            const int col = c0 + c;
            const dd v = dd_norm(s[c], t[c]);
            dd y(v.hi * cd[c], v.lo * cd[c]);
            if (scaled) {
              const dd yi = y * inv_sym_dd(sp, srow, tmus[col], tmus[kTN + col]);
              if (col < je) en.add(y, yi);
              y = yi;
            }
            yhi[r * kYS + col] = y.hi;
            ylo[r * kYS + col] = y.lo;
          }
        }
        group_sync(kBarD, kDrainW * 32);
        for (int idx = tid; idx < h * kTN; idx += kDrainW * 32) {
          const int rr = idx >> 5, c = idx & (kTN - 1);
          const int k = (P == 0) ? 2 * rr + 1 : 2 * rr + 2;
          if (c < je && k <= n)
            st_dd(out + (long long)(k - 1) * m + j0 + c, dd(yhi[rr * kYS + c], ylo[rr * kYS + c]));
        }
        group_sync(kBarD, kDrainW * 32);  // the staged rows and tmus are free again
      }
    }
    fence_before();
    ok = __syncthreads_and(ok ? 1 : 0) != 0;  // every role done: all MMAs of the phase drained
    fence_after();
  }
  if (warp == kDrainW + kBuildW && elect_one()) mma_commit(done);
  // after a timeout `done` tracks every MMA issued: tc_release_cols waits for it (bounded)
  tc_release_cols<512>(ok, true, done, 0u, false, 0u, 0u, tmem, S, true);
  if (scaled && tmode != TM_NONE) {
    const double e = (double)en.get();
    double tot;
    if (last_block_reduce<kNTG>(e, partials, &S->counter[CNT_TIME], gridDim.x, blockIdx.x, red,
                                &tot) &&
        tid == 0) {
      if (tmode == TM_INIT || tmode == TM_RESTART)
        minres_init_scalars_dev(S, tot);
      else
        minres_givens_dev(S, tot);
    }
  }
}

// The digits of sqrt(2/(n+1)) sin(pi a/(n+1)) 2^eS for a = 0 .. 2 n + 1
struct SineDigits {
  short d[kDg][2 * 257];
};

// The digit image of S_n for k_time_tcd: piece (parity P, digit i) at index P * 7 + i, the rows r of
// parity P (k = 2r+1 or 2r+2) by K = hK folded columns, canonical K-major fp16; the digits of S 2^eS
// (integers, |.| <= 2^7) were taken in float64, where they are exact.  A block per digit, parity and
// eight rows, a thread per row and eight columns (filled by the host and copied, the image took 0.2 to
// 0.5 ms of a handle's set-up).
__global__ void k_image_digits(const __grid_constant__ SineDigits S, int n, uint4 *img) {
  const int h = (n + 1) >> 1, hK = 8 * blockDim.y, dg = blockIdx.x, P = blockIdx.y;
  const int r = 8 * blockIdx.z + threadIdx.x, t0 = 8 * threadIdx.y, k = 2 * r + 1 + P;
  uint32_t w[8];
#pragma unroll
  for (int j = 0; j < 8; ++j) {
    const int a = (int)((unsigned)(k * (t0 + j + 1)) % (unsigned)(2 * (n + 1)));
    const int v = r < h && k <= n && t0 + j < h ? S.d[dg][a] : 0;
    const __half_raw x = __int2half_rn(v);
    w[j] = x.x;
  }
  img[((size_t)(P * kDg + dg) * kM * hK * 2 + canon_off(r, t0, hK)) / 16] =
      make_uint4(w[0] | w[1] << 16, w[2] | w[3] << 16, w[4] | w[5] << 16, w[6] | w[7] << 16);
}

}  // namespace

// Multiples of 32 up to 256, and every n from 129 to 256 (ceil(n/2) folded rows, padded to the MMA K
// step; seven S digits of half as many columns plus two 32-column accumulators within the 512
// tensor-memory columns; the layout within the 227 KB a block may opt into, with 1 KB of static
// shared memory).  At 127 x 255 spatial points, one P_H pass with this stage against the
// double-float CUDA-core one: n = 243 923 against 1751 us, n = 200 813 against 1270 (errors against
// float64 equal to 0.2%), but n = 100 521 against 531 and n = 50 377 against 236: between the
// multiples of 32 below 128 the CUDA cores stay.
bool time_tcd_supported(int n) {
  if (n < 32 || n > 256 || (n <= 128 && n % 32 != 0)) return false;
  if (kDg * (tcd_hk(n) / 2) + 2 * kTN > 512) return false;
  return tcd_layout(n).total + 1024u <= 227u * 1024u;
}

size_t time_tcd_bytes(int n) { return (size_t)2 * kDg * kM * (size_t)tcd_hk(n) * 2; }

int time_tcd_build(int n, unsigned char *img, cudaError_t *err) {
  const double PI = 3.14159265358979323846;
  const double sn = std::sqrt(2.0 / (n + 1));
  // S_{k,t} = sn sin(pi a / (n+1)) with a = k t mod 2 (n+1), and every a = 1..n occurs (t = 1)
  const int period = 2 * (n + 1);
  std::vector<double> val(period);
  double smax = 0.0;
  for (int a = 0; a < period; ++a) {
    val[a] = sn * std::sin(PI * (double)a / (n + 1));
    smax = std::fmax(smax, std::fabs(val[a]));
  }
  int E = 0;
  std::frexp(smax, &E);
  const int eS = 7 - E;  // smax 2^eS in [2^6, 2^7)
  SineDigits S;
  for (int a = 0; a < period; ++a) {
    double v = std::ldexp(val[a], eS);
    for (int dg = 0; dg < kDg; ++dg) {
      const double q = std::nearbyint(v);
      v = (v - q) * 128.0;
      S.d[dg][a] = (short)q;
    }
  }
  k_image_digits<<<dim3(kDg, 2, kM / 8), dim3(8, tcd_hk(n) >> 3)>>>(S, n, (uint4 *)img);
  *err = cudaGetLastError();
  return eS;
}

// scaled: scratch = (S_n data)/p with <v, P^-1 v> and the MINRES step; then data = S_n scratch
cudaError_t launch_time_tcd(dd *data, dd *scratch, const Geom &g, const Spec<dd> &sp,
                            const unsigned char *img, int eS, State *S, int tmode,
                            double *partials, int gk, cudaStream_t st) {
  // at least 116 KB of shared memory, so that one block runs per SM: each allocates all 512
  // tensor-memory columns
  uint32_t smem_bytes = tcd_layout(g.n).total;
  if (smem_bytes < 116u * 1024u) smem_bytes = 116u * 1024u;
  cudaError_t e = cudaFuncSetAttribute(k_time_tcd, cudaFuncAttributeMaxDynamicSharedMemorySize,
                                       (int)smem_bytes);
  if (e != cudaSuccess) return e;
  const long long ntiles = (g.m + kTN - 1) / kTN;
  int grid = time_tc_grid();
  if (ntiles < grid) grid = (int)ntiles;
  prof_begin(KC_TIME, st);
  k_time_tcd<<<grid, kNTG, smem_bytes, st>>>(data, scratch, g.n, g.m, g.mx, sp, img, eS, 1, S,
                                             tmode, partials, gk);
  k_time_tcd<<<grid, kNTG, smem_bytes, st>>>(scratch, data, g.n, g.m, g.mx, sp, img, eS, 0, S,
                                             TM_NONE, partials, gk);
  prof_end(st);
  return cudaGetLastError();
}

}  // namespace st
