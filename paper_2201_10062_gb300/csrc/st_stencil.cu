// Space-time stencil kernels: the flipped all-at-once operator Y T (Sec. 1, eq. theta and
// eq. main_system; Sec. 4, eq. matrix_gen / main_system_gem_sym), the all-at-once right-hand side
// and the face-coefficient gradient used by the adjoint.
//
// T is never stored.  Block row k of T v is A0 v_k + A1 v_{k-1} (+ A2 v_{k-2} for BDF2) with
//   theta: A0 = I + theta tau K, A1 = -I + (1-theta) tau K,
//   BDF2:  A0 = 3/2 I + tau K,   A1 = -2 I,  A2 = 1/2 I,
// and Y only reverses the block order, so row k of T v is written to block n-1-k.
// One thread owns one spatial node and walks a chunk of consecutive time levels (and their
// mirror images), carrying neighbouring planes in registers so that each plane of v is read once.
#include <algorithm>
#include <type_traits>

#include "st_internal.cuh"


namespace st {

namespace {

constexpr int kBX2 = 32, kBY2 = 8;   // 2D block: 32 x 8 nodes
constexpr int kBX1 = 256;            // 1D block: 256 nodes (all block reductions assume 256 threads)
constexpr int kNT = 256;

struct Tile {
  int kc, nchunk, gx, gy;
  int bx;  // threads along x (double-float stencil)
};

Tile tile_for(const Geom &g) {
  Tile t;
  if (g.dim == 1) {
    t.gx = (g.mx + kBX1 - 1) / kBX1;
    t.gy = 1;
  } else {
    // 2D blocks over x and the rows (y, and z in 3D)
    t.gx = (g.mx + kBX2 - 1) / kBX2;
    t.gy = (g.my * g.mz + kBY2 - 1) / kBY2;
  }
  // chunks cover the first ceil(n/2) planes (each thread also does their mirror images)
  const int half = (g.n + 1) / 2;
  const long long tiles = (long long)t.gx * t.gy;
  // default: 8 resident 256-thread blocks on each of 152 SMs; the autotuner may change it
  const long long target = g.st_target > 0 ? g.st_target : 152LL * 8;
  long long nchunk = (target + tiles - 1) / tiles;
  if (nchunk < 1) nchunk = 1;
  if (nchunk > half) nchunk = half;
  t.kc = (int)((half + nchunk - 1) / nchunk);
  t.nchunk = (half + t.kc - 1) / t.kc;
  return t;
}

// Weights of the double-float stencil: theta = 1/2, theta = 1, any other theta, BDF2
enum StencilWeights { W_HALF, W_ONE, W_ANY, W_BDF2 };

// Resident blocks of the double-float stencil on an SM.  A uniform coefficient leaves room for
// three (80 registers; 63.6 -> 58.1 us at 255^2 x 256); with a coefficient per face, or 7 points,
// three would spill (511^2 x 128, BDF2: 166 us with two, 182 with three).
constexpr int df_blocks(int dim, bool uni) { return uni && dim < 3 ? 3 : 2; }

// Double-float stencil: two x neighbours a thread, df_blocks blocks on each of 152 SMs.  Of the
// chunk lengths the one with the least waves x (levels + 2) is taken: a chunk starts with two
// extra planes, and a last wave that is nearly empty costs as much as a full one.
Tile tile_df_for(const Geom &g) {
  const int nb = df_blocks(g.dim, g.c_uniform);
  Tile t;
  t.bx = (g.dim == 1) ? kBX1 : std::min(kBX2, g.px / 2);
  t.gx = (g.px / 2 + t.bx - 1) / t.bx;
  t.gy = (g.my * g.mz + kNT / t.bx - 1) / (kNT / t.bx);
  const int half = (g.n + 1) / 2;
  const long long tiles = (long long)t.gx * t.gy;
  if (g.st_target > 0) {
    const long long nchunk = std::min<long long>(half, (g.st_target + tiles - 1) / tiles);
    t.kc = (int)((half + nchunk - 1) / nchunk);
  } else {
    long long best = -1;
    t.kc = half;
    for (int kc = half; kc >= 1; --kc) {
      const long long blocks = tiles * ((half + kc - 1) / kc);
      if (blocks > 2432 && best >= 0) break;
      const long long cost = ((blocks + 152 * nb - 1) / (152 * nb)) * (kc + 2);
      if (best < 0 || cost < best) {
        best = cost;
        t.kc = kc;
      }
    }
  }
  t.nchunk = (half + t.kc - 1) / t.kc;
  return t;
}

template <class Tz>
__device__ __forceinline__ double ld(const Tz *p) {
  return (double)__ldg(p);
}

// tau*K applied at node p = (i, jy, jz) of plane base (zero Dirichlet values outside the grid);
// f holds the node's face coefficients (zero along absent axes, so 1D and 2D add exact zeros).
template <class Tz>
__device__ __forceinline__ double tauK(const Tz *__restrict__ base, long long p, int i, int jy,
                                       int jz, const Geom &g, const Faces6<double> &f, double c) {
  double r = (f.w + f.e + f.s + f.n + f.d + f.u) * c;
  if (i > 0) r -= f.w * ld(base + p - 1);
  if (i < g.mx - 1) r -= f.e * ld(base + p + 1);
  if (g.dim >= 2) {
    if (jy > 0) r -= f.s * ld(base + p - g.mx);
    if (jy < g.my - 1) r -= f.n * ld(base + p + g.mx);
  }
  if (g.dim == 3) {
    const long long pl = (long long)g.mx * g.my;
    if (jz > 0) r -= f.d * ld(base + p - pl);
    if (jz < g.mz - 1) r -= f.u * ld(base + p + pl);
  }
  return r;
}

// The dot products MINRES needs pair the two halves of the time axis: row k of T z lands in
// block n-1-k of Y T z, so <Y T z, z> = sum_k <(T z)_k, z_{n-1-k}>.  Each thread therefore walks
// a chunk of planes k upwards (side A) and the mirrored planes n-1-k downwards (side B) in lock
// step; the centre value of each side is exactly the z the other side's output is paired with,
// so the dot costs no extra loads.  Chunks cover the first ceil(n/2) planes; for odd n the middle
// plane is its own mirror and is done once.
__device__ __forceinline__ void put(double *p, double v) { *p = v; }
__device__ __forceinline__ void put(df *p, double v) { *p = df_of_double(v); }

template <class Tz, int MODE, class TO = double>
__global__ void __launch_bounds__(kNT) k_stencil(Geom g, const Tz *__restrict__ z,
                                                 TO *__restrict__ out,
                                                 const double *__restrict__ fH, State *S,
                                                 double *__restrict__ partials, int kc) {
  __shared__ double red[32];
  if (MODE == SM_MINRES) {
    if (!S->active) return;
    if (S->finish) {
      if (blockIdx.x == 0 && blockIdx.y == 0 && blockIdx.z == 0 && flat_tid() == 0) S->active = 0;
      return;
    }
  }
  if (MODE == SM_RESID_OUTER && !(S->finish && !S->done)) return;
  const int i = blockIdx.x * blockDim.x + threadIdx.x;
  const int j = blockIdx.y * blockDim.y + threadIdx.y;  // row jz*my + jy
  const int mx = g.mx, n = g.n;
  const long long m = g.m;
  const bool valid = (i < mx) && (j < g.my * g.mz);
  const int half = (n + 1) >> 1;
  const int k0 = blockIdx.z * kc;
  const int k1 = min(half, k0 + kc);
  const double s = (MODE == SM_MINRES) ? S->inv_beta : 1.0;
  double acc = 0.0;
  if (valid) {
    const int jz = j / g.my, jy = j - jz * g.my;
    const long long p = (long long)j * mx + i;
    const long long po = std::is_same<TO, df>::value ? (long long)j * g.px + i : p;
    const Faces6<double> fc = faces_at(g, i, jy, jz);
    const double th = g.theta, omth = 1.0 - g.theta;
    auto center = [&](int k) -> double { return ld(z + (long long)k * m + p); };
    auto stiff = [&](int k, double c) -> double {
      return tauK(z + (long long)k * m, p, i, jy, jz, g, fc, c);
    };
    // side A (ascending) carries plane kA-1 (and kA-2); side B (descending) carries plane kB and
    // the planes below it
    double a1 = 0.0, aK1 = 0.0, a2 = 0.0;
    double b0 = 0.0, bK0 = 0.0, b1 = 0.0;
    const bool theta = (g.scheme == ST_THETA);
    if (k0 > 0) {
      a1 = center(k0 - 1);
      if (theta) aK1 = stiff(k0 - 1, a1);
    }
    if (!theta && k0 > 1) a2 = center(k0 - 2);
    {
      const int kb = n - 1 - k0;
      b0 = center(kb);
      if (theta) bK0 = stiff(kb, b0);
      else if (kb > 0) b1 = center(kb - 1);
    }
    for (int kA = k0; kA < k1; ++kA) {
      const int kB = n - 1 - kA;
      const double cA = center(kA);
      const double KA = stiff(kA, cA);
      double yA;
      if (theta) {
        yA = (cA - a1) + th * KA + omth * aK1;
        a1 = cA;
        aK1 = KA;
      } else {
        yA = 1.5 * cA - 2.0 * a1 + 0.5 * a2 + KA;
        a2 = a1;
        a1 = cA;
      }
      const bool twin = (kB != kA);
      double yB = 0.0;
      const double zB = twin ? b0 : cA;  // z in plane kB, partner of yA
      if (twin) {
        if (theta) {
          double nb = 0.0, nK = 0.0;
          if (kB > 0) {
            nb = center(kB - 1);
            nK = stiff(kB - 1, nb);
          }
          yB = (b0 - nb) + th * bK0 + omth * nK;
          b0 = nb;
          bK0 = nK;
        } else {
          const double KB = stiff(kB, b0);
          const double nb2 = (kB > 1) ? center(kB - 2) : 0.0;
          yB = 1.5 * b0 - 2.0 * b1 + 0.5 * nb2 + KB;
          b0 = b1;
          b1 = nb2;
        }
      }
      // block n-1-kA receives row kA, block n-1-kB = kA row kB (double-float output is padded)
      const long long mo = std::is_same<TO, df>::value ? g.mp : m;
      const long long oA = (long long)kB * mo + po;
      const long long oB = (long long)kA * mo + po;
      if (MODE == SM_MINRES) {
        yA *= s;
        put(out + oA, yA);
        acc += yA * (zB * s);
        if (twin) {
          yB *= s;
          put(out + oB, yB);
          acc += yB * (cA * s);
        }
      } else if (MODE == SM_APPLY) {
        put(out + oA, yA);
        if (twin) put(out + oB, yB);
      } else {  // SM_RESID(_OUTER): r = Y f_H - Y T x; block n-1-k of Y f_H is f_H block k
        const double rA = fH[(long long)kA * m + p] - yA;
        if (out) put(out + oA, rA);
        acc += rA * rA;
        if (twin) {
          const double rB = fH[(long long)kB * m + p] - yB;
          if (out) put(out + oB, rB);
          acc += rB * rB;
        }
      }
    }
  }
  if (MODE == SM_MINRES || MODE == SM_RESID || MODE == SM_RESID_OUTER) {
    const int nb = gridDim.x * gridDim.y * gridDim.z;
    const int bid = blockIdx.x + gridDim.x * (blockIdx.y + gridDim.y * blockIdx.z);
    double tot;
    unsigned int *cnt = &S->counter[MODE == SM_MINRES ? CNT_STENCIL : CNT_RESID];
    if (last_block_reduce<kNT>(acc, partials, cnt, nb, bid, red, &tot) && flat_tid() == 0) {
      if (MODE == SM_MINRES) {
        S->alpha = tot;
        S->lz_a = tot / S->beta;
        S->lz_b = (S->k > 0) ? S->beta / S->beta_prev : 0.0;
        refresh_df(S);
      } else {
        S->rnorm2 = tot;
        if (MODE == SM_RESID_OUTER) {
          // refinement decision (mirrors the host-driven mixed solve)
          const double rho = (S->bnorm2 > 0.0) ? sqrt(tot / S->bnorm2) : 0.0;
          S->rho = rho;
          S->total += S->k;
          S->outer += 1;
          if (rho <= S->tol_outer) {
            S->done = 1;
          } else if (S->status != 0 || S->total >= S->maxit_total || S->k == 0) {
            S->done = 1;
            if (S->status == 0) S->status = ST_ERR_NOT_CONVERGED;
          } else {
            const double t = 0.5 * S->tol_outer / rho;
            S->target = t > S->inner_floor ? t : S->inner_floor;
            S->maxit = S->maxit_total - S->total;
            S->k = 0;
            S->upd = 0;  // the grouped update of the new inner run starts from iteration 1
            S->finish = 0;
            S->active = 0;
            S->restart = 1;
          }
        }
      }
    }
  }
}

// ------------------------------------------------------------------ double-float stencil
// Mixed-precision MINRES: z_k is float32, the output Y T z_k is a double-float; the 1/beta_k
// of p = Y T z_k / beta_k is applied by the pass that reads it (SrcLanczos over double-floats).
// Every face term a_f (z_c - z_f) uses the exact float difference (TwoSum) and a TwoProd
// product with the double-float coefficient, and the terms are summed with the high parts
// added error-free, so the result carries ~46 significant bits with no float64 instruction per
// element (GB300 runs float64 at 1/64 of the float32 rate).  Same mirrored-plane walk as the
// float64 kernel; the dot <Y T z, z> is accumulated unscaled and scaled by 1/beta^2 at the end.
// Two float32 values in one 64-bit register pair.  sm_100 and later issue add, sub, mul and fma on
// such pairs as one instruction, each half rounded as the scalar instruction rounds it.
struct f2 {
  unsigned long long v;
};
__device__ __forceinline__ f2 pack2(float a, float b) {
  f2 r;
  asm("mov.b64 %0, {%1, %2};" : "=l"(r.v) : "f"(a), "f"(b));
  return r;
}
__device__ __forceinline__ f2 dup2(float a) { return pack2(a, a); }
__device__ __forceinline__ void unpack2(f2 a, float &x, float &y) {
  asm("mov.b64 {%0, %1}, %2;" : "=f"(x), "=f"(y) : "l"(a.v));
}
__device__ __forceinline__ f2 operator+(f2 a, f2 b) {
  f2 r;
  asm("add.rn.f32x2 %0, %1, %2;" : "=l"(r.v) : "l"(a.v), "l"(b.v));
  return r;
}
__device__ __forceinline__ f2 operator-(f2 a, f2 b) {
  f2 r;
  asm("sub.rn.f32x2 %0, %1, %2;" : "=l"(r.v) : "l"(a.v), "l"(b.v));
  return r;
}
__device__ __forceinline__ f2 operator*(f2 a, f2 b) {
  f2 r;
  asm("mul.rn.f32x2 %0, %1, %2;" : "=l"(r.v) : "l"(a.v), "l"(b.v));
  return r;
}
__device__ __forceinline__ f2 fma2(f2 a, f2 b, f2 c) {
  f2 r;
  asm("fma.rn.f32x2 %0, %1, %2, %3;" : "=l"(r.v) : "l"(a.v), "l"(b.v), "l"(c.v));
  return r;
}

// Two double-float numbers, and a constant one with its high part negated besides: -(a b) is then
// a product, and every difference below is a subtraction, so no sign is flipped on the way.
struct df2 {
  f2 hi, lo;
};
struct cf2 {
  f2 hi, lo, nhi;
};
__device__ __forceinline__ cf2 cf2_of(df a, df b, float w = 1.f) {
  return cf2{pack2(w * a.hi, w * b.hi), pack2(w * a.lo, w * b.lo), pack2(-w * a.hi, -w * b.hi)};
}
__device__ __forceinline__ df2 df2_from_sum(f2 s, f2 t) {
  const f2 hi = s + t;
  return df2{hi, t - (hi - s)};
}

// running double-float sums (see st_df.cuh), two at a time
struct acc2 {
  f2 s, t;
  __device__ __forceinline__ f2 sum(f2 p) {  // s += p, returns the rounding error
    const f2 ss = s + p, bb = ss - s;
    const f2 err = (s - (ss - bb)) + (p - bb);
    s = ss;
    return err;
  }
  __device__ __forceinline__ f2 diff(f2 np) {  // s -= np, returns the rounding error
    const f2 ss = s - np, bb = ss - s;
    const f2 err = (s - (ss - bb)) - (np + bb);
    s = ss;
    return err;
  }
  __device__ __forceinline__ void add(df2 a) {
    const f2 err = sum(a.hi);
    t = t + (err + a.lo);
  }
  __device__ __forceinline__ void add1(f2 p) {
    const f2 err = sum(p);
    t = t + err;
  }
  __device__ __forceinline__ void sub1(f2 p) {
    const f2 err = diff(p);
    t = t + err;
  }
  // add c b
  __device__ __forceinline__ void add_prod(cf2 c, df2 b) {
    const f2 np = c.nhi * b.hi;
    const f2 e = fma2(c.hi, b.lo, fma2(c.lo, b.hi, fma2(c.hi, b.hi, np)));
    const f2 err = diff(np);
    t = t + (err + e);
  }
  // add a b, nb = -b
  __device__ __forceinline__ void add_prod(df2 a, f2 b, f2 nb) {
    const f2 np = a.hi * nb;
    const f2 e = fma2(a.lo, b, fma2(a.hi, b, np));
    const f2 err = diff(np);
    t = t + (err + e);
  }
  __device__ __forceinline__ df2 get() const { return df2_from_sum(s, t); }
};

// A thread owns two x neighbours (i even; the slot after a line's last node is its padding, whose
// result is zero), and every double-float operation acts on both at once.
// One node a thread with scalar instructions was bound by instruction issue: about 167 instructions
// per unknown, 83% of the issue slots.  The pair takes 79 and shares the loads (8 bytes each but
// for the two outer x neighbours), the addresses, which advance by a level instead of being formed
// from k, and the loop; what bounds it now is latency (45% of the issue slots: waits for the loads
// of the next level, the float32 pipe and dependent sums, ncu).  Before and now, us a launch:
// 255^2 x 256 uniform, theta = 1/2: 86 and 58; 63^3 x 64 uniform: 105 and 73; 511^2 x 128 BDF2,
// varying coefficient: 207 and 166; 255^2 x 128 varying, theta = 1: 60 and 49.
// DIM 1, 2, 3: the 3-, 5- or 7-point stencil (planes px my apart in 3D).
// UNI: every face coefficient has the same value c (a constant coefficient on a grid with equal
// spacing along every axis, g.c_uniform): tau K z = c (f z_c - sum_f z_f) over the f faces of the
// node, so the face terms reduce to one exactly summed difference (TwoSum chain over floats) and
// one double-float product, in place of one product per face.
template <int DIM, bool UNI, int W>
__global__ void __launch_bounds__(kNT, df_blocks(DIM, UNI)) k_stencil_df(Geom g, const float *__restrict__ z,
                                                       df *__restrict__ out, State *S,
                                                       double *__restrict__ partials, int kc) {
  __shared__ double red[32];
  if (!S->active) return;
  const bool lead = blockIdx.x == 0 && blockIdx.y == 0 && blockIdx.z == 0 && flat_tid() == 0;
  if (S->finish) {
    if (lead) S->active = 0;
    return;
  }
  // first iteration after a device-side restart: the restart pass is complete
  if (lead && S->restart) S->restart = 0;
  constexpr bool THETA = W != W_BDF2;
  const int i = 2 * (blockIdx.x * blockDim.x + threadIdx.x);
  const int j = blockIdx.y * blockDim.y + threadIdx.y;  // row jz*my + jy
  // z and out are padded: px slots a line, m a level
  const int mx = g.mx, my = g.my, n = g.n, px = g.px;
  const long long m = g.mp, pl = (long long)px * my;
  const bool valid = (i < mx) && (j < my * g.mz);
  const int half = (n + 1) >> 1;
  const int k0 = blockIdx.z * kc;
  const int k1 = min(half, k0 + kc);
  const f2 O = dup2(0.f), neg1 = dup2(-1.f);
  acc2 D{O, O};
  if (valid) {
    const int jz = DIM == 3 ? j / my : 0, jy = j - jz * my;
    const long long p = (long long)j * px + i;
    const bool two = i + 1 < mx;  // the second slot is a node
    const bool hs = DIM >= 2 && jy > 0, hn = DIM >= 2 && jy < my - 1;
    const bool hd = DIM == 3 && jz > 0, hu = DIM == 3 && jz < g.mz - 1;
    cf2 cw, ce, cs, cn, cd, cu;
    // theta = 1/2 scales the coefficients, an exact scaling
    const float sc = W == W_HALF ? 0.5f : 1.f;
    if (UNI) {
      cw = cf2_of(g.c_uni, g.c_uni, sc);
    } else {
      const Faces6<df> a = faces_df_at(g, i, jy, jz), b = two ? faces_df_at(g, i + 1, jy, jz) : a;
      cw = cf2_of(a.w, b.w, sc);
      ce = cf2_of(a.e, b.e, sc);
      cs = cf2_of(a.s, b.s, sc);
      cn = cf2_of(a.n, b.n, sc);
      cd = cf2_of(a.d, b.d, sc);
      cu = cf2_of(a.u, b.u, sc);
    }
    const df2 zero{O, O};
    auto center = [&](const float *b) -> f2 {
      return f2{__ldg(reinterpret_cast<const unsigned long long *>(b))};
    };
    auto combine = [&](f2 c, f2 c1, f2 c2, df2 Kc, df2 K1) -> df2 {
      acc2 A;
      if (THETA) {
        // the exact difference c - c1 starts the sum
        A.s = c;
        A.t = A.diff(c1);
        if (W == W_ANY) {
          A.add_prod(cf2_of(g.th_d, g.th_d), Kc);
          A.add_prod(cf2_of(g.omth_d, g.omth_d), K1);
        } else {
          A.add(Kc);
          if (W == W_HALF) A.add(K1);
        }
      } else {
        const f2 h = dup2(1.5f), np = dup2(-1.5f) * c;
        A.s = O - np;
        A.t = fma2(h, c, np);
        A.sub1(dup2(2.0f) * c1);
        A.add1(dup2(0.5f) * c2);
        A.add(Kc);
      }
      return A.get();
    };
    // The loads of iteration kA + 1 (stencil points of both walks) are issued before the
    // arithmetic of iteration kA, so their latency overlaps it.
    struct P5 {
      f2 c, s, n, d, u;
      float w, e;  // west of the first node, east of the second
    };
    const P5 none{O, O, O, O, O, 0.f, 0.f};
    auto load5 = [&](const float *b) -> P5 {
      P5 r = none;
      r.c = center(b);
      r.w = __ldg(b - 1);  // the padding slots on either side of a line hold the boundary's zeros
      if (two) r.e = __ldg(b + 2);
      if (hs) r.s = center(b - px);
      if (hn) r.n = center(b + px);
      if (hd) r.d = center(b - pl);
      if (hu) r.u = center(b + pl);
      return r;
    };
    auto face = [&](acc2 &A, cf2 a, f2 c, f2 q) {
      const f2 dh = c - q, bb = dh - c;
      const f2 dl = (c - (dh - bb)) - (q + bb);
      A.add_prod(a, df2{dh, dl});
    };
    // tau K at a plane: the face terms in a fixed order
    auto stiff = [&](const P5 &q) -> df2 {
      float c0, c1;
      unpack2(q.c, c0, c1);
      const f2 w = pack2(q.w, c0), e = pack2(c1, q.e);
      if (UNI) {
        // c_uni (f z_c - z_w - z_e - ...): f z_c is exact (f = 2, 4, or 4 + 2 in 3D)
        acc2 A{dup2(DIM >= 2 ? 4.f : 2.f) * q.c, O};
        if (DIM == 3) A.add1(dup2(2.f) * q.c);
        A.sub1(w);
        A.sub1(e);
        if (DIM >= 2) {
          A.sub1(q.s);
          A.sub1(q.n);
        }
        if (DIM == 3) {
          A.sub1(q.d);
          A.sub1(q.u);
        }
        const df2 x = A.get();
        const f2 np = cw.nhi * x.hi;
        const f2 r = fma2(cw.hi, x.lo, fma2(cw.lo, x.hi, fma2(cw.hi, x.hi, np)));
        return df2{O - np, r};  // r is an ulp of the product or so: the sums it enters take it as it is
      }
      acc2 A{O, O};
      face(A, cw, q.c, w);
      face(A, ce, q.c, e);
      if (DIM >= 2) {
        face(A, cs, q.c, q.s);
        face(A, cn, q.c, q.n);
      }
      if (DIM == 3) {
        face(A, cd, q.c, q.d);
        face(A, cu, q.c, q.u);
      }
      return A.get();
    };
    auto store = [&](df *o, df2 y) {
      float h0, h1, l0, l1;
      unpack2(y.hi, h0, h1);
      unpack2(y.lo, l0, l1);
      *reinterpret_cast<float4 *>(o) = make_float4(h0, l0, h1, l1);
    };
    // the padding slot's result is zero
    auto masked = [&](df2 y) -> df2 {
      float h0, h1, l0, l1;
      unpack2(y.hi, h0, h1);
      unpack2(y.lo, l0, l1);
      return df2{pack2(h0, two ? h1 : 0.f), pack2(l0, two ? l1 : 0.f)};
    };
    f2 a1 = O, a2 = O, b0, b1 = O;
    df2 aK1 = zero, bK0 = zero;
    // planes kA = k0 (upwards) and kB = n - 1 - k0 (downwards), and the outputs of their rows
    const float *zA = z + (long long)k0 * m + p, *zB = z + (long long)(n - 1 - k0) * m + p;
    df *oA = out + (long long)(n - 1 - k0) * m + p, *oB = out + (long long)k0 * m + p;
    if (k0 > 0) {
      a1 = center(zA - m);
      if (THETA) aK1 = stiff(load5(zA - m));
    }
    if (!THETA && k0 > 1) a2 = center(zA - 2 * m);
    b0 = center(zB);
    if (THETA) bK0 = stiff(load5(zB));
    else if (n - 1 - k0 > 0) b1 = center(zB - m);
    // planes read by iteration kA: A-walk plane kA; mirrored walk plane kB - 1 (theta) or kB
    // plus the centre of kB - 2 (BDF2)
    auto planes = [&](int kA, P5 &A, P5 &B, f2 &C) {
      const int kB = n - 1 - kA;
      A = load5(zA);
      B = none;
      C = O;
      if (kB != kA) {
        if (THETA) {
          B = load5(zB - m);
        } else {
          B = load5(zB);
          if (kB > 1) C = center(zB - 2 * m);
        }
      }
      zA += m;
      zB -= m;
    };
    P5 pA = none, pB = none;
    f2 pC = O;
    if (k0 < k1) planes(k0, pA, pB, pC);
    // Both walks' arithmetic is one straight piece of code (kB > kA, so kB > 0), so that their two
    // dependent chains overlap; the middle plane of an odd n, its own mirror, follows the loop.
    const int k2 = min(k1, n >> 1);
    for (int kA = k0; kA < k2; ++kA) {
      P5 nA = none, nB = none;
      f2 nC = O;
      if (kA + 1 < k1) planes(kA + 1, nA, nB, nC);
      const f2 cA = pA.c;
      const df2 KA = stiff(pA), KB = stiff(pB);
      const df2 yA = masked(combine(cA, a1, a2, KA, aK1));
      const df2 yB = masked(THETA ? combine(b0, pB.c, O, bK0, KB) : combine(b0, b1, pC, KB, zero));
      D.add_prod(yA, b0, b0 * neg1);  // b0: z in plane kB, partner of yA
      D.add_prod(yB, cA, cA * neg1);
      store(oA, yA);
      store(oB, yB);
      oA -= m;
      oB += m;
      if (THETA) {
        aK1 = KA;
        bK0 = KB;
        b0 = pB.c;
      } else {
        a2 = a1;
        b0 = b1;
        b1 = pC;
      }
      a1 = cA;
      pA = nA;
      pB = nB;
      pC = nC;
    }
    if (k2 < k1) {
      const df2 y = masked(combine(pA.c, a1, a2, stiff(pA), aK1));
      store(oA, y);
      D.add_prod(y, pA.c, pA.c * neg1);
    }
  }
  float s0, s1, t0, t1;
  unpack2(D.s, s0, s1);
  unpack2(D.t, t0, t1);
  const double acc = ((double)s0 + (double)s1) + ((double)t0 + (double)t1);
  const int nb = gridDim.x * gridDim.y * gridDim.z;
  const int bid = blockIdx.x + gridDim.x * (blockIdx.y + gridDim.y * blockIdx.z);
  double tot;
  if (last_block_reduce<kNT>(acc, partials, &S->counter[CNT_STENCIL], nb, bid, red, &tot) &&
      flat_tid() == 0) {
    const double sd = S->inv_beta;
    const double alpha = tot * sd * sd;
    S->alpha = alpha;
    S->lz_a = alpha / S->beta;
    S->lz_b = (S->k > 0) ? S->beta / S->beta_prev : 0.0;
    refresh_df(S);
  }
}

// Time levels per thread of the right-hand-side and gradient kernels: a thread keeps one node and
// walks this many levels, so a level's plane is read once per chunk (and not once as f^(k) and once
// as f^(k-1)), and no index is recovered by a division (assembly, its adjoint and the face
// gradients at 255^2 x 128: 369 -> 250 us for the three calls; one element per thread with a 64-bit
// division each, and one unchunked walk for the faces, before).
constexpr int kRhsLevels = 16;

// f_H (Sec. 1 for theta, Sec. 4 with the start-up history moved into blocks 1-2 for BDF2).
// Bound by memory (24 bytes per unknown with an extra term) and, close behind, by the float64
// pipe: two fused multiply-adds per unknown, one where 1 - theta = 0.  Nodes by the first grid
// axis, chunks of kRhsLevels levels by the second.
template <bool EXTRA>
__global__ void __launch_bounds__(256)
    k_rhs(Geom g, const double *__restrict__ f, const double *__restrict__ u0,
          const double *__restrict__ uprev, const double *__restrict__ extra,
          double *__restrict__ fH) {
  const long long m = g.m;
  const long long p = blockIdx.x * 256LL + threadIdx.x;
  if (p >= m) return;
  const int k0 = blockIdx.y * kRhsLevels, k1 = min(g.n, k0 + kRhsLevels);
  const bool theta = g.scheme == ST_THETA;
  const double a = theta ? g.theta * g.tau : g.tau;
  const double b = theta ? (1.0 - g.theta) * g.tau : 0.0;
  const bool two = theta && g.theta != 1.0;  // f^(k-1) enters block k
  const double *fp = f + (long long)k0 * m + p;
  const double *ep = EXTRA ? extra + (long long)k0 * m + p : nullptr;
  double *op = fH + (long long)k0 * m + p;
  double f0 = two ? __ldg(fp) : 0.0;
#pragma unroll 4
  for (int k = k0; k < k1; ++k, op += m) {
    fp += m;
    const double f1 = __ldg(fp);
    double r = EXTRA ? __ldg(ep) : 0.0;
    if (EXTRA) ep += m;
    if (two) r = EXTRA ? fma(b, f0, r) : b * f0;
    r = (two || EXTRA) ? fma(a, f1, r) : a * f1;
    f0 = f1;
    if (theta) {
      if (k == 0) {
        const int i = (int)(p % g.mx), row = (int)(p / g.mx);
        const int jz = row / g.my, jy = row - jz * g.my;
        const double c = u0[p];
        const double Kc = tauK(u0, p, i, jy, jz, g, faces_at(g, i, jy, jz), c);
        r += c - (1.0 - g.theta) * Kc;
      }
    } else {
      if (k == 0) r += 2.0 * u0[p] - 0.5 * (uprev ? uprev[p] : u0[p]);
      if (k == 1) r -= 0.5 * u0[p];
    }
    *op = r;
  }
}

// Adjoint of the right-hand-side assembly: given lam = dL/df_H, the gradients with respect to
// f (at t_0..t_n), u0 and (BDF2) u^(-1).
//   theta: f_H block k = theta tau f^(k) + (1-theta) tau f^(k-1), block 1 += (I - (1-theta) tau K) u0
//   BDF2:  f_H block k = tau f^(k), block 1 += 2 u0 - u^(-1)/2, block 2 += -u0/2
// Same walk as k_rhs, over the n + 1 levels of f.
__global__ void __launch_bounds__(256)
    k_grad_rhs(Geom g, const double *__restrict__ lam, double *__restrict__ gf,
               double *__restrict__ gu0, double *__restrict__ gup) {
  const long long m = g.m;
  const long long p = blockIdx.x * 256LL + threadIdx.x;
  if (p >= m) return;
  const int n = g.n;
  const int k0 = blockIdx.y * kRhsLevels, k1 = min(n + 1, k0 + kRhsLevels);
  const bool theta = g.scheme == ST_THETA;
  const double a = theta ? g.theta * g.tau : g.tau;
  const double b = theta ? (1.0 - g.theta) * g.tau : 0.0;
  const bool two = theta && g.theta != 1.0;
  const double *lp = lam + (long long)k0 * m + p;
  double *op = gf + (long long)k0 * m + p;
  double l0 = k0 > 0 ? __ldg(lp - m) : 0.0;  // block k - 1 (0-based), paired with theta tau
#pragma unroll 4
  for (int k = k0; k < k1; ++k, lp += m, op += m) {
    const double l1 = k < n ? __ldg(lp) : 0.0;
    double r = a * l0;
    if (two) r = fma(b, l1, r);
    *op = r;
    l0 = l1;
    if (k == 0) {
      if (theta) {
        if (gu0) {
          const int i = (int)(p % g.mx), row = (int)(p / g.mx);
          const int jz = row / g.my, jy = row - jz * g.my;
          const double Kl = tauK(lam, p, i, jy, jz, g, faces_at(g, i, jy, jz), l1);
          gu0[p] = l1 - (1.0 - g.theta) * Kl;
        }
        if (gup) gup[p] = 0.0;
      } else {
        const double l2 = (n > 1) ? lam[m + p] : 0.0;
        if (gu0) gu0[p] = 2.0 * l1 - 0.5 * l2;
        if (gup) gup[p] = -0.5 * l1;
      }
    }
  }
}

// Face terms of dL/da: g_face = -(tau/h^2) sum_k (lam_p - lam_q)(w_p - w_q), with
// w_k = theta u_k + (1-theta) u_{k-1} (u_{-1} = u0) for theta and w_k = u_k for BDF2.
// Thread (j, i) of the (my+1) x (mx+1) face grid owns x-face (j, i) [between nodes (j,i-1) and
// (j,i)] when j < my and y-face (j, i) [between (j-1,i) and (j,i)] when i < mx.
// cx/cy already hold tau*a/h^2; a_face enters linearly, so tau/h^2 = c/a_face is recovered from
// the unit-coefficient spacing passed in sx, sy.
//
// Bound by the float64 pipe: with E = lam_p - lam_q and D = u_p - u_q the sum over k is
// theta sum E_k D_k + (1 - theta) sum E_k D_{k-1}, so a face takes two differences and two fused
// multiply-adds per level (one where theta = 1 or BDF2) and w is never formed.  The levels are
// cut into chunks over the grid's third axis (a 255^2 grid alone has fewer threads than the chip
// holds); every chunk writes its own partial face sums, [chunk][face], added in order by
// k_grad_nodes.
template <bool TWO>
__global__ void __launch_bounds__(256)
    k_grad_faces(Geom g, const double *__restrict__ lam, const double *__restrict__ u,
                 const double *__restrict__ u0, double sx, double sy, int kc,
                 double *__restrict__ gx, double *__restrict__ gy) {
  const int i = blockIdx.x * blockDim.x + threadIdx.x;
  const int j = blockIdx.y * blockDim.y + threadIdx.y;
  const int mx = g.mx, my = g.my;
  if (i > mx || j > my) return;
  const long long m = g.m;
  const bool doX = (j < my);
  const bool doY = (g.dim == 2) && (i < mx);
  if (!doX && !doY) return;
  const double th = (g.scheme == ST_THETA) ? g.theta : 1.0;
  // a node outside the grid has value zero; pc, pl, pd: the face's own node and its west and
  // south neighbours
  const bool hc = i < mx && j < my, hl = i > 0 && j < my, hd = j > 0 && i < mx;
  const long long pc = (long long)j * mx + i, pl = pc - 1, pd = pc - mx;
  const int k0 = blockIdx.z * kc, k1 = min(g.n, k0 + kc);
  double dx = 0.0, dy = 0.0;  // D of the level before
  if (TWO) {
    const double *U = k0 > 0 ? u + (long long)(k0 - 1) * m : u0;
    const double uc = hc ? U[pc] : 0.0;
    dx = uc - (hl ? U[pl] : 0.0);
    dy = uc - (hd ? U[pd] : 0.0);
  }
  double ax = 0.0, ay = 0.0, bx = 0.0, by = 0.0;
  const double *L = lam + (long long)k0 * m, *U = u + (long long)k0 * m;
#pragma unroll 2
  for (int k = k0; k < k1; ++k, L += m, U += m) {
    const double uc = hc ? __ldg(U + pc) : 0.0, lc = hc ? __ldg(L + pc) : 0.0;
    if (doX) {
      const double e = lc - (hl ? __ldg(L + pl) : 0.0), d = uc - (hl ? __ldg(U + pl) : 0.0);
      ax = fma(e, d, ax);
      if (TWO) bx = fma(e, dx, bx);
      dx = d;
    }
    if (doY) {
      const double e = lc - (hd ? __ldg(L + pd) : 0.0), d = uc - (hd ? __ldg(U + pd) : 0.0);
      ay = fma(e, d, ay);
      if (TWO) by = fma(e, dy, by);
      dy = d;
    }
  }
  if (TWO) {
    ax = th * ax + (1.0 - th) * bx;
    ay = th * ay + (1.0 - th) * by;
  }
  const long long fx = (long long)(mx + 1) * my, fy = (long long)mx * (my + 1);
  if (doX) gx[blockIdx.z * fx + (long long)j * (mx + 1) + i] = -sx * ax;
  if (doY) gy[blockIdx.z * fy + (long long)j * mx + i] = -sy * ay;
}

// Nodal gradient: each face gradient (the sum of its chunks' partial sums, in order) is split
// half/half between its two nodes.
__global__ void k_grad_nodes(int dim, int mx, int my, int nchunk, const double *__restrict__ gx,
                             const double *__restrict__ gy, double *__restrict__ grad) {
  const long long nfx = (long long)(mx + 1) * my, nfy = (long long)mx * (my + 1);
  auto sum = [&](const double *p, long long stride) -> double {
    double s = p[0];
    for (int c = 1; c < nchunk; ++c) s += p[c * stride];
    return s;
  };
  const int I = blockIdx.x * blockDim.x + threadIdx.x;  // 0..mx+1
  const int J = blockIdx.y * blockDim.y + threadIdx.y;  // 0..my+1 (0 in 1D)
  if (dim == 1) {
    if (I > mx + 1 || J > 0) return;
    double s = 0.0;
    if (I <= mx) s += 0.5 * sum(gx + I, nfx);      // face I: between nodes I and I+1
    if (I >= 1) s += 0.5 * sum(gx + I - 1, nfx);   // face I-1: between nodes I-1 and I
    grad[I] = s;
    return;
  }
  if (I > mx + 1 || J > my + 1) return;
  double s = 0.0;
  // x-faces lie on interior rows j = J-1; face (j, i) joins nodal columns i and i+1
  if (J >= 1 && J <= my) {
    const int j = J - 1;
    if (I <= mx) s += 0.5 * sum(gx + (long long)j * (mx + 1) + I, nfx);
    if (I >= 1) s += 0.5 * sum(gx + (long long)j * (mx + 1) + I - 1, nfx);
  }
  // y-faces lie on interior columns i = I-1; face (j, i) joins nodal rows j and j+1
  if (I >= 1 && I <= mx) {
    const int i = I - 1;
    if (J <= my) s += 0.5 * sum(gy + (long long)J * mx + i, nfy);
    if (J >= 1) s += 0.5 * sum(gy + (long long)(J - 1) * mx + i, nfy);
  }
  grad[(long long)J * (mx + 2) + I] = s;
}

}  // namespace

int stencil_blocks(const Geom &g) {
  const Tile t = tile_for(g), d = tile_df_for(g);
  return std::max(t.gx * t.gy * t.nchunk, d.gx * d.gy * d.nchunk);
}

template <class Tz>
cudaError_t launch_stencil(const Geom &g, int mode, const Tz *z, double *out, const double *fH,
                           State *S, double *partials, int, cudaStream_t st) {
  Tile t = tile_for(g);
  dim3 block = (g.dim == 1) ? dim3(kBX1, 1) : dim3(kBX2, kBY2);
  dim3 grid(t.gx, t.gy, t.nchunk);
  prof_begin(mode == SM_RESID ? KC_RESID : KC_STENCIL, st);
  switch (mode) {
    case SM_MINRES:
      k_stencil<Tz, SM_MINRES><<<grid, block, 0, st>>>(g, z, out, fH, S, partials, t.kc);
      break;
    case SM_APPLY:
      k_stencil<Tz, SM_APPLY><<<grid, block, 0, st>>>(g, z, out, fH, S, partials, t.kc);
      break;
    case SM_RESID:
      k_stencil<Tz, SM_RESID><<<grid, block, 0, st>>>(g, z, out, fH, S, partials, t.kc);
      break;
    default:
      return cudaErrorInvalidValue;
  }
  prof_end(st);
  return cudaGetLastError();
}

cudaError_t launch_stencil_df(const Geom &g, const float *z, df *q, State *S, double *partials,
                              cudaStream_t st) {
  const Tile t = tile_df_for(g);
  const dim3 block(t.bx, kNT / t.bx), grid(t.gx, t.gy, t.nchunk);
  const double th = g.theta;
  prof_begin(KC_STENCIL, st);
  auto go = [&](auto dim, auto uni) {
    constexpr int D = decltype(dim)::value;
    constexpr bool U = decltype(uni)::value;
    if (g.scheme != ST_THETA)
      k_stencil_df<D, U, W_BDF2><<<grid, block, 0, st>>>(g, z, q, S, partials, t.kc);
    else if (th == 0.5)
      k_stencil_df<D, U, W_HALF><<<grid, block, 0, st>>>(g, z, q, S, partials, t.kc);
    else if (th == 1.0)
      k_stencil_df<D, U, W_ONE><<<grid, block, 0, st>>>(g, z, q, S, partials, t.kc);
    else
      k_stencil_df<D, U, W_ANY><<<grid, block, 0, st>>>(g, z, q, S, partials, t.kc);
  };
  auto pick = [&](auto dim) {
    if (g.c_uniform)
      go(dim, std::true_type{});
    else
      go(dim, std::false_type{});
  };
  if (g.dim == 3)
    pick(std::integral_constant<int, 3>{});
  else if (g.dim == 2)
    pick(std::integral_constant<int, 2>{});
  else
    pick(std::integral_constant<int, 1>{});
  prof_end(st);
  return cudaGetLastError();
}

cudaError_t launch_resid_outer(const Geom &g, const double *x, df *r_out, const double *fH,
                               State *S, double *partials, cudaStream_t st) {
  Tile t = tile_for(g);
  dim3 block = (g.dim == 1) ? dim3(kBX1, 1) : dim3(kBX2, kBY2);
  dim3 grid(t.gx, t.gy, t.nchunk);
  prof_begin(KC_RESID, st);
  k_stencil<double, SM_RESID_OUTER, df><<<grid, block, 0, st>>>(g, x, r_out, fH, S, partials, t.kc);
  prof_end(st);
  return cudaGetLastError();
}

cudaError_t launch_resid_df(const Geom &g, const double *x, df *r_out, const double *fH, State *S,
                            double *partials, cudaStream_t st) {
  Tile t = tile_for(g);
  dim3 block = (g.dim == 1) ? dim3(kBX1, 1) : dim3(kBX2, kBY2);
  dim3 grid(t.gx, t.gy, t.nchunk);
  prof_begin(KC_RESID, st);
  k_stencil<double, SM_RESID, df><<<grid, block, 0, st>>>(g, x, r_out, fH, S, partials, t.kc);
  prof_end(st);
  return cudaGetLastError();
}

template cudaError_t launch_stencil<double>(const Geom &, int, const double *, double *,
                                            const double *, State *, double *, int, cudaStream_t);
template cudaError_t launch_stencil<float>(const Geom &, int, const float *, double *,
                                           const double *, State *, double *, int, cudaStream_t);

cudaError_t launch_rhs(const Geom &g, const double *f, const double *u0, const double *uprev,
                       const double *extra, double *fH, cudaStream_t st) {
  const dim3 gr((unsigned)((g.m + 255) / 256), (unsigned)((g.n + kRhsLevels - 1) / kRhsLevels));
  prof_begin(KC_AUX, st);
  if (extra)
    k_rhs<true><<<gr, 256, 0, st>>>(g, f, u0, uprev, extra, fH);
  else
    k_rhs<false><<<gr, 256, 0, st>>>(g, f, u0, uprev, extra, fH);
  prof_end(st);
  return cudaGetLastError();
}

cudaError_t launch_grad_rhs(const Geom &g, const double *lam, double *gf, double *gu0,
                            double *gup, cudaStream_t st) {
  const dim3 gr((unsigned)((g.m + 255) / 256), (unsigned)(g.n / kRhsLevels + 1));
  prof_begin(KC_AUX, st);
  k_grad_rhs<<<gr, 256, 0, st>>>(g, lam, gf, gu0, gup);
  prof_end(st);
  return cudaGetLastError();
}

// scratch: room for cap doubles, used for the chunks' partial face sums when there is more than one
cudaError_t launch_grad_a(const Geom &g, const double *lam, const double *u, const double *u0,
                          double *gface_x, double *gface_y, double *scratch, long long cap,
                          double *grad, cudaStream_t st) {
  const double hx = 1.0 / (g.mx + 1), hy = 1.0 / (g.my + 1);
  const double sx = g.tau / (hx * hx), sy = g.tau / (hy * hy);
  dim3 b(32, 8);
  const int fy = (g.dim == 2) ? g.my + 1 : 1;
  const long long nfx = (long long)(g.mx + 1) * g.my, nfy = (long long)g.mx * (g.my + 1);
  const long long tiles = ((g.mx + 1 + 31) / 32) * (long long)((fy + 7) / 8);
  // chunks of levels: enough blocks for eight per SM, at least eight levels each (a chunk rereads
  // one level), and no more than the scratch holds
  long long nc = (152LL * 8 + tiles - 1) / tiles;
  if (nc > (g.n + 7) / 8) nc = (g.n + 7) / 8;
  if (nc > cap / (nfx + nfy)) nc = cap / (nfx + nfy);
  if (nc < 1) nc = 1;
  const int kc = (int)((g.n + nc - 1) / nc);
  nc = (g.n + kc - 1) / kc;
  double *gx = nc > 1 ? scratch : gface_x, *gy = nc > 1 ? scratch + nc * nfx : gface_y;
  dim3 gr((g.mx + 1 + 31) / 32, (fy + 7) / 8, (unsigned)nc);
  prof_begin(KC_AUX, st);
  if (g.scheme == ST_THETA && g.theta != 1.0)
    k_grad_faces<true><<<gr, b, 0, st>>>(g, lam, u, u0, sx, sy, kc, gx, gy);
  else
    k_grad_faces<false><<<gr, b, 0, st>>>(g, lam, u, u0, sx, sy, kc, gx, gy);
  prof_end(st);
  cudaError_t e = cudaGetLastError();
  if (e != cudaSuccess) return e;
  const int ny = (g.dim == 2) ? g.my + 2 : 1;
  dim3 gn((g.mx + 2 + 31) / 32, (ny + 7) / 8);
  prof_begin(KC_AUX, st);
  k_grad_nodes<<<gn, b, 0, st>>>(g.dim, g.mx, g.my, (int)nc, gx, gy, grad);
  prof_end(st);
  return cudaGetLastError();
}

}  // namespace st
