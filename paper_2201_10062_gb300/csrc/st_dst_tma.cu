// Sine transforms of the mixed path on the tensor cores (tcgen05), fed and drained by tensor copies
// (TMA): one DST-I along x, y, z or time (k_dst_tma) and the whole time stage, DST-I -> spectral
// scaling -> DST-I (k_time_tma).  Float32 data in the padded layout (Geom::px), any axis length
// from 16 to 256.
//
// The folded transform is two dense products per parity of the output index k (Sec. 3.1.1):
//   odd  k = 2r+1:  Y_k = sum_{t=1..h} S_{k,t} (x_t + x_{n+1-t})
//   even k = 2r+2:  Y_k = sum_{t=1..h} S_{k,t} (x_t - x_{n+1-t}),     h = ceil(n/2),
// i.e. D_P[r][j] = sum_t A_P[r][t] B_P[t][j] with A_P fixed and B_P the folded data of a tile of
// columns j; for odd n the middle element folds with nothing.  Both operands are split into two fp16
// pieces (hi + lo, 22 bits); hi*hi + hi*lo + lo*hi accumulate in float32 in tensor memory.  Columns
// of B are scaled by a power of two so that fp16 keeps its range; S is scaled by 8.
//
// What bounds these passes is the latency of a tile's way through the roles (ncu, 255^2 x 256: issue
// slots 51% busy in the time stage and 31% in a y or x pass, tensor pipe 20%, DRAM 14% and 30%; the
// stalls are waits for tensor memory and for the role before).  So:
//   - a tile is loaded by one thread with a few tensor copies (128-byte-swizzled boxes of 32
//     floats), two or more tiles ahead, into a ring of buffers; its result is written back into
//     the buffer it came from and leaves by tensor copies as well.  No thread computes a global
//     address, and ragged edges are the copies' zero fill and clipping.
//   - the fold reads 16 bytes a thread (four columns of a row, or four elements of an x line), and
//     the B operand's column groups are 16 bytes further apart than a multiple of 128, so its
//     16-byte stores fall in distinct banks;
//   - short axes take more columns per tile, so that a tile is 8192 elements whatever the length:
//     G = 1, 2 or 4 groups of 32 columns for h up to 128, 64 or 32.  With h <= 64 the two
//     parities (and for h <= 32 two halves of the groups as well) are stacked in the 128 rows of
//     the MMA: slot s holds its rows of A and zeros elsewhere, every slot's product accumulates into
//     the same accumulator columns, and every thread of the epilogue has 64 values to take out;
//   - MMAs are issued under elect.sync (see elect_one); two accumulators share the K steps (see
//     issue_pair).
// S (all slots, hi and lo) stays in tensor memory for the whole launch; one block per SM walks the
// tiles with its warps in separate roles that hand off through mbarriers, every wait bounded.  On a
// timeout the block records ST_ERR_TIMEOUT and stops; before it frees its tensor memory every MMA
// must be known to be complete, else it keeps it and sets State::tmem_held (see tc_release_cols).
#include <cmath>
#include <cstdlib>
#include <type_traits>

#include "st_tma.cuh"

namespace st {
namespace {

// slots of 128 / SL rows: h <= 128 / SL
int slots_for(int len) {
  const int h = (len + 1) / 2;
  return h > 64 ? 1 : (h > 32 ? 2 : 4);
}

__host__ __device__ constexpr int num_slots(int SL) { return SL < 2 ? 2 : SL; }

struct TmaDim {
  int len, h, hK, h8;      // axis length, folded rows, padded to the MMA's K step, to 8 rows
  uint32_t gin;            // bytes of one staged input group of 32 columns (y, z, time)
  uint32_t rb;             // bytes of a ring buffer
  uint32_t sbo, ph, bb;    // B operand: bytes between 8-column groups, of one column set's hi (or
                           // lo) piece, and in all
};

__host__ __device__ inline TmaDim tma_dim(int len, int SL) {
  TmaDim d;
  d.len = len;
  d.h = (len + 1) >> 1;
  d.hK = (d.h + 15) & ~15;
  d.h8 = (d.h + 7) & ~7;
  d.gin = (uint32_t)((len + 7) & ~7) * 128u;
  const uint32_t out = 2u * (uint32_t)d.h8 * 128u;
  d.rb = (uint32_t)SL * (d.gin > out ? d.gin : out);
  d.sbo = 16u * (uint32_t)d.hK + 16u;
  d.ph = (SL == 1 ? 4u : 8u) * d.sbo;
  d.bb = 4u * (SL == 4 ? 2u : 1u) * d.ph;
  return d;
}

// B operand: [parity][column set][hi, lo][8-column group], a column set being the columns that one
// slot multiplies: the tile's 32 (SL 1) or 64 (SL 2) columns, or half of its 128 (SL 4).
template <int SL>
__device__ __forceinline__ uint32_t b_off(const TmaDim &D, int P, int c) {
  if (SL == 4) return (uint32_t)((P * 2 + (c >> 6)) * 2) * D.ph + (uint32_t)((c >> 3) & 7) * D.sbo;
  return (uint32_t)(P * 2) * D.ph + (uint32_t)(c >> 3) * D.sbo;
}

// All MMAs of one transform of a tile: slot s = parity (SL 1, 2) or 2 parity + column set (SL 4).
// Accumulators (see issue_pair): a pair of 32 columns for each parity with SL 1; else one pair of 64,
// which the first slot overwrites (a slot's zero rows of A add exact zeros to the others' rows).
template <int SL>
__device__ __forceinline__ void issue_tile(uint32_t a_base, uint32_t bop, const TmaDim &D,
                                           uint32_t dcol) {
  const int KS = D.hK >> 4;
  const uint32_t vc = (uint32_t)(D.hK >> 1);
  const uint64_t lo = D.ph >> 4;
  if constexpr (SL == 1) {
    issue_two_pairs<32, 8>(dcol, dcol + 64u, a_base, a_base + 2u * vc, vc, make_desc_sbo(bop, D.sbo),
                           make_desc_sbo(bop + 2u * D.ph, D.sbo), lo, KS, KS);
  } else {
#pragma unroll 1
    for (int s = 0; s < num_slots(SL); ++s)
      issue_pair<64, 8 / SL>(dcol, a_base + (uint32_t)(2 * s) * vc, vc,
                             make_desc_sbo(bop + (uint32_t)(2 * s) * D.ph, D.sbo), lo, KS,
                             s > 0 ? 1u : 0u);
  }
}

// ---------------------------------------------------------------- fold, scale, split
// A build set is 128 threads (256 with two columns a thread).  Each thread holds vectors of eight folded
// rows: strided lines, four (two) adjacent columns of one t-block; x lines, four t-blocks of one line.
template <int NC>
__device__ __forceinline__ void lds_cols(uint32_t a, float (&v)[NC]) {
  if constexpr (NC == 4) {
    const float4 x = lds4(a);
    v[0] = x.x;
    v[1] = x.y;
    v[2] = x.z;
    v[3] = x.w;
  } else {
    asm volatile("ld.shared.v2.f32 {%0, %1}, [%2];" : "=f"(v[0]), "=f"(v[1]) : "r"(a));
  }
}
template <int NC>
__device__ __forceinline__ void sts_cols(uint32_t a, const float (&v)[NC]) {
  if constexpr (NC == 4)
    sts4f(a, v[0], v[1], v[2], v[3]);
  else
    sts2f(a, v[0], v[1]);
}

// Build of strided lines by a set of 512 / NC threads, NC = 4 or 2 adjacent columns each.  buf: the
// staged tile, rows of 32 columns (128 bytes, 16-byte chunk c stored at c ^ (row & 7)): natural rows t
// (PAR false), or split by parity of t as the epilogue leaves them (PAR true: row t at
// ((g 2 + (t & 1)) h8 + t / 2)).  `ready` waits until the B buffer and the factors may be written.
// Returns false if a wait ran out in any thread of the set.  One named barrier inside, one at the end.
template <int SL, bool PAR, int NC, class Ready>
__device__ __forceinline__ bool build_lines(uint32_t buf, uint32_t zero, uint32_t bop,
                                            uint32_t colinv, uint32_t part, const TmaDim &D, int bt,
                                            int bar, bool ok, Ready ready) {
  constexpr int NT = 512 / NC, CQ = 32 / NC, IPW = 32 / CQ;  // threads, lanes a row, t-blocks a warp
  constexpr int TS = 16 / SL, WPG = TS / IPW;                // t-blocks, warps of a group
  const int lane = bt & 31, w = bt >> 5, cq = lane & (CQ - 1);
  const int it = w * IPW + lane / CQ, g = it / TS, tb = it - g * TS;
  const uint32_t cb = (uint32_t)(cq * NC * 4);  // byte of the thread's columns in a row
  auto row = [&](int t) -> uint32_t {
    if (PAR) {
      const int r = t >> 1;
      return buf + (uint32_t)(((g * 2 + (t & 1)) * D.h8 + r) * 128) + (cb ^ (uint32_t)((r & 7) << 4));
    }
    return buf + (uint32_t)g * D.gin + (uint32_t)(t * 128) + (cb ^ (uint32_t)((t & 7) << 4));
  };
  float u[NC][8], d[NC][8], mx[NC];
#pragma unroll
  for (int j = 0; j < NC; ++j) mx[j] = 0.f;
  if (ok) {
#pragma unroll
    for (int q = 0; q < 8; ++q) {
      const int t = tb * 8 + q, tm = D.len - 1 - t;
      // rows past the fold read zeros; the middle row of an odd length folds with nothing
      float a[NC], b[NC];
      lds_cols<NC>(t < D.h ? row(t) : zero, a);
      lds_cols<NC>(t < D.h && tm != t ? row(tm) : zero, b);
#pragma unroll
      for (int j = 0; j < NC; ++j) {
        u[j][q] = a[j] + b[j];
        d[j][q] = a[j] - b[j];
        mx[j] = fmaxf(mx[j], fmaxf(fabsf(u[j][q]), fabsf(d[j][q])));
      }
    }
  }
#pragma unroll
  for (int o = CQ; o <= 16; o <<= 1) {
#pragma unroll
    for (int j = 0; j < NC; ++j) mx[j] = fmaxf(mx[j], __shfl_xor_sync(0xffffffffu, mx[j], o));
  }
  if (lane < CQ) sts_cols<NC>(part + (uint32_t)(w * 128) + cb, mx);
  if (ok) ok = ready();
  if (!group_sync_and(ok, bar, NT)) return false;
#pragma unroll
  for (int i = 0; i < WPG; ++i) {
    float x[NC];
    lds_cols<NC>(part + (uint32_t)((g * WPG + i) * 128) + cb, x);
#pragma unroll
    for (int j = 0; j < NC; ++j) mx[j] = fmaxf(mx[j], x[j]);
  }
#pragma unroll
  for (int j = 0; j < NC; ++j) mx[j] = scale_of(mx[j]);
  if (tb == 0) {
    float ci[NC];
#pragma unroll
    for (int j = 0; j < NC; ++j) ci[j] = inv_scale(mx[j]);
    sts_cols<NC>(colinv + (uint32_t)(g * 128) + cb, ci);
  }
  if (tb * 8 < D.hK) {
#pragma unroll
    for (int j = 0; j < NC; ++j) {
      const int c = g * 32 + NC * cq + j;
      const uint32_t a = bop + (uint32_t)(tb * 128 + (c & 7) * 16);
      put_piece(a + b_off<SL>(D, 0, c), D.ph, u[j], mx[j]);
      put_piece(a + b_off<SL>(D, 1, c), D.ph, d[j], mx[j]);
    }
  }
  fence_async_smem();
  group_sync(bar, NT);
  return true;
}

// Build of x lines: buf holds [px / 32][32 SL lines][32 floats], 16-byte chunks swizzled by line & 7.
// A thread takes one line and the t-blocks w', w' + WPG, ... of it.
template <int SL, class Ready>
__device__ __forceinline__ bool build_xlines(uint32_t buf, uint32_t bop, uint32_t colinv,
                                             uint32_t part, const TmaDim &D, int bt, int bar,
                                             bool ok, Ready ready) {
  constexpr int WPG = 4 / SL;
  const int lane = bt & 31, w = bt >> 5;
  const int g = w / WPG, w0 = w - g * WPG;
  const int line = g * 32 + lane, nb = D.hK >> 3, px = D.len + 1;
  const uint32_t lbase = buf + (uint32_t)line * 128u, lsw = (uint32_t)(line & 7) << 4;
  auto chunk = [&](int e) -> uint32_t {  // the 16-byte chunk that starts at element e
    return lbase + (uint32_t)(e >> 5) * (uint32_t)(SL * 32 * 128) +
           ((uint32_t)((e & 31) << 2) ^ lsw);
  };
  float u[4][8], d[4][8];
  float mx = 0.f;
  if (ok) {
#pragma unroll
    for (int i = 0; i < 4; ++i) {
      const int tb = w0 + WPG * i;
      if (tb >= nb) {
#pragma unroll
        for (int q = 0; q < 8; ++q) u[i][q] = d[i][q] = 0.f;
        continue;
      }
      const int e = tb * 8;
      const float4 a0 = lds4(chunk(e)), a1 = lds4(chunk(e + 4));
      // mirrored elements px - 2 - e - q: the chunks at px - 4 - e and px - 8 - e, and the last
      // element of the one before; the middle element (odd length) folds with nothing
      const float4 b0 = lds4(chunk(px - 4 - e)), b1 = lds4(chunk(px - 8 - e));
      const float b7 = (px - 9 - e == e + 7) ? 0.f : lds1(chunk(px - 12 - e) + 12u);
      const float a[8] = {a0.x, a0.y, a0.z, a0.w, a1.x, a1.y, a1.z, a1.w};
      const float b[8] = {b0.z, b0.y, b0.x, b1.w, b1.z, b1.y, b1.x, b7};
#pragma unroll
      for (int q = 0; q < 8; ++q) {
        u[i][q] = a[q] + b[q];
        d[i][q] = a[q] - b[q];
        mx = fmaxf(mx, fmaxf(fabsf(u[i][q]), fabsf(d[i][q])));
      }
    }
  }
  if (WPG > 1) sts1f(part + (uint32_t)(w * 128 + lane * 4), mx);
  if (ok) ok = ready();
  if (!group_sync_and(ok, bar, 128)) return false;
  if (WPG > 1) {
#pragma unroll
    for (int i = 0; i < WPG; ++i) mx = fmaxf(mx, lds1(part + (uint32_t)((g * WPG + i) * 128 + lane * 4)));
  }
  const float sc = scale_of(mx);
  if (w0 == 0) sts1f(colinv + (uint32_t)line * 4u, inv_scale(sc));
#pragma unroll
  for (int i = 0; i < 4; ++i) {
    const int tb = w0 + WPG * i;
    if (tb < nb) {
      const uint32_t a = bop + (uint32_t)(tb * 128 + (line & 7) * 16);
      put_piece(a + b_off<SL>(D, 0, line), D.ph, u[i], sc);
      put_piece(a + b_off<SL>(D, 1, line), D.ph, d[i], sc);
    }
  }
  fence_async_smem();
  group_sync(bar, 128);
  return true;
}

// 16 values of one unit: its two accumulators summed
template <int SL>
__device__ __forceinline__ void tmem_unit16(uint32_t acc, int j, int k, float (&v)[16]) {
  tmem_sum16(acc + (SL == 1 ? 64u : 32u) * (uint32_t)j + 16u * (uint32_t)k, SL == 1 ? 32u : 64u, v);
}
template <int SL>
__device__ __forceinline__ void tmem_unit(uint32_t acc, int j, float (&v)[32]) {
  float a[16];
#pragma unroll
  for (int k = 0; k < 2; ++k) {
    tmem_unit16<SL>(acc, j, k, a);
#pragma unroll
    for (int c = 0; c < 16; ++c) v[16 * k + c] = a[c];
  }
}

// The two (parity, group) units of an epilogue thread at accumulator row R: P and g of unit j, and
// the folded row r.
template <int SL>
struct Unit {
  static __device__ __forceinline__ int row(int R) { return R & (kM / SL - 1); }
  static __device__ __forceinline__ int P(int R, int j) {
    return SL == 1 ? j : (SL == 2 ? R >> 6 : R >> 6);
  }
  static __device__ __forceinline__ int g(int R, int j) {
    return SL == 1 ? 0 : (SL == 2 ? j : 2 * ((R >> 5) & 1) + j);
  }
};

// 16 columns (half k) of an unscaled row of one unit into the tile's buffer, split by parity (row r
// of box (g, P))
template <int NV>
__device__ __forceinline__ void put_row(uint32_t buf, const TmaDim &D, int g, int P, int r, int k,
                                        const float (&v)[NV], uint32_t ci) {
  const uint32_t a = buf + (uint32_t)(((g * 2 + P) * D.h8 + r) * 128), sw = (uint32_t)(r & 7) << 4;
#pragma unroll
  for (int c = 0; c < NV / 4; ++c) {
    const uint32_t o = 64u * (uint32_t)k + 16u * c;
    const float4 f = lds4(ci + o);
    sts4f(a + (o ^ sw), v[4 * c] * f.x, v[4 * c + 1] * f.y, v[4 * c + 2] * f.z,
          v[4 * c + 3] * f.w);
  }
}

// ---------------------------------------------------------------- one transform
// Warps 0..3: epilogue (one per lane quadrant); then two build sets that take alternate tiles, each
// with its own B buffer; then one warp each for the MMAs, the loads and the stores.
// kNC: strided lines, columns a build thread (2: sets of 8 warps)
constexpr int kBuildW = 4;
constexpr int kMmaWarpS = 4 + 2 * kBuildW, kLoadWarpS = kMmaWarpS + 1, kStoreWarpS = kMmaWarpS + 2;
constexpr int kNTS = (kMmaWarpS + 3) * 32;
constexpr int kMaxRing = 8;

// Shared memory: the small arrays first, at offsets known at compile time, then the ring (1024-byte
// aligned, as the swizzle wants) and the two B buffers.
template <int SL>
struct DstSmem {
  // full, ofull, oempty [8 each], bfull, bempty, afull, aempty [2 each], done
  static constexpr uint32_t mbar = 0, tmem = (3u * kMaxRing + 9u) * 8u, zero = (tmem + 8u + 15u) & ~15u,
                            colinv = zero + 16u, part = colinv + 2u * 128u * SL,
                            ring = (part + 2u * 512u + 1023u) & ~1023u;
  static __host__ __device__ uint32_t bop(const TmaDim &D, int NB) { return ring + (uint32_t)NB * D.rb; }
  // with room to align the start
  static __host__ __device__ uint32_t total(const TmaDim &D, int NB) { return bop(D, NB) + 2u * D.bb + 1008u; }
};

// XL: `groups` is the number of lines, chunks = px / 32, out0 takes the result, unless `user`
// takes the lines without their padding (contiguous, not aligned: the store warp copies them); else
// groups of 32 columns, `chunks` of them in a plane, and out0 / out1 take the odd and even outputs.
template <int SL, bool XL>
__global__ void __launch_bounds__(kNTS, 1)
    k_dst_tma(const __grid_constant__ CUtensorMap in0, const __grid_constant__ CUtensorMap out0,
              const __grid_constant__ CUtensorMap out1, int len, int NB, int chunks,
              unsigned groups, float *user, const uint4 *img, State *S, int gk) {
  if (gate_closed(S, gk)) return;
  extern __shared__ unsigned char smem_raw[];
  const TmaDim D = tma_dim(len, SL);
  using L = DstSmem<SL>;
  const uint32_t sm = (smem_u32(smem_raw) + 1023u) & ~1023u;
  const int tid = threadIdx.x, warp = tid >> 5, lane = tid & 31;
  const uint32_t ring = sm + L::ring, bop = sm + L::bop(D, NB), colinv = sm + L::colinv,
                 zero = sm + L::zero;
  const uint32_t full = sm + L::mbar, ofull = full + 8u * kMaxRing, oempty = ofull + 8u * kMaxRing,
                 bfull = oempty + 8u * kMaxRing, bempty = bfull + 16u, afull = bempty + 16u,
                 aempty = afull + 16u, done = aempty + 16u, tslot = sm + L::tmem;
  const unsigned per = XL ? 32u * SL : (unsigned)SL;  // lines or groups in a tile
  const unsigned ntiles = (groups + per - 1) / per;
  if (tid == 0) {
    for (int i = 0; i < 3 * kMaxRing + 9; ++i) {
      uint32_t cnt = 1u;
      if (i >= kMaxRing && i < 2 * kMaxRing) cnt = 4u;         // ofull: epilogue warps
      const int j = i - 3 * kMaxRing;
      if (j == 2 || j == 3) cnt = 5u;                          // bempty: MMA commit + epilogue
      if (j == 6 || j == 7) cnt = 4u;                          // aempty: epilogue warps
      asm volatile("mbarrier.init.shared::cta.b64 [%0], %1;" ::"r"(full + 8u * i), "r"(cnt)
                   : "memory");
    }
    sts4(zero, 0u, 0u, 0u, 0u);
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
  const uint32_t dcol = tmem + 256u;  // two 128-column accumulators after S
  const unsigned first = blockIdx.x, step = gridDim.x;
  auto load = [&](unsigned tile, int s) {
    const uint32_t mb = full + 8u * s, dst = ring + (uint32_t)s * D.rb;
    if (XL) {
      mbar_expect_tx(mb, (uint32_t)chunks * 32u * SL * 128u);
      for (int c = 0; c < chunks; ++c)
        tma_load3(dst + (uint32_t)c * (32u * SL * 128u), &in0, c * 32, (int)(tile * per), 0, mb);
    } else {
      mbar_expect_tx(mb, (uint32_t)SL * (uint32_t)len * 128u);
      for (int g = 0; g < SL; ++g) {
        // past the last group: that group once more (its result is not stored)
        const unsigned gi = min(tile * per + g, groups - 1);
        const unsigned pl = gi / (unsigned)chunks;
        tma_load3(dst + (uint32_t)g * D.gin, &in0, (int)(gi - pl * chunks) * 32, 0, (int)pl, mb);
      }
    }
  };
  // the first ring of loads flies while S is copied
  uint32_t preloaded = 0;
  if (warp == kLoadWarpS && elect_one())
    for (unsigned tile = first; tile < ntiles && preloaded < (uint32_t)NB; tile += step)
      load(tile, (int)preloaded++);
  __syncwarp();
  load_a_variants(img, 2 * num_slots(SL), D.hK, tmem, warp, kNTS / 32, lane);
  fence_before();
  __syncthreads();
  fence_after();
  bool ok = true;
  bool drained = true;  // the loading thread: no copy into shared memory left in flight
  if (warp == kLoadWarpS) {
    // ------------------------------------------------------------------ loads
    if (elect_one()) {
      int s = preloaded == (uint32_t)NB ? 0 : (int)preloaded;
      uint32_t ph = 0u, n = preloaded;
      for (unsigned tile = first + preloaded * step; tile < ntiles; tile += step, ++n) {
        if (!mbar_wait(oempty + 8u * s, ph)) {
          ok = false;
          break;
        }
        load(tile, s);
        if (++s == NB) {
          s = 0;
          ph ^= 1u;
        }
      }
      // a load must have landed before the block ends: wait (bounded) for the last NB of them
      const uint32_t lo = n > (uint32_t)NB ? n - NB : 0u;
      for (uint32_t i = lo; i < n; ++i)
        if (!mbar_wait(full + 8u * (i % NB), (i / NB) & 1u)) drained = false;
    }
    __syncwarp();
  } else if (warp == kStoreWarpS) {
    // ------------------------------------------------------------------ stores
    if (XL && user != nullptr) {
      int s = 0;
      uint32_t ph = 0u;
      for (unsigned tile = first; tile < ntiles; tile += step) {
        ok = __all_sync(0xffffffffu, mbar_wait(ofull + 8u * s, ph) ? 1 : 0) != 0;
        if (!ok) break;
        const uint32_t src = ring + (uint32_t)s * D.rb;
        const int lines = (int)min(per, groups - tile * per);
        float *dst = user + (long long)tile * per * len + lane;
        for (int l = 0; l < lines; ++l, dst += len) {
          const uint32_t a = src + (uint32_t)l * 128u + (((uint32_t)lane * 4u) ^ ((uint32_t)(l & 7) << 4));
#pragma unroll
          for (int c = 0; c < 8 / SL; ++c)
            if (c < chunks && c * 32 + lane < len) dst[c * 32] = lds1(a + (uint32_t)c * (4096u * SL));
        }
        __syncwarp();
        if (lane == 0) mbar_arrive(oempty + 8u * s);
        if (++s == NB) {
          s = 0;
          ph ^= 1u;
        }
      }
    } else if (elect_one()) {
      int s = 0;
      uint32_t ph = 0u;
      for (unsigned tile = first; tile < ntiles; tile += step) {
        if (!mbar_wait(ofull + 8u * s, ph)) {
          ok = false;
          break;
        }
        const uint32_t src = ring + (uint32_t)s * D.rb;
        if (XL) {
          for (int c = 0; c < chunks; ++c)
            tma_store3(&out0, src + (uint32_t)c * (32u * SL * 128u), c * 32, (int)(tile * per), 0);
        } else {
          for (int g = 0; g < SL; ++g) {
            const unsigned gi = tile * per + g;
            if (gi >= groups) break;
            const unsigned pl = gi / (unsigned)chunks;
            const int x = (int)(gi - pl * chunks) * 32;
            const uint32_t b = src + (uint32_t)(2 * g * D.h8) * 128u;
            tma_store3(&out0, b, x, 0, (int)pl);
            tma_store3(&out1, b + (uint32_t)D.h8 * 128u, x, 0, (int)pl);
          }
        }
        bulk_commit();
        bulk_wait_read();
        mbar_arrive(oempty + 8u * s);
        if (++s == NB) {
          s = 0;
          ph ^= 1u;
        }
      }
      bulk_wait_done();
    }
    __syncwarp();
  } else if (warp == kMmaWarpS) {
    // ------------------------------------------------------------------ MMA thread
    if (elect_one()) {
      uint32_t n = 0;
      for (unsigned tile = first; tile < ntiles; tile += step, ++n) {
        const uint32_t b = n & 1u, ph = (n >> 1) & 1u;
        if (!mbar_wait(bfull + 8u * b, ph) || !mbar_wait(aempty + 8u * b, ph ^ 1u)) {
          ok = false;
          break;
        }
        fence_after();
        issue_tile<SL>(tmem, bop + b * D.bb, D, dcol + 128u * b);
        mma_commit(afull + 8u * b);
        mma_commit(bempty + 8u * b);
      }
      mma_commit(done);
    }
    __syncwarp();
  } else if (warp >= 4) {
    // ------------------------------------------------------------------ build sets
    const uint32_t k = (uint32_t)(warp - 4) >> 2;
    const int bt = tid - 128 - 128 * (int)k;
    uint32_t n = 0;
    int s = 0;
    uint32_t ph = 0u;
    for (unsigned tile = first; tile < ntiles; tile += step, ++n) {
      if ((n & 1u) == k) {
        const uint32_t bph = ((n >> 1) & 1u) ^ 1u;
        ok = mbar_wait(full + 8u * s, ph);
        auto ready = [&]() { return mbar_wait(bempty + 8u * k, bph); };
        const uint32_t buf = ring + (uint32_t)s * D.rb, bo = bop + k * D.bb;
        const uint32_t ci = colinv + k * 128u * SL, pa = sm + L::part + k * 512u;
        if (XL)
          ok = build_xlines<SL>(buf, bo, ci, pa, D, bt, 1 + (int)k, ok, ready);
        else
          ok = build_lines<SL, false, 4>(buf, zero, bo, ci, pa, D, bt, 1 + (int)k, ok, ready);
        if (!ok) break;
        if (bt == 0) mbar_arrive(bfull + 8u * k);
      }
      if (++s == NB) {
        s = 0;
        ph ^= 1u;
      }
    }
  } else {
    // ------------------------------------------------------------------ epilogue
    const int R = warp * 32 + lane, r = Unit<SL>::row(R);
    const uint32_t lanes = (uint32_t)(warp * 32) << 16;
    uint32_t n = 0;
    int s = 0;
    for (unsigned tile = first; tile < ntiles; tile += step, ++n) {
      const uint32_t b = n & 1u, ph = (n >> 1) & 1u;
      ok = __all_sync(0xffffffffu, mbar_wait(bfull + 8u * b, ph) ? 1 : 0) != 0;
      if (ok) ok = __all_sync(0xffffffffu, mbar_wait(afull + 8u * b, ph) ? 1 : 0) != 0;
      if (!ok) break;
      fence_after();
      float v[2][32];
      tmem_unit<SL>(dcol + 128u * b + lanes, 0, v[0]);
      tmem_unit<SL>(dcol + 128u * b + lanes, 1, v[1]);
      fence_before();
      __syncwarp();
      if (lane == 0) mbar_arrive(aempty + 8u * b);  // the accumulator is free
      const uint32_t buf = ring + (uint32_t)s * D.rb, ci = colinv + b * 128u * SL;
      if (r < D.h) {
        if (XL && SL == 1) {
          // both parities of row r: elements 2r and 2r + 1 of every line
          const uint32_t a = buf + (uint32_t)(r >> 4) * 4096u;
          const uint32_t e = (uint32_t)((r & 15) << 3);
#pragma unroll
          for (int c4 = 0; c4 < 8; ++c4) {
            const float4 f4 = lds4(ci + 16u * c4);
            const float f[4] = {f4.x, f4.y, f4.z, f4.w};
#pragma unroll
            for (int j = 0; j < 4; ++j) {
              const uint32_t c = 4u * c4 + j;
              sts2f(a + c * 128u + (e ^ ((c & 7u) << 4)), v[0][c] * f[j],
                    v[1][c] * f[j]);
            }
          }
        } else if (XL) {
#pragma unroll
          for (int j2 = 0; j2 < 2; ++j2) {
            const int P = Unit<SL>::P(R, j2), g = Unit<SL>::g(R, j2), el = 2 * r + P;
            const uint32_t a = buf + (uint32_t)(el >> 5) * (4096u * SL) + (uint32_t)g * 4096u;
            const uint32_t e = (uint32_t)((el & 31) << 2);
#pragma unroll
            for (int c4 = 0; c4 < 8; ++c4) {
              const float4 f4 = lds4(ci + (uint32_t)g * 128u + 16u * c4);
              const float f[4] = {f4.x, f4.y, f4.z, f4.w};
#pragma unroll
              for (int j = 0; j < 4; ++j) {
                const uint32_t c = 4u * c4 + j;
                sts1f(a + c * 128u + (e ^ ((c & 7u) << 4)), v[j2][c] * f[j]);
              }
            }
          }
        } else {
#pragma unroll
          for (int j = 0; j < 2; ++j) {
            const int g = Unit<SL>::g(R, j);
            put_row(buf, D, g, Unit<SL>::P(R, j), r, 0, v[j], ci + (uint32_t)g * 128u);
          }
        }
      }
      fence_async_smem();
      __syncwarp();
      if (lane == 0) {
        mbar_arrive(bempty + 8u * b);  // the column factors are read
        mbar_arrive(ofull + 8u * s);
      }
      if (++s == NB) s = 0;
    }
  }
  fence_before();
  const bool all_ok = __syncthreads_and(ok ? 1 : 0) != 0;
  const bool copies = __syncthreads_and(drained ? 1 : 0) != 0;
  tc_release_cols<512>(all_ok, true, done, 0u, false, 0u, 0u, tmem, S, copies);
}

// ---------------------------------------------------------------- the time stage
// Eight warpgroups: two of epilogue 1 (1/p, energy, the scaled transform back into the tile's
// buffer; one unit each), epilogue 2 (the result into the buffer), two of build 1, two of build 2, and
// one for the MMA threads of the two transforms, the loads and the stores.  The builds hold 32 folded
// values a thread and take their registers from the other groups (kRegs*; their sum stays within the
// 8 x 64 of the launch), as with equal shares they spill more (now 4 to 64 bytes, in most of the nine
// instantiations).
constexpr int kNTT = 32 * 32, kMiscWarpT = 28, kLoadWarpT = 30, kStoreWarpT = 31;
constexpr int kRegsLaunch = 64, kRegsEpi = 56, kRegsBuild = 72, kRegsMisc = 56;
static_assert(3 * kRegsEpi + 4 * kRegsBuild + kRegsMisc <= 8 * kRegsLaunch, "register split");

// A warpgroup's share changes at the start and back at the end of its role; its warps meet before the
// second change (the instruction wants that).
template <int N>
__device__ __forceinline__ void regs_dec() {
  asm volatile("setmaxnreg.dec.sync.aligned.u32 %0;" ::"n"(N) : "memory");
}
template <int N>
__device__ __forceinline__ void regs_inc() {
  asm volatile("setmaxnreg.inc.sync.aligned.u32 %0;" ::"n"(N) : "memory");
}
__device__ __forceinline__ void warpgroup_sync() { group_sync(3 + (threadIdx.x >> 7), 128); }

template <int SL>
struct TimeSmem {
  // full, yfull, ofull, oempty [8 each]; b1full, b1empty, b2full, b2empty, a1full, a1empty, a2full,
  // a2empty; c1full, c1empty, c2full, c2empty [2 each]; done1, done2
  static constexpr uint32_t mbar = 0, tmem = (4u * kMaxRing + 8u + 8u + 2u) * 8u,
                            zero = (tmem + 8u + 15u) & ~15u, ci1 = zero + 16u,
                            ci2 = ci1 + 2u * 128u * SL, tmu = ci2 + 2u * 128u * SL,
                            part = tmu + 2u * 128u * SL,
                            ring = (part + 2u * 1024u + 1023u) & ~1023u;
  static __host__ __device__ uint32_t b1(const TmaDim &D, int NB) { return ring + (uint32_t)NB * D.rb; }
  static __host__ __device__ uint32_t total(const TmaDim &D, int NB) { return b1(D, NB) + 2u * D.bb + 1008u; }
};

template <int SL, int KIND>
__global__ void __launch_bounds__(kNTT, 1)
    k_time_tma(const __grid_constant__ CUtensorMap in0, const __grid_constant__ CUtensorMap out0,
               const __grid_constant__ CUtensorMap out1, int n, int NB, unsigned groups,
               long long m, int mx, int px, Spec<float> sp, const uint4 *img, State *S, int tmode,
               double *__restrict__ partials, int gk) {
  __shared__ double red[32];
  if (gate_closed(S, gk)) return;
  extern __shared__ unsigned char smem_raw[];
  const TmaDim D = tma_dim(n, SL);
  using L = TimeSmem<SL>;
  const uint32_t sm = (smem_u32(smem_raw) + 1023u) & ~1023u;
  const int tid = threadIdx.x, warp = tid >> 5, lane = tid & 31;
  const uint32_t ring = sm + L::ring, zero = sm + L::zero;
  const uint32_t full = sm + L::mbar, yfull = full + 8u * kMaxRing, ofull = yfull + 8u * kMaxRing,
                 oempty = ofull + 8u * kMaxRing, b1full = oempty + 8u * kMaxRing,
                 b1empty = b1full + 8u, b2full = b1empty + 8u, b2empty = b2full + 8u,
                 a1full = b2empty + 8u, a1empty = a1full + 8u, a2full = a1empty + 8u,
                 a2empty = a2full + 8u, c1full = a2empty + 8u, c1empty = c1full + 16u,
                 c2full = c1empty + 16u, c2empty = c2full + 16u, done1 = c2empty + 16u,
                 done2 = done1 + 8u, tslot = sm + L::tmem;
  const unsigned ntiles = (groups + SL - 1) / SL;
  if (tid == 0) {
    for (int i = 0; i < 4 * kMaxRing + 18; ++i) {
      uint32_t cnt = 1u;
      if (i >= kMaxRing && i < 2 * kMaxRing) cnt = 8u;      // yfull: the warps of epilogue 1
      if (i >= 2 * kMaxRing && i < 3 * kMaxRing) cnt = 4u;  // ofull: of epilogue 2
      const int j = i - 4 * kMaxRing - 4;                   // a1full .. done2
      if (j == 1 || j == 6 || j == 7) cnt = 8u;             // a1empty, c1empty
      if (j == 3 || j == 10 || j == 11) cnt = 4u;           // a2empty, c2empty
      asm volatile("mbarrier.init.shared::cta.b64 [%0], %1;" ::"r"(full + 8u * i), "r"(cnt)
                   : "memory");
    }
    sts4(zero, 0u, 0u, 0u, 0u);
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
  const uint32_t dcol1 = tmem + 256u, dcol2 = tmem + 384u;  // 128-column accumulators
  const unsigned first = blockIdx.x, step = gridDim.x;
  auto load = [&](unsigned tile, int s) {
    mbar_expect_tx(full + 8u * s, (uint32_t)SL * (uint32_t)n * 128u);
    for (int g = 0; g < SL; ++g) {
      const unsigned gi = min(tile * SL + g, groups - 1);
      tma_load3(ring + (uint32_t)s * D.rb + (uint32_t)g * D.gin, &in0, (int)gi * 32, 0, 0,
                full + 8u * s);
    }
  };
  // the first ring of loads flies while S is copied
  uint32_t preloaded = 0;
  if (warp == kLoadWarpT && elect_one())
    for (unsigned tile = first; tile < ntiles && preloaded < (uint32_t)NB; tile += step)
      load(tile, (int)preloaded++);
  __syncwarp();
  load_a_variants(img, 2 * num_slots(SL), D.hK, tmem, warp, kNTT / 32, lane);
  fence_before();
  __syncthreads();
  fence_after();
  bool ok = true, drained = true;
  float esum = 0.f, ecomp = 0.f;
  if (warp >= kMiscWarpT) {
    regs_dec<kRegsMisc>();
    const bool one = elect_one();
    if (warp == kLoadWarpT && one) {
      // ---------------------------------------------------------------- loads
      int s = preloaded == (uint32_t)NB ? 0 : (int)preloaded;
      uint32_t ph = 0u, cnt = preloaded;
      for (unsigned tile = first + preloaded * step; tile < ntiles; tile += step, ++cnt) {
        if (!mbar_wait(oempty + 8u * s, ph)) {
          ok = false;
          break;
        }
        load(tile, s);
        if (++s == NB) {
          s = 0;
          ph ^= 1u;
        }
      }
      const uint32_t lo = cnt > (uint32_t)NB ? cnt - NB : 0u;
      for (uint32_t i = lo; i < cnt; ++i)
        if (!mbar_wait(full + 8u * (i % NB), (i / NB) & 1u)) drained = false;
    } else if (warp == kStoreWarpT && one) {
      // ---------------------------------------------------------------- stores
      int s = 0;
      uint32_t ph = 0u;
      for (unsigned tile = first; tile < ntiles; tile += step) {
        if (!mbar_wait(ofull + 8u * s, ph)) {
          ok = false;
          break;
        }
        for (int g = 0; g < SL; ++g) {
          const unsigned gi = tile * SL + g;
          if (gi >= groups) break;
          const uint32_t b = ring + (uint32_t)s * D.rb + (uint32_t)(2 * g * D.h8) * 128u;
          tma_store3(&out0, b, (int)gi * 32, 0, 0);
          tma_store3(&out1, b + (uint32_t)D.h8 * 128u, (int)gi * 32, 0, 0);
        }
        bulk_commit();
        bulk_wait_read();
        mbar_arrive(oempty + 8u * s);
        if (++s == NB) {
          s = 0;
          ph ^= 1u;
        }
      }
      bulk_wait_done();
    } else if (warp < kLoadWarpT && one) {
      // ---------------------------------------------------------------- MMA threads
      const bool w2 = warp == kMiscWarpT + 1;
      const uint32_t bf = w2 ? b2full : b1full, be = w2 ? b2empty : b1empty;
      const uint32_t af = w2 ? a2full : a1full, ae = w2 ? a2empty : a1empty;
      const uint32_t bo = sm + L::b1(D, NB) + (w2 ? D.bb : 0u), dc = w2 ? dcol2 : dcol1;
      uint32_t cnt = 0;
      for (unsigned tile = first; tile < ntiles; tile += step, ++cnt) {
        const uint32_t b = cnt & 1u;
        if (!mbar_wait(bf, b) || !mbar_wait(ae, b ^ 1u)) {
          ok = false;
          break;
        }
        fence_after();
        issue_tile<SL>(tmem, bo, D, dc);
        mma_commit(af);
        mma_commit(be);
      }
      mma_commit(w2 ? done2 : done1);
    }
    __syncwarp();
    warpgroup_sync();
    regs_inc<kRegsLaunch>();
  } else if (warp >= 12) {
    // ------------------------------------------------------------------ builds
    regs_inc<kRegsBuild>();
    auto role = [&](auto second) {
      constexpr bool W2 = decltype(second)::value;
      const int bt = tid - (W2 ? 640 : 384);
      const uint32_t bo = sm + L::b1(D, NB) + (W2 ? D.bb : 0u);
      uint32_t cnt = 0, ph = 0u;
      int s = 0;
      for (unsigned tile = first; tile < ntiles; tile += step, ++cnt) {
        const uint32_t b = cnt & 1u;
        // the columns' spectral values, read by epilogue 1 along with the factors
        float tv = 0.f;
        if (!W2 && bt < 32 * SL)
          tv = tmu_col(sp, (long long)(tile * SL + (unsigned)(bt >> 5)) * 32 + (bt & 31), mx, px,
                       m);
        ok = mbar_wait((W2 ? yfull : full) + 8u * s, ph);
        auto ready = [&]() -> bool {
          const bool o = mbar_wait(W2 ? b2empty : b1empty, b ^ 1u) &&
                         mbar_wait((W2 ? c2empty : c1empty) + 8u * b, ((cnt >> 1) & 1u) ^ 1u);
          if (!W2 && bt < 32 * SL) sts1f(sm + L::tmu + b * 128u * SL + (uint32_t)bt * 4u, tv);
          return o;
        };
        ok = build_lines<SL, W2, 2>(ring + (uint32_t)s * D.rb, zero, bo,
                                    sm + (W2 ? L::ci2 : L::ci1) + b * 128u * SL,
                                    sm + L::part + (W2 ? 1024u : 0u), D, bt, W2 ? 2 : 1, ok, ready);
        if (!ok) break;
        if (bt == 0) {
          mbar_arrive((W2 ? c2full : c1full) + 8u * b);
          mbar_arrive(W2 ? b2full : b1full);
        }
        if (++s == NB) {
          s = 0;
          ph ^= 1u;
        }
      }
    };
    if (warp >= 20)
      role(std::true_type{});
    else
      role(std::false_type{});
    warpgroup_sync();
    regs_dec<kRegsLaunch>();
  } else {
    // ------------------------------------------------------------------ epilogues
    regs_dec<kRegsEpi>();
    const bool w2 = warp >= 8;
    const int R = (warp & 3) * 32 + lane, r = Unit<SL>::row(R);
    const uint32_t lanes = (uint32_t)((warp & 3) * 32) << 16;
    if (w2) {
      uint32_t cnt = 0;
      int s = 0;
      for (unsigned tile = first; tile < ntiles; tile += step, ++cnt) {
        const uint32_t b = cnt & 1u;
        ok = __all_sync(0xffffffffu, mbar_wait(c2full + 8u * b, (cnt >> 1) & 1u) ? 1 : 0) != 0;
        if (ok) ok = __all_sync(0xffffffffu, mbar_wait(a2full, b) ? 1 : 0) != 0;
        if (!ok) break;
        fence_after();
        const uint32_t buf = ring + (uint32_t)s * D.rb, ci = sm + L::ci2 + b * 128u * SL;
#pragma unroll 1
        for (int i = 0; i < 4; ++i) {
          const int j = i >> 1, k = i & 1, g = Unit<SL>::g(R, j);
          float v[16];
          tmem_unit16<SL>(dcol2 + lanes, j, k, v);
          if (i == 3) {
            fence_before();
            __syncwarp();
            if (lane == 0) mbar_arrive(a2empty);  // the accumulator is free
          }
          if (r < D.h) put_row(buf, D, g, Unit<SL>::P(R, j), r, k, v, ci + (uint32_t)g * 128u);
        }
        fence_async_smem();
        __syncwarp();
        if (lane == 0) {
          mbar_arrive(c2empty + 8u * b);  // the column factors are read
          mbar_arrive(ofull + 8u * s);
        }
        if (++s == NB) s = 0;
      }
    } else {
      const int j = warp >> 2, g = Unit<SL>::g(R, j), P = Unit<SL>::P(R, j);
      const int k = 2 * r + 1 + P;  // a row past n holds zeros
      const SymRow sr = sym_row(sp, k <= n ? k : n);
      const float omth = 1.0f - sp.theta;
      uint32_t cnt = 0;
      int s = 0;
      for (unsigned tile = first; tile < ntiles; tile += step, ++cnt) {
        const uint32_t b = cnt & 1u;
        ok = __all_sync(0xffffffffu, mbar_wait(c1full + 8u * b, (cnt >> 1) & 1u) ? 1 : 0) != 0;
        if (ok) ok = __all_sync(0xffffffffu, mbar_wait(a1full, b) ? 1 : 0) != 0;
        if (!ok) break;
        fence_after();
        const uint32_t buf = ring + (uint32_t)s * D.rb;
#pragma unroll 1
        for (int h = 0; h < 2; ++h) {
          float v[16];
          tmem_unit16<SL>(dcol1 + lanes, j, h, v);
          if (h == 1) {
            fence_before();
            __syncwarp();
            if (lane == 0) mbar_arrive(a1empty);  // the accumulator is free
          }
          if (r < D.h) {
            const uint32_t a = buf + (uint32_t)(((g * 2 + P) * D.h8 + r) * 128);
            const uint32_t sw = (uint32_t)(r & 7) << 4;
            const uint32_t ci = sm + L::ci1 + b * 128u * SL + (uint32_t)g * 128u;
            const uint32_t tm = sm + L::tmu + b * 128u * SL + (uint32_t)g * 128u;
            float rs = 0.f;
#pragma unroll
            for (int c = 0; c < 4; ++c) {
              const uint32_t co = 64u * (uint32_t)h + 16u * c;
              const float4 f4 = lds4(ci + co), t4 = lds4(tm + co);
              const float f[4] = {f4.x, f4.y, f4.z, f4.w}, t[4] = {t4.x, t4.y, t4.z, t4.w};
              float o[4];
#pragma unroll
              for (int e = 0; e < 4; ++e) {
                const float y = v[4 * c + e] * f[e];
                o[e] = y * inv_sym_k<KIND>(sr, omth, t[e]);
                rs = fmaf(y, o[e], rs);
              }
              sts4f(a + (co ^ sw), o[0], o[1], o[2], o[3]);
            }
            if (tile * SL + (unsigned)g < groups) {  // not the repeat of the last group
              const float term = rs - ecomp;
              const float t = esum + term;
              ecomp = (t - esum) - term;
              esum = t;
            }
          }
        }
        __syncwarp();
        if (lane == 0) {
          mbar_arrive(c1empty + 8u * b);  // the column factors are read
          mbar_arrive(yfull + 8u * s);
        }
        if (++s == NB) s = 0;
      }
    }
    warpgroup_sync();
    regs_inc<kRegsLaunch>();
  }
  fence_before();
  const bool all_ok = __syncthreads_and(ok ? 1 : 0) != 0;
  const bool copies = __syncthreads_and(drained ? 1 : 0) != 0;
  tc_release_cols<512>(all_ok, true, done1, 0u, true, done2, 0u, tmem, S, copies);
  if (tmode != TM_NONE) {
    const double e = (double)esum - (double)ecomp;
    double tot;
    if (last_block_reduce<kNTT>(e, partials, &S->counter[CNT_TIME], gridDim.x, blockIdx.x, red,
                                &tot) &&
        tid == 0) {
      if (tmode == TM_INIT || tmode == TM_RESTART)
        minres_init_scalars_dev(S, tot);
      else
        minres_givens_dev(S, tot);
    }
  }
}

// Operand image of 8 S_len: rows of each slot (odd k = 2r + 1 for parity 0, even k = 2r + 2 for parity 1)
// in the slot's rows of the MMA, zeros elsewhere, hi and lo fp16 pieces: [slot][piece][K step][row][16].
// A block per K step and slot, a thread per row.
__global__ void __launch_bounds__(kM) k_image_tma(const __grid_constant__ SinePieces S, int len, int SL,
                                                  uint4 *img) {
  const int h = (len + 1) >> 1, KS = gridDim.x, ks = blockIdx.x, s = blockIdx.y, row = threadIdx.x;
  const int P = SL == 4 ? s >> 1 : s, r = row - (SL == 1 ? 0 : s * (kM / SL));
  uint4 hi[2], lo[2];
  image_row(S, len, h, r >= 0 && r < h ? 2 * r + 1 + P : len + 1, ks * 16, hi, lo);
  uint4 *q = img + ((size_t)(2 * s * KS + ks) * kM + row) * 2;
  q[0] = hi[0];
  q[1] = hi[1];
  q += (size_t)KS * kM * 2;
  q[0] = lo[0];
  q[1] = lo[1];
}

// ---------------------------------------------------------------- host
constexpr uint32_t kSmemMax = 227u * 1024u;

int ring_of(uint32_t fixed, uint32_t rb) {
  int nb = (int)((kSmemMax - 1024u - fixed) / rb);
  return nb > kMaxRing ? kMaxRing : nb;
}

template <int SL, bool XL>
cudaError_t launch_dst(const float *in, float *out, int len, long long cols, long long planes,
                       long long rs, long long ps, const unsigned short *img, State *S, int gk,
                       int kc, cudaStream_t st, float *user = nullptr) {
  const TmaDim D = tma_dim(len, SL);
  const int NB = ring_of(DstSmem<SL>::total(D, 0), D.rb);
  if (NB < 2) return cudaErrorInvalidConfiguration;
  uint32_t smem = DstSmem<SL>::total(D, NB);
  if (smem < 116u * 1024u) smem = 116u * 1024u;  // one block per SM: each takes all tensor memory
  CUtensorMap mi, m0, m1;
  cudaError_t e;
  unsigned groups;
  int chunks;
  if (XL) {
    chunks = (len + 1) / 32;
    groups = (unsigned)planes;  // lines
    e = tma_encode(&mi, in, len + 1, planes, 1, len + 1, (long long)(len + 1) * planes, 32 * SL);
    if (e == cudaSuccess)
      e = tma_encode(&m0, out, len + 1, planes, 1, len + 1, (long long)(len + 1) * planes, 32 * SL);
    m1 = m0;
  } else {
    chunks = (int)((cols + 31) / 32);
    groups = (unsigned)(planes * chunks);
    e = tma_encode(&mi, in, cols, len, planes, rs, ps, len);
    if (e == cudaSuccess)
      e = tma_encode(&m0, out, cols, (len + 1) / 2, planes, 2 * rs, ps, D.h);
    if (e == cudaSuccess) e = tma_encode(&m1, out + rs, cols, len / 2, planes, 2 * rs, ps, D.h);
  }
  if (e != cudaSuccess) return e;
  auto kern = k_dst_tma<SL, XL>;
  e = cudaFuncSetAttribute(kern, cudaFuncAttributeMaxDynamicSharedMemorySize, (int)smem);
  if (e != cudaSuccess) return e;
  const unsigned per = XL ? 32u * SL : (unsigned)SL;
  const unsigned ntiles = (groups + per - 1) / per;
  unsigned grid = (unsigned)time_tc_grid();
  if (ntiles < grid) grid = ntiles;
  prof_begin(kc, st);
  kern<<<grid, kNTS, smem, st>>>(mi, m0, m1, len, NB, chunks, groups, user,
                                 reinterpret_cast<const uint4 *>(img), S, gk);
  prof_end(st);
  return cudaGetLastError();
}

template <bool XL>
cudaError_t launch_dst_any(const float *in, float *out, int len, long long cols, long long planes,
                           long long rs, long long ps, const unsigned short *img, State *S, int gk,
                           int kc, cudaStream_t st, float *user = nullptr) {
  switch (slots_for(len)) {
    case 1: return launch_dst<1, XL>(in, out, len, cols, planes, rs, ps, img, S, gk, kc, st, user);
    case 2: return launch_dst<2, XL>(in, out, len, cols, planes, rs, ps, img, S, gk, kc, st, user);
    default: return launch_dst<4, XL>(in, out, len, cols, planes, rs, ps, img, S, gk, kc, st, user);
  }
}

template <int SL>
cudaError_t launch_time(float *data, const Geom &g, const Spec<float> &sp,
                        const unsigned short *img, State *S, int tmode, double *partials, int gk,
                        cudaStream_t st) {
  const TmaDim D = tma_dim(g.n, SL);
  const int NB = ring_of(TimeSmem<SL>::total(D, 0), D.rb);
  if (NB < 2) return cudaErrorInvalidConfiguration;
  uint32_t smem = TimeSmem<SL>::total(D, NB);
  if (smem < 116u * 1024u) smem = 116u * 1024u;
  const unsigned groups = (unsigned)((g.mp + 31) / 32);
  CUtensorMap mi, m0, m1;
  cudaError_t e = tma_encode(&mi, data, g.mp, g.n, 1, g.mp, g.Np, g.n);
  if (e == cudaSuccess) e = tma_encode(&m0, data, g.mp, (g.n + 1) / 2, 1, 2 * g.mp, g.Np, D.h);
  if (e == cudaSuccess) e = tma_encode(&m1, data + g.mp, g.mp, g.n / 2, 1, 2 * g.mp, g.Np, D.h);
  if (e != cudaSuccess) return e;
  auto kern = sp.prec == ST_PREC_PTHETA ? k_time_tma<SL, 2>
              : sp.scheme == ST_THETA    ? k_time_tma<SL, 0>
                                         : k_time_tma<SL, 1>;
  e = cudaFuncSetAttribute(kern, cudaFuncAttributeMaxDynamicSharedMemorySize, (int)smem);
  if (e != cudaSuccess) return e;
  const unsigned ntiles = (groups + SL - 1) / SL;
  unsigned grid = (unsigned)time_tc_grid();
  if (ntiles < grid) grid = ntiles;
  prof_begin(KC_TIME, st);
  kern<<<grid, kNTT, smem, st>>>(mi, m0, m1, g.n, NB, groups, g.mp, g.mx, g.px, sp,
                                 reinterpret_cast<const uint4 *>(img), S, tmode, partials, gk);
  prof_end(st);
  return cudaGetLastError();
}

}  // namespace

bool dst_tma_supported(int len) { return len >= 16 && len <= 256; }

size_t dst_tma_image_halves(int len) {
  const int SL = slots_for(len), hK = ((len + 1) / 2 + 15) & ~15;
  return (size_t)2 * num_slots(SL) * kM * hK;
}

cudaError_t dst_tma_build_image(int len, unsigned short *img) {
  const int SL = slots_for(len), hK = ((len + 1) / 2 + 15) & ~15;
  k_image_tma<<<dim3(hK >> 4, num_slots(SL)), kM>>>(SinePieces(len), len, SL, (uint4 *)img);
  return cudaGetLastError();
}

cudaError_t launch_dst_tma_x(const float *in, float *out, const Geom &g, const unsigned short *img,
                             State *S, int gk, cudaStream_t st, float *user) {
  return launch_dst_any<true>(in, out, g.mx, 0, (long long)g.n * g.my * g.mz, 0, 0, img, S, gk,
                              KC_DSTX, st, user);
}

// y lines: px apart, planes of px*my (one per time level and z)
cudaError_t launch_dst_tma_y(float *data, const Geom &g, const unsigned short *img, State *S,
                             int gk, cudaStream_t st) {
  return launch_dst_any<false>(data, data, g.my, g.px, (long long)g.n * g.mz, g.px,
                               (long long)g.px * g.my, img, S, gk, KC_DSTY, st);
}

// z lines (3D): px*my apart, planes of mp (one per time level)
cudaError_t launch_dst_tma_z(float *data, const Geom &g, const unsigned short *img, State *S,
                             int gk, cudaStream_t st) {
  const long long pl = (long long)g.px * g.my;
  return launch_dst_any<false>(data, data, g.mz, pl, g.n, pl, g.mp, img, S, gk, KC_DSTY, st);
}

cudaError_t launch_time_tma_single(const float *in, float *out, const Geom &g,
                                   const unsigned short *img, State *S, int gk, cudaStream_t st) {
  return launch_dst_any<false>(in, out, g.n, g.mp, 1, g.mp, g.Np, img, S, gk, KC_TIME, st);
}

cudaError_t launch_time_tma(float *data, const Geom &g, const Spec<float> &sp,
                            const unsigned short *img, State *S, int tmode, double *partials,
                            int gk, cudaStream_t st) {
  switch (slots_for(g.n)) {
    case 1: return launch_time<1>(data, g, sp, img, S, tmode, partials, gk, st);
    case 2: return launch_time<2>(data, g, sp, img, S, tmode, partials, gk, st);
    default: return launch_time<4>(data, g, sp, img, S, tmode, partials, gk, st);
  }
}

}  // namespace st
