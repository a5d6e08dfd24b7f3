// Split-precision tensor-core product kernel for sm_103a (tcgen05 + TMEM + TMA).
//
// Computes the products of the SP2 path with the hi/lo splitting of Eq.
// doubleHalf and the three-product form of Eq. MixPrecMult / Eq. mults (lo*lo
// dropped):
//     P Q ~ P_hi Q_lo + P_lo Q_hi + P_hi Q_hi,
// evaluated over a concatenated K axis, [P_hi | P_lo | P_hi] . [Q_lo ; Q_hi ; Q_hi],
// into FP32 accumulators in tensor memory: the smaller terms first, hi*hi last.
// Every right factor Q is symmetric, so its row-major planes are directly the
// K-major B operand.
//   BF16X2: bfloat16 planes, one weight for all segments.
//   BF16X3: three bfloat16 planes (hi + mid + lo = the FP32 value) and six
//           segments [P_l|P_m|P_h|P_m|P_h|P_h] . [Q_h;Q_m;Q_l;Q_h;Q_m;Q_h]: every
//           term down to 2^-16 relative, no scaling.
//   FP16X2: the lo planes hold residuals times 2^11; chunks of the hi*lo and
//           lo*hi segments are weighted by 2^-11 when they are drained from
//           TMEM. P may carry a per-matrix power-of-two scale that the epilogue
//           divides out.
// Epilogues:
//   EPI_SQUARE  X_{n+1} = sigma_n > 0 ? X_n^2 : 2 X_n - X_n^2 (Eq. DM0), upper
//               tiles only, mirrored; partials of Tr X_{n+1}, ||X_{n+1}||_F^2 and
//               ||X_n - X_n^2||_F^2 for the branch and stop decisions.
//   EPI_PLAIN   C = P Q stored as it is, or each batch entry transposed (FP32).
//   EPI_SYMM    Y_{n+1} = sigma_n > 0 ? Y_n X_n + X_n Y_n : 2 Y_n - (Y_n X_n + X_n Y_n)
//               (Eqs. DM1, DM2, DM3) for a stacked batch of symmetric Y. With X
//               and Y symmetric, (X Y)(I, J) = X(I, :) Y(:, J), so each upper tile
//               of Y X + X Y is ONE accumulation over the doubled K axis
//               [P | Q] . [Q ; P] (P = Y, Q = X): no Z buffer and no transpose
//               pass. Partials of ||Y_{n+1}||_F^2 per tile (FP16X2 plane scales).
//
// CTA tile 128 x 256, K step 64 (one 128-byte swizzle row of 16-bit values),
// 4-stage TMA -> shared-memory ring guarded by mbarriers. Persistent: one CTA
// per SM walks tiles b, b+G, b+2G, ... of a static list. The K axis is
// accumulated in chunks, alternately in two TMEM buffers, and each chunk is
// added into FP32 registers by the epilogue warps (the tensor core's own FP32
// accumulation truncates, with a bias that grows with the chunk): 256-wide for
// hi*hi, up to 16384-wide (FP16X2, weight 2^-11) or 2048-wide (bfloat16 modes,
// 2^-8) for the cross terms. A tile starts with the long chunks, so the spare
// TMEM buffer covers the previous tile's stores.
//
// CTA pairs (CG = 2, a cluster of two): a 256 x 256 tile per pair, one
// tcgen05.mma.cta_group::2 stream of M = 256 issued by rank 0. Each CTA loads
// its own 128 rows of the A tile and 128 rows of the B tile into a 6-stage ring
// of 32 KB stages and drains its own 128 accumulator rows; rank 1's warp 1
// passes each landed stage on to rank 0's barrier, and rank 1's epilogue warps
// report drained TMEM buffers there. Same arithmetic and order as one SM.
//
// Warp roles:
//   warp 0                TMA producer   } whole warps in uniform control flow, one
//   warp 1                tcgen05.mma issuer (pair: rank 1's relays stages) } elected
//                         lane issuing; warp 1 owns the TMEM allocation
//   warps 2-17            epilogue: tcgen05.ld of each chunk (warp w reads TMEM lanes
//                         32*(w%4) .. +31, the 64 columns of group (w-2)/4), then
//                         the epilogue above. With 64 columns per thread the chunk
//                         drain (the tensor pipe's critical path: the MMA warp runs
//                         at most one chunk ahead) and the tile-end stores are spread
//                         over twice as many warps as with 128.
// Every mbarrier wait is bounded in time (a launch parameter, default 2 s); on
// expiry the CTA raises the state's abort flag, waits (bounded) for its own
// copies and tensor-core operations in flight, frees its TMEM and returns, and
// later CTAs exit at once.
#include <cuda.h>

#include <stdio.h>
#include <string.h>

#include <mutex>

#include "decide.cuh"
#include "per_device.h"
#include "sp2_internal.h"
#include "tc_ptx.cuh"

namespace sp2 {

namespace {

constexpr int BM = 128;        // output rows per CTA (a CTA pair's tile has 2 BM)
constexpr int BN_FULL = 256;   // tile columns (narrower tiles: 128 and 64, on CTA pairs)
constexpr int BK = 64;
constexpr int A_BYTES = BM * BK * 2;
// Per-CTA ring geometry for CG CTAs per tile of BN columns: a CTA of a pair holds
// half of the right factor's rows, so its stage is 32 KB (BN = 256) and six stages fit.
template <int CG, int BN>
struct Ring {
  static constexpr int B_ROWS = BN / CG;
  static constexpr int B_BYTES = B_ROWS * BK * 2;
  static constexpr int STAGE_BYTES = A_BYTES + B_BYTES;
  static constexpr int STAGES = CG == 1 ? 4 : (BN == 256 ? 6 : 8);
  static constexpr int SMEM_BYTES = STAGES * STAGE_BYTES + 1024 /*align slack*/ + 256 /*barriers*/;
};
constexpr int EPI_WARPS = 16;                    // four warps per TMEM lane quarter
constexpr int EPI_THREADS = 32 * EPI_WARPS;
constexpr int NUM_THREADS = 64 + EPI_THREADS;    // TMA warp, MMA warp, epilogue warps
constexpr int COL_GROUPS = EPI_WARPS / 4;        // column groups of a tile
constexpr unsigned long long DRAIN_NS = 200000000ull;

// Instruction descriptor, kind::f16: D=F32 (bits 4-5 = 1), A and B format at
// bits 7-9 / 10-12 (BF16 = 1, F16 = 0; always the same for A and B), both
// K-major (bits 15,16 = 0), N>>3 at bit 17, M>>4 at bit 24. M is the rows of
// one instruction: BM, or 2 BM for a CTA pair.
constexpr uint32_t idesc_for(bool f16, int m, int n) {
  return (1u << 4) | ((f16 ? 0u : 1u) << 7) | ((f16 ? 0u : 1u) << 10) |
         ((uint32_t)(n >> 3) << 17) | ((uint32_t)(m >> 4) << 24);
}

// A sum of squares of FP32 values kept to about 2^-45 of its value before it goes to
// FP64, at FP32 rates (GB300's FP64 rate is a small fraction of its FP32 rate), two
// values at a time: each square enters as its rounded value plus its residual
// (exact), each addition as TwoSum (Knuth) with its rounding error carried in c. The
// packed operations are never contracted, which would lose the error terms.
__device__ __forceinline__ float two_sum(float a, float b, float& err) {
  const float t = __fadd_rn(a, b), bp = __fsub_rn(t, a);
  err = __fadd_rn(__fsub_rn(a, __fsub_rn(t, bp)), __fsub_rn(b, bp));   // a + b - t
  return t;
}
// the sum of (hi + lo) over the lanes whose indices differ in the bits W, W/2, .. 1
template <int W>
__device__ __forceinline__ void pair_sum(float& hi, float& lo) {
#pragma unroll
  for (int o = W; o > 0; o >>= 1) {
    const float gh = __shfl_xor_sync(0xffffffffu, hi, o), gl = __shfl_xor_sync(0xffffffffu, lo, o);
    float err;
    hi = two_sum(hi, gh, err);
    lo = __fadd_rn(__fadd_rn(lo, gl), err);
  }
}
struct ExactSqSum {
  uint64_t s = 0, c = 0;
  __device__ __forceinline__ void add_sq(uint64_t x) {
    const uint64_t p = mul2(x, x);
    const uint64_t e = fma2(x, x, mul2(p, kMinus1x2));   // x^2 - p exactly
    const uint64_t t = add2(s, p);
    const uint64_t bp = sub2(t, s);
    const uint64_t err = add2(sub2(s, sub2(t, bp)), sub2(p, bp));   // s + p - t
    c = add2(c, add2(err, e));
    s = t;
  }
  // both halves as one sum and its error
  __device__ __forceinline__ void fold(float& hi, float& lo) const {
    float s0, s1, c0, c1;
    upk2(s, s0, s1);
    upk2(c, c0, c1);
    float err;
    hi = two_sum(s0, s1, err);
    lo = __fadd_rn(__fadd_rn(c0, c1), err);
  }
};

// 16-bit planes of two values, packed (the first in the low half): the values'
// rounding and the residual's are those of split_bf16 / split_fp16 / split_bf16x3
__device__ __forceinline__ uint32_t cvt_bf16x2(float a, float b) {
  uint32_t r;
  asm("cvt.rn.bf16x2.f32 %0, %1, %2;" : "=r"(r) : "f"(b), "f"(a));
  return r;
}
__device__ __forceinline__ uint32_t cvt_f16x2(float a, float b) {
  uint32_t r;
  asm("cvt.rn.f16x2.f32 %0, %1, %2;" : "=r"(r) : "f"(b), "f"(a));
  return r;
}
__device__ __forceinline__ uint64_t bf16x2_floats(uint32_t h) {
  return pk2(__uint_as_float(h << 16), __uint_as_float(h & 0xffff0000u));
}

// plane kinds of the product kernel
constexpr int KIND_BF16X2 = 0, KIND_FP16X2 = 1, KIND_BF16X3 = 2;
// plane indices of an operand: 0 = hi, 1 = lo, 2 = mid (BF16X3)
constexpr int PL_HI = 0, PL_LO = 1, PL_MID = 2;

// Planes of the left and right factor in base segment `seg` of a split product
// of nbase segments (K-concatenated), smallest terms first and hi*hi last: the
// FP32 register sum then adds terms in increasing size, and a tile starts with
// the long cross-term chunks, which is what the spare TMEM buffer overlaps with
// the previous tile's stores. nbase == 1 (split-tail bulk): hi*hi alone.
template <int KIND>
__device__ __forceinline__ void seg_planes(int seg, int nbase, int& pa, int& pb) {
  if (seg == nbase - 1) {
    pa = pb = PL_HI;
  } else if constexpr (KIND == KIND_BF16X3) {
    // lh, mm, hl (2^-16 of hh), mh, hm (2^-8), then hh
    pa = seg == 0 ? PL_LO : ((seg == 1 || seg == 3) ? PL_MID : PL_HI);
    pb = seg == 2 ? PL_LO : ((seg == 1 || seg == 4) ? PL_MID : PL_HI);
  } else {
    // hl, lh, then hh
    pa = seg == 1 ? PL_LO : PL_HI;
    pb = seg == 0 ? PL_LO : PL_HI;
  }
}

// planes of two consecutive values (scale: FP16X2)
template <int KIND>
__device__ __forceinline__ void split2(float x0, float x1, float scale, uint32_t& h, uint32_t& m,
                                       uint32_t& l) {
  if constexpr (KIND == KIND_FP16X2) {
    const uint64_t v = mul2(pk2(x0, x1), pk2(scale, scale));
    float a, b;
    upk2(v, a, b);
    h = cvt_f16x2(a, b);
    const float2 hf = __half22float2(*reinterpret_cast<const __half2*>(&h));
    const uint64_t r = mul2(sub2(v, pk2(hf.x, hf.y)), pk2(kLoScale, kLoScale));
    upk2(r, a, b);
    l = cvt_f16x2(a, b);
    m = 0;
  } else {
    float a, b;
    const uint64_t v = pk2(x0, x1);
    h = cvt_bf16x2(x0, x1);
    const uint64_t r1 = sub2(v, bf16x2_floats(h));
    upk2(r1, a, b);
    if constexpr (KIND == KIND_BF16X3) {
      m = cvt_bf16x2(a, b);
      const uint64_t r2 = sub2(r1, bf16x2_floats(m));
      upk2(r2, a, b);
    } else {
      m = 0;
    }
    l = cvt_bf16x2(a, b);
  }
}

struct KParams {
  int nkb;                 // k-blocks (of BK) per segment: np / BK
  int ch;                  // k-blocks per TMEM chunk of a product's leading (hi x hi) segment
  int ch_lo;               // k-blocks per TMEM chunk of its other segments
  int nbase;               // segments of one split product (3, or 6 for BF16X3)
  int nseg;                // segments on the K axis (nbase, or 2 nbase for EPI_SYMM)
  int64_t np;
  float* out;
  uint16_t* out_hi;
  uint16_t* out_lo;
  uint16_t* out_mid;
  const float* prev;       // EPI_SQUARE: X_n; EPI_SYMM: Y_n (stacked like out)
  Part3* part;             // per-tile partials
  const Tile* tiles;
  int ntiles;
  DevState* st;
  int step;
  const float* p_scale;    // FP16X2: per batch entry of P, the plane scale to divide out
  const float* q_scale;    // FP16X2: the plane scale of Q (nullable)
  const float* o_scale;    // FP16X2 EPI_SYMM: per batch entry, scale of the output planes
  float* zmax;             // FP16X2 EPI_PLAIN: per batch entry, receives max |C|
  float* zero;             // EPI_PLAIN: nzero values cleared for the launch that follows
  int nzero;
  int trans;               // EPI_PLAIN: store each batch entry of C transposed
  unsigned long long wait_ns;
  int withhold;            // test hook: CTA 0 never issues its first load
  int tail;                // split-tail mode: st->plane1[step] selects the hi planes alone
  // block-sparse square (SPARSE kernels): the tile count, and per tile its listed
  // 256-wide K blocks klist[tix * nbk .. + kcnt[tix]], all written on the device
  const int* dyn_ntiles;
  const int* kcnt;
  const uint16_t* klist;
  int nbk;
  SimtDecide dec;          // narrow square tiles: the last CTA takes the step decision
};

// Tensor maps of one launch: the left factor's planes with 128-row boxes (A role)
// and the right factor's with 256-row boxes (B role; 128 rows for a CTA pair,
// which loads each half separately); EPI_SYMM also reads X in
// the A role and Y in the B role (its second half, [X | .] . [. ; Y]).
struct KMaps {
  CUtensorMap pa[3];   // P planes (hi, lo, mid), A role
  CUtensorMap qb[3];   // Q planes, B role
  CUtensorMap qa[3];   // Q planes, A role (EPI_SYMM)
  CUtensorMap pb[3];   // P planes, B role (EPI_SYMM)
};

// The stores and partials of one finished tile: row r of the tile, columns
// [grp * 64, grp * 64 + 64); acc holds this thread's FP32 sums; the tile's
// partials (of this CTA's rows) go to p.part[pidx]. The epilogue
// is a template parameter, so that each kernel carries only its own code (a
// smaller kernel keeps the producer's and the MMA issuer's loops in the
// instruction cache).
template <int KIND, int EPI, int TCOLS>
__device__ __forceinline__ void tile_end(const KParams& p, float (&acc)[TCOLS], int tix, int pidx,
                                         int it, int e, int lane, int grp, int r, int sg,
                                         float2 (*red)[3][EPI_WARPS]) {
  constexpr bool F16 = KIND == KIND_FP16X2;
  constexpr bool X3 = KIND == KIND_BF16X3;
  const int64_t np = p.np;
  const Tile t = p.tiles[tix];
  const int64_t bat = EPI == EPI_SQUARE ? 0 : t.row0 / (int)np;   // batch entry (stacked P)
  const int64_t gi = t.row0 + r;                               // stacked row
  const int64_t li = gi - bat * np;                            // row within its matrix
  float inv_s = 1.0f;
  if constexpr (F16) {
    if (p.p_scale) inv_s = 1.0f / p.p_scale[bat];
    if (p.q_scale) inv_s /= p.q_scale[0];
  }
  if constexpr (EPI == EPI_PLAIN) {
    float zm = 0.0f;
#pragma unroll
    for (int c0 = 0; c0 < TCOLS; c0 += 16) {
      float* dst = p.out + gi * np + t.col0 + grp * TCOLS + c0;
      float v[16];
#pragma unroll
      for (int j = 0; j < 16; ++j) {
        v[j] = acc[c0 + j] * inv_s;
        zm = fmaxf(zm, fabsf(v[j]));
      }
      if (p.trans) {   // down a column: consecutive rows (lanes) are consecutive addresses
        float* dt = p.out + bat * np * np + (int64_t)(t.col0 + grp * TCOLS + c0) * np + li;
#pragma unroll
        for (int j = 0; j < 16; ++j) {
          *dt = v[j];
          dt += np;
        }
        continue;
      }
      st256f(dst, v);
      st256f(dst + 8, v + 8);
    }
    if (p.zmax) {
      for (int o = 16; o > 0; o >>= 1) zm = fmaxf(zm, __shfl_xor_sync(0xffffffffu, zm, o));
      if (lane == 0 && zm > 0.0f) atomicMax(reinterpret_cast<int*>(&p.zmax[bat]), __float_as_int(zm));
    }
  } else {
    // X_{n+1} (EPI_SQUARE: C = X_n^2) or Y_{n+1} (EPI_SYMM: C = Y_n X_n + X_n Y_n) is
    // C for sigma > 0 and 2 M_n - C for sigma < 0 (M_n the previous iterate)
    const float os = (F16 && EPI == EPI_SYMM && p.o_scale) ? p.o_scale[bat] : 1.0f;
    const int64_t mbase = bat * np * np;   // first entry of this batch entry's matrix
    // per-thread partials over at most 64 entries of one row, the squares summed
    // with their rounding errors; lanes add pairs of FP32 words, warps and tiles FP64
    // (Tr X - ||X||_F^2 of results up to N = 4096 within 4 units in the last place of the
    // sums, as with FP64 additions over lanes): Tr, ||.||_F^2 and (EPI_SQUARE) ||X_n - X_n^2||_F^2, whose residual is
    // X_n - X_{n+1} up to its sign in either branch. Tr takes the one diagonal
    // entry a thread's row segment can hold, as it is. Entries above the diagonal
    // count twice, the diagonal once (on2, onf).
    float t1 = 0.0f, on2 = 0.0f, onf = 0.0f;
    ExactSqSum t2, f;
    const int wli = (int)li - lane;   // first row of this warp (within its matrix)
#pragma unroll
    for (int c0 = 0; c0 < TCOLS; c0 += 16) {
      const int gj0 = t.col0 + grp * TCOLS + c0;
      if (gj0 + 15 >= wli) {          // else: the whole group below the warp's rows
        // the diagonal's column within the group: entries before it enter the sums as
        // zeros and are not stored (negative: the whole row segment is above)
        const int dj = (int)li - gj0;
        float val[16];
        const float* xp = p.prev + gi * np + gj0;
#pragma unroll
        for (int hf = 0; hf < 16; hf += 8) {
          float xin[8];
          if (EPI == EPI_SQUARE || sg < 0) ld256f(xp + hf, xin);
#pragma unroll
          for (int j = 0; j < 8; ++j) {
            float v = EPI == EPI_SQUARE ? acc[c0 + hf + j] : acc[c0 + hf + j] * inv_s;
            if (sg < 0) v = 2.0f * xin[j] - v;
            val[hf + j] = v;
          }
#pragma unroll
          for (int j = 0; j < 8; j += 2) {
            const int k = hf + j;
            t2.add_sq(pk2(k > dj ? val[k] : 0.0f, k + 1 > dj ? val[k + 1] : 0.0f));
            if constexpr (EPI == EPI_SQUARE) {
              const float r0 = xin[j] - val[k], r1 = xin[j + 1] - val[k + 1];
              f.add_sq(pk2(k > dj ? r0 : 0.0f, k + 1 > dj ? r1 : 0.0f));
              onf = k == dj ? r0 : (k + 1 == dj ? r1 : onf);
            }
            on2 = k == dj ? val[k] : (k + 1 == dj ? val[k + 1] : on2);
          }
        }
        uint32_t wh[8], wl[8], wm[8];
#pragma unroll
        for (int j = 0; j < 8; ++j)
          split2<KIND>(val[2 * j], val[2 * j + 1], os, wh[j], wm[j], wl[j]);
        const int64_t o = gi * np + gj0;          // this row segment
        if (dj <= 0) {
          st256f(p.out + o, val);
          st256f(p.out + o + 8, val + 8);
          st256(p.out_hi + o, wh);
          st256(p.out_lo + o, wl);
          if constexpr (X3) st256(p.out_mid + o, wm);
        } else {
#pragma unroll
          for (int j = 0; j < 16; ++j) {
            const int sh = 16 * (j & 1);
            if (j >= dj) {
              p.out[o + j] = val[j];
              p.out_hi[o + j] = (uint16_t)(wh[j >> 1] >> sh);
              p.out_lo[o + j] = (uint16_t)(wl[j >> 1] >> sh);
              if constexpr (X3) p.out_mid[o + j] = (uint16_t)(wm[j >> 1] >> sh);
            }
          }
        }
        // its mirror, down a column
        int64_t om = mbase + (int64_t)gj0 * np + li;
#pragma unroll
        for (int j = 0; j < 16; ++j) {
          const int sh = 16 * (j & 1);
          if (j > dj) {
            p.out[om] = val[j];
            p.out_hi[om] = (uint16_t)(wh[j >> 1] >> sh);
            p.out_lo[om] = (uint16_t)(wl[j >> 1] >> sh);
            if constexpr (X3) p.out_mid[om] = (uint16_t)(wm[j >> 1] >> sh);
          }
          om += np;
        }
      }
    }
    t1 = on2;
    // This thread's sums as FP32 pairs (hi + lo), entries above the diagonal twice and
    // the diagonal's square, exactly, beside them. The warp adds pairs (one exchange
    // puts ||.||_F^2 into its lower half and f into its upper), and only the tile's sums
    // over warps are FP64: an FP64 instruction of a warp takes 64 clocks, and the
    // shuffled additions of 16 warps took a third of a narrow tile's end. A pair keeps
    // about 2^-46 of its value, as the threads' sums do.
    float h2, l2, h3, l3;
    t2.fold(h2, l2);
    f.fold(h3, l3);
    h2 *= 2.0f, l2 *= 2.0f, h3 *= 2.0f, l3 *= 2.0f;
    const bool diag = t.col0 + grp * TCOLS <= wli + 31;   // may hold diagonal entries
    const bool up = lane >= 16;
    const int pb = it & 1;
    if (diag) {
      const float p2 = __fmul_rn(on2, on2), pf = __fmul_rn(onf, onf);
      float err, l1 = 0.0f;
      h2 = two_sum(h2, p2, err);
      l2 = __fadd_rn(l2, __fadd_rn(err, fmaf(on2, on2, -p2)));
      h3 = two_sum(h3, pf, err);
      l3 = __fadd_rn(l3, __fadd_rn(err, fmaf(onf, onf, -pf)));
      pair_sum<16>(t1, l1);
      if (lane == 0) red[pb][0][e] = make_float2(t1, l1);
    } else if (lane == 0) {
      red[pb][0][e] = make_float2(0.0f, 0.0f);
    }
    {
      const float gh = __shfl_xor_sync(0xffffffffu, up ? h2 : h3, 16);
      const float gl = __shfl_xor_sync(0xffffffffu, up ? l2 : l3, 16);
      float err, h = two_sum(up ? h3 : h2, gh, err);
      float l = __fadd_rn(__fadd_rn(up ? l3 : l2, gl), err);
      pair_sum<8>(h, l);
      if ((lane & 15) == 0) red[pb][up ? 2 : 1][e] = make_float2(h, l);
    }
    // epilogue warps only (named barrier 1): one warp adds the tile's partials in FP64
    asm volatile("bar.sync 1, %0;" ::"r"(EPI_THREADS) : "memory");
    if (e == 0) {
      const float2 v = red[pb][up ? 2 : 1][lane & 15];
      double s = (double)v.x + (double)v.y, s1 = 0.0;
      for (int o = 8; o > 0; o >>= 1) s += __shfl_xor_sync(0xffffffffu, s, o);
      if (t.col0 < (int)(t.row0 - bat * np) + 2 * BM) {   // the tile meets the diagonal
        const float2 w = red[pb][0][lane & 15];
        s1 = (double)w.x + (double)w.y;
        for (int o = 8; o > 0; o >>= 1) s1 += __shfl_xor_sync(0xffffffffu, s1, o);
      }
      const double s3 = __shfl_sync(0xffffffffu, s, 16);
      if (lane == 0) p.part[pidx] = Part3{s1, s, s3};
    }
  }
}

// Block-sparse squares: the end (exclusive) of the run of listed K blocks that
// starts at list position q0 and stays inside one dense cross-term chunk (gsz
// blocks of 256), so that with every block listed the chunks are the dense ones.
__device__ __forceinline__ int sparse_run_end(const uint16_t* kl, int kc, int gsz, int q0) {
  const int grp = kl[q0] / gsz;
  int q1 = q0 + 1;
  while (q1 < kc && kl[q1] / gsz == grp) ++q1;
  return q1;
}

// SPARSE (square on CTA pairs only): the tile list, its length and every tile's
// K blocks come from the device (the block-sparse plan); a tile's K axis is its
// listed 256-wide blocks in each segment, hi*hi drained per block and a cross
// term per run of listed blocks inside one dense cross-term chunk, so that with
// every block listed the chunks, and the results, are the dense kernel's. The
// sparse loops are separate from the dense ones, which the SPARSE = false
// kernels alone contain.
template <int KIND, int EPI, int CG, int BN = BN_FULL, bool SPARSE = false>
__global__ void __launch_bounds__(NUM_THREADS, 1)
k_gemm_tc(const __grid_constant__ KMaps maps, const __grid_constant__ KParams p) {
  static_assert(!SPARSE || (EPI == EPI_SQUARE && CG == 2), "block-sparse squares run on pairs");
  static_assert(BN == BN_FULL || CG == 2, "narrow tiles run on pairs");
  using R = Ring<CG, BN>;
  constexpr uint32_t ACC_COLS = BN;                // one 128 x BN FP32 accumulator
  constexpr uint32_t TMEM_COLS = 2 * ACC_COLS;     // two chunk buffers
  constexpr int TCOLS = BN / COL_GROUPS;           // columns per epilogue thread
  constexpr int STAGES = R::STAGES;
  constexpr int STAGE_BYTES = R::STAGE_BYTES;
  constexpr bool PAIR = CG == 2;
  constexpr bool F16 = KIND == KIND_FP16X2;
  constexpr uint32_t kIdesc = idesc_for(F16, BM * CG, BN);
  DevState* st = p.st;
  extern __shared__ uint8_t smem_raw[];
  uint8_t* smem = reinterpret_cast<uint8_t*>((reinterpret_cast<uintptr_t>(smem_raw) + 1023) &
                                             ~(uintptr_t)1023);
  uint64_t* full = reinterpret_cast<uint64_t*>(smem + STAGES * STAGE_BYTES);
  uint64_t* empty = full + STAGES;
  uint64_t* pfull = empty + STAGES;   // pair, rank 0: the peer's stage s has landed
  uint64_t* tfull = pfull + STAGES;   // [2] chunk accumulated in TMEM buffer b
  uint64_t* tempty = tfull + 2;       // [2] TMEM buffer b drained by the epilogue warps
  uint64_t* mdone = tempty + 2;       // abort path: the MMA issuer's last operations done
  uint32_t* tmem_slot = reinterpret_cast<uint32_t*>(mdone + 1);
  __shared__ float2 red[2][3][EPI_WARPS];   // per-tile partials (FP32 pairs), double-buffered by tile parity

  // (uniform over the warp, also to the compiler)
  const int warp = __shfl_sync(0xffffffffu, (int)(threadIdx.x >> 5), 0), lane = threadIdx.x & 31;
  int* abortf = &st->abort_flag;
  // a pair: each CTA loads its own halves of both operands (rows rank*128 .. of the
  // A tile and of the B tile) and drains its own TMEM rows; rank 0 issues the MMAs
  // once its own stage and (relayed by rank 1's warp 1) the peer's have landed.
  // Tiles are indexed per pair.
  const uint32_t rank = PAIR ? cluster_rank() : 0u;
  const bool issuer = rank == 0;
  const int unit = PAIR ? (int)(blockIdx.x >> 1) : (int)blockIdx.x;
  const int nunits = PAIR ? (int)(gridDim.x >> 1) : (int)gridDim.x;
  if (threadIdx.x == 0) {
    for (int s = 0; s < STAGES; ++s) {
      mbar_init(&full[s], 1);
      mbar_init(&empty[s], 1);
      mbar_init(&pfull[s], 1);
    }
    for (int b = 0; b < 2; ++b) {
      mbar_init(&tfull[b], 1);
      mbar_init(&tempty[b], CG * EPI_WARPS);   // a pair's rank 0 hears both CTAs' warps
    }
    mbar_init(mdone, 1);
    asm volatile("fence.mbarrier_init.release.cluster;" ::: "memory");
    asm volatile("prefetch.tensormap [%0];" ::"l"(reinterpret_cast<uint64_t>(&maps.pa[0])) : "memory");
    asm volatile("prefetch.tensormap [%0];" ::"l"(reinterpret_cast<uint64_t>(&maps.qb[0])) : "memory");
  }
  if (warp == 1) {
    // a pair allocates the same columns in both CTAs, one warp of each taking part
    if constexpr (PAIR) {
      asm volatile("tcgen05.alloc.cta_group::2.sync.aligned.shared::cta.b32 [%0], %1;" ::"r"(
                       smem_u32(tmem_slot)),
                   "r"(TMEM_COLS)
                   : "memory");
      asm volatile("tcgen05.relinquish_alloc_permit.cta_group::2.sync.aligned;" ::: "memory");
    } else {
      asm volatile("tcgen05.alloc.cta_group::1.sync.aligned.shared::cta.b32 [%0], %1;" ::"r"(
                       smem_u32(tmem_slot)),
                   "r"(TMEM_COLS)
                   : "memory");
      asm volatile("tcgen05.relinquish_alloc_permit.cta_group::1.sync.aligned;" ::: "memory");
    }
  }
  tc_fence_before();
  __syncthreads();
  if constexpr (PAIR) cluster_sync();
  tc_fence_after();
  const uint32_t tmem = *tmem_slot;

  // Up to here nothing of the launches before is read: the barriers' and TMEM's setup
  // (2500 clocks) overlaps their end. A halted launch runs no tile (stop_at is fixed
  // for the launch, so a pair agrees; the abort flag is seen in the waits).
  dep_sync();
  const int stopped = *((volatile const int*)&st->stop_at);
  const bool halted = stopped != 0 && p.step > stopped;
  // segments of this launch: the split product, or in the split-tail mode's bulk
  // steps the hi planes alone (one segment; two for the symmetric response)
  const int nbase = (p.tail && st->plane1[p.step]) ? 1 : p.nbase;
  const int nseg = EPI == EPI_SYMM ? 2 * nbase : nbase;
  const int total_kb = nseg * p.nkb;
  // TMEM chunks: the hi x hi segment of each split product (the last of its
  // nbase segments; every segment in the split-tail bulk) every ch k-blocks, the
  // smaller cross terms every ch_lo; both divide nkb, so no chunk spans two segments
  const int ch_hi = p.ch, ch_lo = nbase == 1 ? p.ch : p.ch_lo;
  const int nchunks = (nseg / nbase) * (p.nkb / ch_hi + (nbase - 1) * (p.nkb / ch_lo));
  auto chunk_len = [&](int kb0) {
    return ((kb0 / p.nkb) % nbase) == nbase - 1 ? ch_hi : ch_lo;
  };
  // persistent static schedule: this CTA (pair) handles tiles unit, unit + nunits, ...
  // (block-sparse: the tile count comes from the device)
  int ntiles = p.ntiles;
  if constexpr (SPARSE) ntiles = *((volatile const int*)p.dyn_ntiles);
  const int my_tiles = !halted && unit < ntiles ? (ntiles - 1 - unit) / nunits + 1 : 0;
  // block-sparse: a cross-term chunk is a run of listed K blocks inside one dense
  // chunk of ch_lo k-blocks (gsz K blocks of 256)
  const int gsz = p.ch_lo >> 2;

  if constexpr (EPI == EPI_PLAIN) {
    if (blockIdx.x == 0 && !halted)
      for (int i = threadIdx.x; i < p.nzero; i += NUM_THREADS) p.zero[i] = 0.0f;
  }

  if (warp == 0) {
    // copy issuer: the whole warp (the waits by every lane, the copies by an elected one)
    const uint32_t ring = smem_u32(smem);
    if constexpr (SPARSE) {
      // block-sparse square: every segment walks the tile's listed K blocks
      int64_t g = 0;
      RingPos<STAGES> rp;
      bool ok = true;
      for (int it = 0; it < my_tiles && ok; ++it) {
        const int tix = unit + it * nunits;
        const Tile t = p.tiles[tix];
        const int kc = p.kcnt[tix];
        const uint16_t* kl = p.klist + (int64_t)tix * p.nbk;
        for (int seg = 0; seg < nseg && ok; ++seg) {
          int pa, pb;
          seg_planes<KIND>(seg, nbase, pa, pb);
          for (int u = 0; u < 4 * kc; ++u, ++g, rp.next()) {
            const int s = rp.s;
            const uint32_t ph = rp.ph;
            ok = __all_sync(0xffffffffu, mbar_wait<PAIR>(&empty[s], ph ^ 1u, abortf, p.wait_ns));
            if (!ok) break;
            if (p.withhold && blockIdx.x == 0 && g == 0) continue;  // test hook: never completes
            const int kx = (int)kl[u >> 2] * (4 * BK) + (u & 3) * BK;
            const uint32_t sa = ring + (uint32_t)(s * STAGE_BYTES);
            tma_load_stage(&full[s], STAGE_BYTES, &maps.pa[pa], &maps.qb[pb], sa, sa + A_BYTES, kx,
                           t.row0 + (int)rank * BM, t.col0 + (int)rank * R::B_ROWS);
          }
        }
      }
      if (!ok) {
        const int64_t first = g > STAGES ? g - STAGES : 0;
        for (int64_t q = first; q < g; ++q) {
          if (p.withhold && blockIdx.x == 0 && q == 0) continue;
          mbar_wait_drain(&full[q % STAGES], (uint32_t)(q / STAGES) & 1u, DRAIN_NS);
        }
      }
    } else {
      const int64_t np = p.np;
      const int nkb = p.nkb;
      // k-block counter g runs on across tiles: stage g % STAGES, phase (g / STAGES) & 1
      int64_t g = 0;
      RingPos<STAGES> rp;
      bool ok = true;
      for (int it = 0; it < my_tiles && ok; ++it) {
        const Tile t = p.tiles[unit + it * nunits];
        const int bat = (int)(t.row0 / np);
        for (int seg = 0; seg < nseg && ok; ++seg) {
          // the segment's operands and tile rows, fixed over its k-blocks
          const bool swap = EPI == EPI_SYMM && seg >= nbase;   // second half: [Q | .] . [. ; P]
          int pa, pb;
          seg_planes<KIND>(swap ? seg - nbase : seg, nbase, pa, pb);
          const CUtensorMap* ma = swap ? &maps.qa[pa] : &maps.pa[pa];
          const CUtensorMap* mb = swap ? &maps.pb[pb] : &maps.qb[pb];
          // this CTA's halves: rows [rank*128, +128) of the A tile, [rank*B_ROWS, +B_ROWS)
          // of the B tile (one CTA: all of both)
          const int arow = (swap ? t.row0 - bat * (int)np : t.row0) + (int)rank * BM;
          const int brow = (swap ? bat * (int)np + t.col0 : t.col0) + (int)rank * R::B_ROWS;
          for (int kx = 0; kx < nkb * BK; kx += BK, ++g, rp.next()) {
            const int s = rp.s;
            ok = __all_sync(0xffffffffu, mbar_wait<PAIR>(&empty[s], rp.ph ^ 1u, abortf, p.wait_ns));
            if (!ok) break;
            if (p.withhold && blockIdx.x == 0 && g == 0) continue;  // test hook: never completes
            const uint32_t sa = ring + (uint32_t)(s * STAGE_BYTES);
            tma_load_stage(&full[s], STAGE_BYTES, ma, mb, sa, sa + A_BYTES, kx, arow, brow);
          }
        }
      }
      if (!ok) {
        // aborted: let the copies already issued land before the CTA exits
        const int64_t first = g > STAGES ? g - STAGES : 0;
        for (int64_t q = first; q < g; ++q) {
          if (p.withhold && blockIdx.x == 0 && q == 0) continue;
          mbar_wait_drain(&full[q % STAGES], (uint32_t)(q / STAGES) & 1u, DRAIN_NS);
        }
      }
    }
  } else if (warp == 1) {
    if (PAIR && !issuer) {
     if (lane == 0) {
      // rank 1: pass each landed stage of this CTA on to rank 0's MMA issuer
      const uint32_t pfull_peer = cluster_addr(smem_u32(pfull), 0);
      int64_t total = (int64_t)my_tiles * total_kb;
      if constexpr (SPARSE) {
        total = 0;
        for (int it = 0; it < my_tiles; ++it) total += (int64_t)nseg * 4 * p.kcnt[unit + it * nunits];
      }
      RingPos<STAGES> rp;
      for (int64_t g = 0; g < total; ++g, rp.next()) {
        if (!mbar_wait<PAIR>(&full[rp.s], rp.ph, abortf, p.wait_ns)) break;
        mbar_arrive_cluster_release(pfull_peer + (uint32_t)(rp.s * sizeof(uint64_t)));
      }
     }
    } else if constexpr (SPARSE) {
      bool ok = true;
      int64_t g = 0, gc = 0;
      RingPos<STAGES> rp;
      const uint64_t adesc0 = sdesc_sw128(smem_u32(smem));
      for (int it = 0; it < my_tiles && ok; ++it) {
        const int tix = unit + it * nunits;
        const int kc = p.kcnt[tix];
        const uint16_t* kl = p.klist + (int64_t)tix * p.nbk;
        for (int seg = 0; seg < nseg && ok; ++seg) {
          const bool hh = seg == nbase - 1;
          for (int q0 = 0; q0 < kc && ok; ++gc) {
            const int q1 = hh ? q0 + 1 : sparse_run_end(kl, kc, gsz, q0);
            const int b = (int)(gc & 1);
            ok = __all_sync(0xffffffffu, mbar_wait<PAIR>(&tempty[b], ((uint32_t)(gc >> 1) & 1u) ^ 1u,
                                                        abortf, p.wait_ns));
            if (!ok) break;
            tc_fence_after();
            const uint32_t dtm = tmem + (uint32_t)b * ACC_COLS;
            for (int u = 4 * q0; u < 4 * q1; ++u, ++g, rp.next()) {
              const int s = rp.s;
              const uint32_t ph = rp.ph;
              ok = __all_sync(0xffffffffu, mbar_wait<false>(&full[s], ph, abortf, p.wait_ns) &&
                                               mbar_wait<PAIR>(&pfull[s], ph, abortf, p.wait_ns));
              if (!ok) break;
              tc_fence_after();
              const uint64_t adesc = adesc0 + (uint64_t)(s * (STAGE_BYTES >> 4));
              const uint64_t bdesc = adesc + (uint64_t)(A_BYTES >> 4);
              umma_kblock<CG>(dtm, adesc, bdesc, kIdesc, u > 4 * q0 ? 1u : 0u);
              umma_commit_both(&empty[s]);
            }
            if (ok) umma_commit_both(&tfull[b]);
            q0 = q1;
          }
        }
      }
      if (!ok) {
        umma_commit<CG>(mdone);
        mbar_wait_drain(mdone, 0, DRAIN_NS);
      }
    } else {
      // whole warp (the waits by every lane, the instructions by an elected one)
      bool ok = true;
      int64_t g = 0, gc = 0;   // k-block and chunk counters across tiles
      RingPos<STAGES> rp;
      // descriptors of a stage: the ring's base descriptor plus the stage offset in
      // 16-byte units (the address field holds bits 4-17 of a shared-memory address
      // below 256 KB, so the addition never carries out of it)
      const uint64_t adesc0 = sdesc_sw128(smem_u32(smem));
      for (int it = 0; it < my_tiles && ok; ++it) {
        int kb0 = 0;   // first k-block of chunk c within the tile
        int segb = 0, kin = 0;   // base segment (seg % nbase) and k-block within the segment
        for (int c = 0; c < nchunks && ok; ++c, ++gc) {
          const int len = segb == nbase - 1 ? ch_hi : ch_lo;   // chunk_len(kb0), no division
          kin += len;
          if (kin == p.nkb) {
            kin = 0;
            if (++segb == nbase) segb = 0;
          }
          const int b = (int)(gc & 1);
          // the epilogue (of both CTAs of a pair) has drained buffer b (chunk gc-2)
          ok = __all_sync(0xffffffffu, mbar_wait<PAIR>(&tempty[b], ((uint32_t)(gc >> 1) & 1u) ^ 1u,
                                                      abortf, p.wait_ns));
          if (!ok) break;
          tc_fence_after();
          const uint32_t dtm = tmem + (uint32_t)b * ACC_COLS;
          for (int kb = kb0; kb < kb0 + len; ++kb, ++g, rp.next()) {
            const int s = rp.s;
            const uint32_t ph = rp.ph;
            // this CTA's own stage (its own copies: CTA-scope acquire), then, on a
            // pair, the peer's stage as relayed by its warp 1
            ok = __all_sync(0xffffffffu,
                            mbar_wait<false>(&full[s], ph, abortf, p.wait_ns) &&
                                (!PAIR || mbar_wait<PAIR>(&pfull[s], ph, abortf, p.wait_ns)));
            if (!ok) break;
            tc_fence_after();
            const uint64_t adesc = adesc0 + (uint64_t)(s * (STAGE_BYTES >> 4));
            const uint64_t bdesc = adesc + (uint64_t)(A_BYTES >> 4);
            umma_kblock<CG>(dtm, adesc, bdesc, kIdesc, kb > kb0 ? 1u : 0u);
            // the stage is free in both CTAs once these MMAs have read it
            if constexpr (PAIR) umma_commit_both(&empty[s]);
            else umma_commit<CG>(&empty[s]);
          }
          if (ok) {
            if constexpr (PAIR) umma_commit_both(&tfull[b]);
            else umma_commit<CG>(&tfull[b]);
          }
          kb0 += len;
        }
      }
      if (!ok) {
        // aborted: the tensor-core operations already issued still read the ring and
        // write TMEM; one more commit tracks all of them (bounded wait) before dealloc
        umma_commit<CG>(mdone);
        mbar_wait_drain(mdone, 0, DRAIN_NS);
      }
    }
  } else {
    // epilogue warps 2 .. 2+EPI_WARPS-1: warp w reads TMEM lanes 32*(w%4) .. +31 and
    // columns [grp*64, grp*64+64). Each K chunk is drained from TMEM into
    // FP32 registers with round-to-nearest adds; the tile's stores follow while
    // the MMA warp already fills the freed TMEM buffers with the next tile's chunks.
    // The drain loop is the tensor pipe's critical path (the MMA warp runs at most
    // one chunk ahead), so it keeps nothing live beyond the accumulator.
    const int e = warp - 2;
    const int q = warp & 3;
    const int grp = e >> 2;
    const int r = (int)rank * BM + q * 32 + lane;   // row within the (pair) tile
    const uint32_t trow = tmem + ((uint32_t)(q * 32) << 16) + (uint32_t)(grp * TCOLS);
    // a pair's rank 1 reports drained buffers to rank 0's barrier
    const uint32_t tempty_peer = PAIR && !issuer ? cluster_addr(smem_u32(tempty), 0) : 0u;
    // the branch of this step (uniform over the launch); the previous iterate is
    // read by the square and, for sigma < 0, by the response update
    const int sg = EPI == EPI_PLAIN ? 1 : p.st->sigma[p.step];
    const bool need_prev = EPI == EPI_SQUARE || (EPI == EPI_SYMM && sg < 0);
    bool ok = true;
    int64_t gc = 0;
    for (int it = 0; it < my_tiles && ok; ++it) {
      const int tix = unit + it * nunits;
      // the previous-iterate entries the tile-end epilogue reads (256 B of this
      // thread's row), pulled into L2 two chunks ahead of the tile's end
      const float* pf = nullptr;
      if (need_prev) {
        const Tile t = p.tiles[tix];
        pf = p.prev + ((int64_t)t.row0 + r) * p.np + t.col0 + grp * TCOLS;
      }
      float acc[TCOLS];
#pragma unroll
      for (int j = 0; j < TCOLS; ++j) acc[j] = 0.0f;
      if constexpr (SPARSE) {
        // the listed K blocks: hi*hi chunks one block each, cross-term chunks by runs
        const int kc = p.kcnt[tix];
        const uint16_t* kl = p.klist + (int64_t)tix * p.nbk;
        int nruns = 0;
        for (int q0 = 0; q0 < kc; q0 = sparse_run_end(kl, kc, gsz, q0)) ++nruns;
        const int nch = (nbase - 1) * nruns + kc;
        int c = 0;
        for (int seg = 0; seg < nseg && ok; ++seg) {
          const bool hh = seg == nbase - 1;
          for (int q0 = 0; q0 < kc; ++c, ++gc) {
            q0 = hh ? q0 + 1 : sparse_run_end(kl, kc, gsz, q0);
            const int b = (int)(gc & 1);
            bool w = mbar_wait<PAIR>(&tfull[b], (uint32_t)(gc >> 1) & 1u, abortf, p.wait_ns);
            w = __all_sync(0xffffffffu, w);
            if (!w) {
              ok = false;
              break;
            }
            tc_fence_after();
            if (pf && c == nch - 2)
              asm volatile("cp.async.bulk.prefetch.L2.global [%0], %1;" ::"l"(pf),
                           "r"((uint32_t)(TCOLS * sizeof(float)))
                           : "memory");
            float wgt = 1.0f;
            if constexpr (F16) wgt = hh ? 1.0f : 1.0f / kLoScale;
#pragma unroll
            for (int c0 = 0; c0 < TCOLS; c0 += 16) {
              uint32_t v[16];
              tmem_ld16(trow + (uint32_t)b * ACC_COLS + (uint32_t)c0, v);
#pragma unroll
              for (int j = 0; j < 16; ++j) acc[c0 + j] = fmaf(wgt, __uint_as_float(v[j]), acc[c0 + j]);
            }
            tc_fence_before();
            __syncwarp();
            if (lane == 0) {
              if (!issuer)
                mbar_arrive_cluster(tempty_peer + (uint32_t)(b * sizeof(uint64_t)));
              else
                mbar_arrive(&tempty[b]);
            }
          }
        }
        if (!ok || *((volatile int*)abortf)) break;
        tile_end<KIND, EPI, TCOLS>(p, acc, tix, tix * CG + (int)rank, it, e, lane, grp, r, sg, red);
        continue;
      }
      int kb0 = 0;
      for (int c = 0; c < nchunks; ++c, ++gc) {
        const int b = (int)(gc & 1);
        const int seg = kb0 / p.nkb;
        kb0 += chunk_len(kb0);
        bool w = mbar_wait<PAIR>(&tfull[b], (uint32_t)(gc >> 1) & 1u, abortf, p.wait_ns);
        w = __all_sync(0xffffffffu, w);
        if (!w) {
          ok = false;
          break;
        }
        tc_fence_after();
        if (pf && c == nchunks - 2)
          asm volatile("cp.async.bulk.prefetch.L2.global [%0], %1;" ::"l"(pf),
                       "r"((uint32_t)(TCOLS * sizeof(float)))
                       : "memory");
        float wgt = 1.0f;
        if constexpr (F16) wgt = (seg % nbase) == nbase - 1 ? 1.0f : 1.0f / kLoScale;
#pragma unroll
        for (int c0 = 0; c0 < TCOLS; c0 += 16) {
          uint32_t v[16];
          tmem_ld16(trow + (uint32_t)b * ACC_COLS + (uint32_t)c0, v);
#pragma unroll
          for (int j = 0; j < 16; ++j) acc[c0 + j] = fmaf(wgt, __uint_as_float(v[j]), acc[c0 + j]);
        }
        tc_fence_before();
        __syncwarp();
        if (lane == 0) {
          if (PAIR && !issuer)
            mbar_arrive_cluster(tempty_peer + (uint32_t)(b * sizeof(uint64_t)));
          else
            mbar_arrive(&tempty[b]);
        }
      }
      if (!ok || *((volatile int*)abortf)) break;
      tile_end<KIND, EPI, TCOLS>(p, acc, tix, tix * CG + (int)rank, it, e, lane, grp, r, sg, red);
    }
  }

  // a CTA (pair) leaves only when every copy into its shared memory and every
  // tensor-core operation on its TMEM is done or drained above
  tc_fence_before();
  __syncthreads();
  if constexpr (PAIR) cluster_sync();
  if (warp == 1) {
    __syncwarp();
    tc_fence_after();
    if constexpr (PAIR)
      asm volatile("tcgen05.dealloc.cta_group::2.sync.aligned.b32 %0, %1;" ::"r"(tmem),
                   "r"(TMEM_COLS)
                   : "memory");
    else
      asm volatile("tcgen05.dealloc.cta_group::1.sync.aligned.b32 %0, %1;" ::"r"(tmem),
                   "r"(TMEM_COLS)
                   : "memory");
  }
  if constexpr (EPI == EPI_SQUARE && BN < BN_FULL) {
    // the last CTA to get here takes the step decision (the wide-tile kernels leave
    // it to its own launch: its code beside theirs costs them instruction cache)
    if (p.dec.done && !halted) last_block_decides(p.part, p.dec);
  }
}

// The tensor maps of a launch are a function of its plane addresses, shapes and
// box sizes alone, and a solve uses a handful of such combinations (the two X
// buffers, the response buffers), so they are encoded once and reused: encoding
// the twelve maps of a launch anew cost tens of microseconds of host time per
// step, which bounds the step rate of small problems. A small table, replaced
// round robin, shared by every thread of the process.
struct MapKey {
  const void* planes[6];
  int64_t prows, qrows, np;
  int cg, bn, f16;
};

bool cached_maps(const MapKey& k, KMaps* out) {
  constexpr int kSlots = 32;
  static std::mutex mu;
  static MapKey keys[kSlots];
  static KMaps maps[kSlots];
  static bool used[kSlots] = {};
  static int next = 0;
  std::lock_guard<std::mutex> lock(mu);
  for (int i = 0; i < kSlots; ++i)
    if (used[i] && memcmp(&keys[i], &k, sizeof k) == 0) {
      *out = maps[i];
      return true;
    }
  KMaps m;
  bool ok = true;
  for (int i = 0; i < 3; ++i) {
    ok = ok && make_map(&m.pa[i], k.planes[i], k.prows, k.np, BM, k.f16) &&
         make_map(&m.qb[i], k.planes[3 + i], k.qrows, k.np, k.bn / k.cg, k.f16);
    // EPI_SYMM's second half reads X as the left and Y as the right factor
    ok = ok && make_map(&m.qa[i], k.planes[3 + i], k.qrows, k.np, BM, k.f16) &&
         make_map(&m.pb[i], k.planes[i], k.prows, k.np, k.bn / k.cg, k.f16);
  }
  if (!ok) return false;
  keys[next] = k;
  maps[next] = m;
  used[next] = true;
  next = (next + 1) % kSlots;
  *out = m;
  return true;
}

// one launch of the (KIND, EPI, CG) kernel over `units` CTAs or CTA pairs (at most
// the resident ones), with its shared-memory attribute and its resident-pair
// count queried once
template <int KIND, int EPI, int CG, int BN = BN_FULL, bool SPARSE = false>
cudaError_t launch_kind(const KMaps& maps, const KParams& p, int units, cudaStream_t s) {
  auto kern = k_gemm_tc<KIND, EPI, CG, BN, SPARSE>;
  constexpr int smem = Ring<CG, BN>::SMEM_BYTES;
  static PerDevice kept;   // CTAs (pairs) resident at a time
  int dev = 0, resident = 0;
  cudaError_t e = cudaGetDevice(&dev);
  if (e != cudaSuccess) return e;
  e = kept.get(dev, cudaErrorInvalidDevice, &resident, [&](int* res) {
    int nsm = 0;
    cudaError_t r = cudaFuncSetAttribute(kern, cudaFuncAttributeMaxDynamicSharedMemorySize, smem);
    if (r == cudaSuccess) r = cudaDeviceGetAttribute(&nsm, cudaDevAttrMultiProcessorCount, dev);
    if (r != cudaSuccess) return r;
    if (CG == 1) {
      *res = nsm;   // one CTA per SM: the ring leaves no room for a second
      return cudaSuccess;
    }
    cudaLaunchConfig_t cfg = {};
    cudaLaunchAttribute at[1];
    at[0].id = cudaLaunchAttributeClusterDimension;
    at[0].val.clusterDim.x = CG;
    at[0].val.clusterDim.y = 1;
    at[0].val.clusterDim.z = 1;
    cfg.gridDim = dim3((unsigned)(CG * (nsm / CG)));
    cfg.blockDim = dim3(NUM_THREADS);
    cfg.dynamicSmemBytes = smem;
    cfg.attrs = at;
    cfg.numAttrs = 1;
    r = cudaOccupancyMaxActiveClusters(res, kern, &cfg);
    return r == cudaSuccess && *res < 1 ? cudaErrorNotSupported : r;
  });
  if (e != cudaSuccess) return e;
  const int n = units < resident ? units : resident;
  if (CG == 1) return launch_dep(kern, n, NUM_THREADS, smem, s, maps, p);
  cudaLaunchConfig_t cfg = {};
  cudaLaunchAttribute at[2];
  at[1].id = cudaLaunchAttributeProgrammaticStreamSerialization;
  at[1].val.programmaticStreamSerializationAllowed = 1;
  at[0].id = cudaLaunchAttributeClusterDimension;
  at[0].val.clusterDim.x = CG;
  at[0].val.clusterDim.y = 1;
  at[0].val.clusterDim.z = 1;
  cfg.gridDim = dim3((unsigned)(CG * n));
  cfg.blockDim = dim3(NUM_THREADS);
  cfg.dynamicSmemBytes = smem;
  cfg.stream = s;
  cfg.attrs = at;
  cfg.numAttrs = SPARSE ? 1 : 2;   // (block-sparse steps lose by early residency)
  return cudaLaunchKernelEx(&cfg, kern, maps, p);
}

template <int KIND, int CG>
cudaError_t launch_epi(int epi, const KMaps& maps, const KParams& p, int units, cudaStream_t s) {
  if (epi == EPI_SQUARE) return launch_kind<KIND, EPI_SQUARE, CG>(maps, p, units, s);
  if (epi == EPI_SYMM) return launch_kind<KIND, EPI_SYMM, CG>(maps, p, units, s);
  return launch_kind<KIND, EPI_PLAIN, CG>(maps, p, units, s);
}

// narrow tiles (BN < 256) on CTA pairs
template <int KIND, int BN>
cudaError_t launch_narrow(int epi, const KMaps& maps, const KParams& p, int units, cudaStream_t s) {
  if (epi == EPI_SQUARE) return launch_kind<KIND, EPI_SQUARE, 2, BN>(maps, p, units, s);
  return launch_kind<KIND, EPI_PLAIN, 2, BN>(maps, p, units, s);
}

template <int BN>
cudaError_t launch_bn(int kind, int epi, const KMaps& maps, const KParams& p, int units,
                      cudaStream_t s) {
  if (kind == KIND_FP16X2) return launch_narrow<KIND_FP16X2, BN>(epi, maps, p, units, s);
  if (kind == KIND_BF16X3) return launch_narrow<KIND_BF16X3, BN>(epi, maps, p, units, s);
  return launch_narrow<KIND_BF16X2, BN>(epi, maps, p, units, s);
}

// the block-sparse square: one launch over every resident pair, the tile count
// read on the device
cudaError_t launch_sparse(int kind, const KMaps& maps, const KParams& p, int units, cudaStream_t s) {
  if (kind == KIND_FP16X2) return launch_kind<KIND_FP16X2, EPI_SQUARE, 2, BN_FULL, true>(maps, p, units, s);
  if (kind == KIND_BF16X3) return launch_kind<KIND_BF16X3, EPI_SQUARE, 2, BN_FULL, true>(maps, p, units, s);
  return launch_kind<KIND_BF16X2, EPI_SQUARE, 2, BN_FULL, true>(maps, p, units, s);
}

template <int CG>
cudaError_t launch_cg(int kind, int epi, const KMaps& maps, const KParams& p, int units,
                      cudaStream_t s) {
  if (kind == KIND_FP16X2) return launch_epi<KIND_FP16X2, CG>(epi, maps, p, units, s);
  if (kind == KIND_BF16X3) return launch_epi<KIND_BF16X3, CG>(epi, maps, p, units, s);
  return launch_epi<KIND_BF16X2, CG>(epi, maps, p, units, s);
}

}  // namespace

void tc_tile_shape(int pair, int* bm, int* bn) {
  *bm = pair ? 2 * BM : BM;
  *bn = BN_FULL;
}

// Upper tiles (first row at most the last column) or all tiles of a rows x np product.
static int64_t tile_count(int64_t rows, int64_t np, int bn, bool upper) {
  if (!upper) return rows / (2 * BM) * (np / bn);
  int64_t n = 0;
  for (int64_t r0 = 0; r0 < np; r0 += 2 * BM) n += (np - r0) / bn;
  return n;
}

// By an estimate that only has to order the widths, for the three segments of two planes
// (more or fewer segments scale all widths alike but for the tile's end): 600, 400 or 320
// clocks a k-block of 256, 128 or 64 columns, 140 clocks a column for a square's end with
// its sums and mirror and 30 for a plain one, waves of 76 pairs. Narrower only when 5 %
// better. (The square at N = 2048, 72 tiles of 128 columns: 56000 clocks; 36 us by ncu.)
int tc_tile_width(int64_t rows, int64_t np, bool upper) {
  constexpr int kPairs = 76;
  const double kb = (double)(np / BK);
  int best = BN_FULL;
  double tbest = 0.0;
  for (int bn = BN_FULL; bn >= 64; bn /= 2) {
    const int64_t waves = (tile_count(rows, np, bn, upper) + kPairs - 1) / kPairs;
    const double kclk = bn == 256 ? 600.0 : (bn == 128 ? 400.0 : 320.0);
    const double end = (upper ? 140.0 : 30.0) * bn;
    const double t = (double)waves * 3.0 * kb * kclk + end;
    if (tbest == 0.0 || t < 0.95 * tbest) {
      tbest = t;
      best = bn;
    }
  }
  return best;
}

cudaError_t launch_gemm_tc(const TcLaunch& L, cudaStream_t s, char* errbuf, size_t errlen) {
  if (L.ntiles <= 0) return cudaSuccess;
  const int mode = L.mode;
  const int kind = mode == SP2_MODE_FP16X2 ? KIND_FP16X2
                                           : (mode == SP2_MODE_BF16X3 ? KIND_BF16X3 : KIND_BF16X2);
  const bool f16 = kind == KIND_FP16X2, x3 = kind == KIND_BF16X3;
  const int cg = L.tune.pair ? 2 : 1;   // the tile list was built for this tile shape
  const TcOperand& P = L.P;
  const TcOperand& Q = L.Q;
  // the middle planes exist only in BF16X3; elsewhere the hi maps stand in (never read)
  const uint16_t* p_mid = x3 ? P.mid : P.hi;
  const uint16_t* q_mid = x3 ? Q.mid : Q.hi;
  const bool sym_out = L.epi != EPI_PLAIN;
  if (x3 && (!p_mid || !q_mid || (sym_out && !L.out.mid))) {
    snprintf(errbuf, errlen, "tcgen05 product: BF16X3 operand without its middle plane");
    return cudaErrorInvalidValue;
  }
  if (sym_out && !L.prev) {
    snprintf(errbuf, errlen, "tcgen05 product: symmetric epilogue without the previous iterate");
    return cudaErrorInvalidValue;
  }
  // TMA box/stride rules: 16-byte aligned bases, np*2-byte row pitch (np % 256 == 0),
  // every x coordinate a multiple of 64 elements; tiles never leave their operand.
  const int64_t np = L.np;
  if ((reinterpret_cast<uintptr_t>(P.hi) | reinterpret_cast<uintptr_t>(P.lo) |
       reinterpret_cast<uintptr_t>(Q.hi) | reinterpret_cast<uintptr_t>(Q.lo) |
       reinterpret_cast<uintptr_t>(p_mid) | reinterpret_cast<uintptr_t>(q_mid)) & 15u ||
      np % 256 != 0 || P.rows % np != 0 || Q.rows % np != 0 || P.rows % (BM * cg) != 0 ||
      Q.rows % L.bn != 0 || (L.bn != BN_FULL && (cg != 2 || L.epi == EPI_SYMM || L.dyn_ntiles)) || (L.epi == EPI_SYMM && Q.rows != np) ||
      (L.epi == EPI_SQUARE && P.rows != np) || P.rows > (int64_t)1 << 30) {
    snprintf(errbuf, errlen, "tcgen05 product: operand alignment/shape violates the TMA rules");
    return cudaErrorInvalidValue;
  }
  KMaps maps;
  MapKey key;
  memset(&key, 0, sizeof key);   // padding bytes too: the key is compared bytewise
  key.planes[0] = P.hi;
  key.planes[1] = P.lo;
  key.planes[2] = p_mid;
  key.planes[3] = Q.hi;
  key.planes[4] = Q.lo;
  key.planes[5] = q_mid;
  key.prows = P.rows;
  key.qrows = Q.rows;
  key.np = np;
  key.cg = cg;
  key.bn = L.bn;
  key.f16 = f16 ? 1 : 0;
  if (!cached_maps(key, &maps)) {
    snprintf(errbuf, errlen, "cuTensorMapEncodeTiled failed (driver entry point unavailable?)");
    return cudaErrorInvalidValue;
  }
  KParams p;
  p.nkb = (int)(np / BK);
  // K chunk drained from TMEM into FP32 registers: 4 k-blocks (256 products per
  // accumulator pass). np is a multiple of 256, so 4 divides every segment and
  // the lo-plane weight changes only at a chunk boundary. The tensor core's
  // FP32 accumulation truncates, and its bias grows with the chunk length: at
  // N=4096 (FP16X2) 256-wide chunks give a 1.0e-5 density error against the
  // exact form, 512-wide 2.5e-5 and 2048-wide 7.6e-4, for 3% more time per
  // product than 512-wide chunks.
  p.ch = 4;
  // The cross terms (hi*lo, lo*hi; in BF16X3 everything after hi*hi) are small
  // once weighted, so the truncation bias of a longer TMEM accumulation shrinks
  // with them: a chunk's bias scales with its length times the size of its
  // terms. Every chunk boundary costs the MMA issuer a commit and a wait, so the
  // cross terms take the longest chunk whose bias stays a few percent of the
  // hi*hi chunks' (256 x 1): FP16X2 (weight 2^-11) up to 16384 wide (256
  // k-blocks, 16384 x 2^-11 = 8), the bfloat16 modes (2^-8) up to 2048 (32
  // k-blocks, also 8); the largest power of two up to that which divides np / BK.
  p.ch_lo = f16 ? 256 : 32;
  while ((np / BK) % p.ch_lo != 0) p.ch_lo >>= 1;
  p.nbase = x3 ? 6 : 3;
  p.nseg = L.epi == EPI_SYMM ? 2 * p.nbase : p.nbase;
  p.np = np;
  p.out = static_cast<float*>(L.out.master);
  p.out_hi = L.out.hi;
  p.out_lo = L.out.lo;
  p.out_mid = L.out.mid;
  p.prev = L.prev;
  p.part = L.part;
  p.tiles = L.tiles;
  p.ntiles = L.ntiles;
  p.st = L.st;
  p.step = L.step;
  p.p_scale = f16 ? L.p_scale : nullptr;
  p.q_scale = f16 ? L.q_scale : nullptr;
  p.o_scale = f16 ? L.o_scale : nullptr;
  p.zmax = f16 ? L.zmax : nullptr;
  p.zero = L.zero;
  p.nzero = L.zero ? L.nzero : 0;
  p.trans = L.trans;
  p.wait_ns = L.tune.wait_ns;
  p.withhold = L.tune.withhold;
  p.tail = L.tail;
  // persistent: one CTA per SM (the shared-memory ring allows no second one)
  p.dyn_ntiles = L.dyn_ntiles;
  p.kcnt = L.kcnt;
  p.klist = L.klist;
  p.nbk = L.nbk;
  if (L.dec) p.dec = *L.dec;
  if (L.dyn_ntiles) {
    if (cg != 2 || L.epi != EPI_SQUARE || L.tail || !L.kcnt || !L.klist || L.nbk * 256 != np) {
      snprintf(errbuf, errlen, "tcgen05 product: block-sparse launches are squares on CTA pairs");
      return cudaErrorInvalidValue;
    }
    return launch_sparse(kind, maps, p, L.ntiles, s);
  }
  // persistent: one CTA (pair) per SM (pair of SMs), the launch's tiles spread over them
  if (L.bn == 128) return launch_bn<128>(kind, L.epi, maps, p, L.ntiles, s);
  if (L.bn == 64) return launch_bn<64>(kind, L.epi, maps, p, L.ntiles, s);
  if (cg == 2) return launch_cg<2>(kind, L.epi, maps, p, L.ntiles, s);
  return launch_cg<1>(kind, L.epi, maps, p, L.ntiles, s);
}

}  // namespace sp2
