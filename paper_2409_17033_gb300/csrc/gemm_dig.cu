// FP64 products on the 16-bit tensor cores of sm_103a, by error-free splitting
// into digits (the scheme of Ozaki, Ogita, Oishi and Rump, "Error-free
// transformations of matrix multiplication by using fast routines of matrix
// multiplication and its applications", Numer. Algorithms 59, 2012).
//
// Why: GB300's FP64 pipe does about 2 FMA per clock and SM (1.25 TFLOP/s), its
// 16-bit tensor pipe a thousand times that, so 36 tensor products in place of one
// FP64 product are still some 30 times faster once a product fills the GPU.
//
// Splitting. Row i of a factor is scaled by a power of two 2^ex_i > its 2-norm and
// rounded to a 63-bit fixed-point number, which is cut into 8 signed digits of 8
// bits: x = 2^(ex - 63) sum_i d_i 2^(56 - 8 i), d_i in [-128, 128]. Digits are exact
// in bfloat16, a product of two is at most 2^14, and a sum of 256 of them at most
// 2^22, so the tensor core's FP32 accumulation of a 256-wide K chunk is exact
// whatever the inputs, and one FP32 addition of 1.5 2^23 turns it into an integer's
// bits. The chunks of all digit pairs (i, j) of one weight s = i + j add up in INT32
// registers (exact to K = 8192) and are stored, one 32-bit plane per weight (and per
// part of a longer or divided K axis). The passes below add a product's planes into a
// 64-bit integer T(i, j) of unit 2^(ex_i + ex_j - 62): |C_ij| <= 2^(ex_i + ex_j) by
// Cauchy-Schwarz, so T never leaves 63 bits. The 36 pairs with s <= 7 are formed. What
// is dropped (s >= 8) and rounded is of the order sqrt(K) 2^-64 of the two rows'
// scales, below the rounding of an FP64 dot product. A tile's work may be cut into
// parts, by weight and along K: integer additions commute, so the result has the same
// bits for every cut. (Sums that met in T by 64-bit atomics cost 25000 clocks per
// weight and tile, a third of a product's time at N = 1024.)
//
// (7 digits of 9 bits need 28 products, but their chunks reach 2^24, and the
// conversions to integers (16 a clock and SM) made a chunk's drain as long as its
// MMAs.)
//
// Layout. The planes are stored transposed, G[j * rows + i] for entry (i, j): a warp's
// lanes hold consecutive rows i, so its stores are whole lines.
//
// A step that carries responses forms Y_n X_n and X_n^2 in one launch, X_n stacked below
// the batch Y_n (upper tiles only): its digits are made once, and at small N the square's
// tiles run on CTA pairs that the response's leave idle (SCF of 16 fields at N = 256,
// where the square took 30 us of a step on the CUDA cores: 28.7 -> 21.4 ms).
//
// Per product: k_digits (each factor), k_gemm_dig, then one pass that turns the sums
// into FP64 and applies the recursion's update: k_dig_step, or k_dig_square
// (Eq. DM0, with the traces and the step decision), k_dig_symm (Eqs. DM1-DM3) or
// k_dig_plain.
//
// k_gemm_dig is tensor-bound at large N (36 bfloat16 products) and bound by
// latency and by the number of resident CTA pairs at small N. Tile, pipeline and
// warp roles are those of the split-precision kernel on CTA pairs: 256 x BN tiles
// (BN = 256, or 128 where more and smaller tiles fill the GPU better), one
// tcgen05.mma.cta_group::2 stream per pair, TMA ring, two TMEM chunk buffers
// drained by 16 warps.
#include <math.h>
#include <stdio.h>
#include <string.h>

#include "decide.cuh"
#include "per_device.h"
#include "sp2_internal.h"
#include "tc_ptx.cuh"

namespace sp2 {

namespace {

constexpr int kDigits = kDigPlanes;
constexpr int kGroups = 8;        // digit-pair weights s = i + j <= 7
constexpr int kPairs = kGroups * (kGroups + 1) / 2;
constexpr int kFixBits = 63;      // fixed-point bits of a scaled entry
constexpr int kTBits = 62;        // T's unit is 2^(ex_i + ex_j - kTBits)
constexpr int kBadRow = 1 << 20;  // exponent of a row with a NaN or an infinity

constexpr int BM = 128;           // tile rows per CTA
constexpr int BK = kBoxCols;
constexpr int KCH = 4;            // k-blocks per TMEM chunk: 256 products, exact in FP32
constexpr int KSEG_MAX = 128;     // k-blocks an INT32 sum of 8 digit pairs may span (K = 8192)
constexpr int EPI_WARPS = 16;
constexpr int NUM_THREADS = 64 + 32 * EPI_WARPS;
constexpr unsigned long long DRAIN_NS = 200000000ull;

template <int BN>
struct Geo {
  static constexpr int A_BYTES = BM * BK * 2;
  static constexpr int B_ROWS = BN / 2;
  static constexpr int STAGE_BYTES = A_BYTES + B_ROWS * BK * 2;
  static constexpr int STAGES = BN == 256 ? 6 : 8;
  static constexpr int SMEM_BYTES = STAGES * STAGE_BYTES + 1024 /*align slack*/ + 256 /*barriers*/;
  static constexpr uint32_t TMEM_COLS = 2 * BN;
  static constexpr int TCOLS = BN / (EPI_WARPS / 4);
  // kind::f16: D = F32, A and B bfloat16, K-major, M = 256 over the pair, N = BN
  static constexpr uint32_t IDESC = (1u << 4) | (1u << 7) | (1u << 10) |
                                    ((uint32_t)(BN >> 3) << 17) | ((uint32_t)(2 * BM >> 4) << 24);
};

// The weights of part `part` of `parts`: 36 digit pairs split evenly (weight s has s + 1).
__device__ __forceinline__ uint32_t part_mask(int parts, int part) {
  if (parts == 1) return 0xffu;
  if (parts == 2) return part == 0 ? 0xc4u : 0x3bu;                  // {7,6,2}, {5,4,3,1,0}
  return part == 0 ? 0x81u : (part == 1 ? 0x42u : (part == 2 ? 0x24u : 0x18u));   // {7,0} ..
}

struct DParams {
  int nkb;             // k-blocks of the K axis (np / 64)
  int kseg;            // k-blocks of one K part (a multiple of KCH, at most KSEG_MAX)
  int ksplit;          // K parts
  int parts;           // weight parts (1, 2 or 4)
  int64_t rows;        // rows of A (plane stride of its map, leading dimension of G)
  int64_t np;
  int64_t xrows;       // rows of X's map per plane, and the first of X's own
  int xoff;
  int* G;              // planes (K part x weight) of np x rows sums
  const Tile* tiles;
  int nunits;          // tiles x parts x ksplit
  DevState* st;
  int step;
  unsigned long long wait_ns;
  int withhold;
};

struct Unit {
  Tile t;
  uint32_t mask;
  int ks, kb0, kb1;
};

__device__ __forceinline__ Unit unit_of(const DParams& p, int u) {
  const int per = p.parts * p.ksplit;
  const int tix = u / per, rem = u - tix * per;
  const int part = rem / p.ksplit, ks = rem - part * p.ksplit;
  Unit r;
  r.t = p.tiles[tix];
  r.mask = part_mask(p.parts, part);
  r.ks = ks;
  r.kb0 = ks * p.kseg;
  r.kb1 = r.kb0 + p.kseg < p.nkb ? r.kb0 + p.kseg : p.nkb;
  return r;
}

template <int BN>
__global__ void __launch_bounds__(NUM_THREADS, 1)
k_gemm_dig(const __grid_constant__ CUtensorMap amap, const __grid_constant__ CUtensorMap bmap,
           const __grid_constant__ DParams p) {
  using G = Geo<BN>;
  constexpr int STAGES = G::STAGES;
  DevState* st = p.st;
  extern __shared__ uint8_t smem_raw[];
  uint8_t* smem = reinterpret_cast<uint8_t*>((reinterpret_cast<uintptr_t>(smem_raw) + 1023) &
                                             ~(uintptr_t)1023);
  uint64_t* full = reinterpret_cast<uint64_t*>(smem + STAGES * G::STAGE_BYTES);
  uint64_t* empty = full + STAGES;
  uint64_t* pfull = empty + STAGES;   // rank 0: the peer's stage has landed
  uint64_t* tfull = pfull + STAGES;   // [2] chunk accumulated in TMEM buffer b
  uint64_t* tempty = tfull + 2;       // [2] TMEM buffer b drained by both CTAs
  uint64_t* mdone = tempty + 2;
  uint32_t* tmem_slot = reinterpret_cast<uint32_t*>(mdone + 1);

  const int warp = __shfl_sync(0xffffffffu, (int)(threadIdx.x >> 5), 0), lane = threadIdx.x & 31;
  int* abortf = &st->abort_flag;
  const uint32_t rank = cluster_rank();
  const bool issuer = rank == 0;
  const int pair = (int)(blockIdx.x >> 1), npairs = (int)(gridDim.x >> 1);
  const int pairs_per_part = kPairs / p.parts;   // digit pairs of a unit

  if (threadIdx.x == 0) {
    for (int s = 0; s < STAGES; ++s) {
      mbar_init(&full[s], 1);
      mbar_init(&empty[s], 1);
      mbar_init(&pfull[s], 1);
    }
    for (int b = 0; b < 2; ++b) {
      mbar_init(&tfull[b], 1);
      mbar_init(&tempty[b], 2 * EPI_WARPS);
    }
    mbar_init(mdone, 1);
    asm volatile("fence.mbarrier_init.release.cluster;" ::: "memory");
    asm volatile("prefetch.tensormap [%0];" ::"l"(reinterpret_cast<uint64_t>(&amap)) : "memory");
    asm volatile("prefetch.tensormap [%0];" ::"l"(reinterpret_cast<uint64_t>(&bmap)) : "memory");
  }
  if (warp == 1) {
    asm volatile("tcgen05.alloc.cta_group::2.sync.aligned.shared::cta.b32 [%0], %1;" ::"r"(
                     smem_u32(tmem_slot)),
                 "r"(G::TMEM_COLS)
                 : "memory");
    asm volatile("tcgen05.relinquish_alloc_permit.cta_group::2.sync.aligned;" ::: "memory");
  }
  tc_fence_before();
  __syncthreads();
  cluster_sync();
  tc_fence_after();
  const uint32_t tmem = *tmem_slot;

  // nothing of the launches before is read up to here; a halted launch runs no unit
  // (stop_at is fixed for the launch, so a pair agrees)
  dep_sync();
  const int stopped = *((volatile const int*)&st->stop_at);
  const int nunits = stopped != 0 && p.step > stopped ? 0 : p.nunits;

  if (warp == 0) {
    // copy issuer: the whole warp (the waits by every lane, the copies by an elected one)
    int64_t g = 0;
    RingPos<STAGES> rp;
    const uint32_t ring = smem_u32(smem);
    bool ok = true;
    for (int u = pair; u < nunits && ok; u += npairs) {
      const Unit w = unit_of(p, u);
      const int arow = w.t.row0 + (int)rank * BM;
      const int brow = w.t.col0 + (int)rank * G::B_ROWS;
      for (int s = kGroups - 1; s >= 0 && ok; --s) {
        if (!((w.mask >> s) & 1u)) continue;
        for (int i = 0; i <= s && ok; ++i) {
          const int ay = i * (int)p.rows + arow, by = (s - i) * (int)p.xrows + p.xoff + brow;
          for (int kx = w.kb0 * BK; kx < w.kb1 * BK; kx += BK, ++g, rp.next()) {
            ok = __all_sync(0xffffffffu, mbar_wait<true>(&empty[rp.s], rp.ph ^ 1u, abortf, p.wait_ns));
            if (!ok) break;
            if (p.withhold && blockIdx.x == 0 && g == 0) continue;  // test hook: never completes
            const uint32_t sa = ring + (uint32_t)(rp.s * G::STAGE_BYTES);
            tma_load_stage(&full[rp.s], G::STAGE_BYTES, &amap, &bmap, sa, sa + G::A_BYTES, kx, ay, by);
          }
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
  } else if (warp == 1) {
    if (!issuer) {
      if (lane == 0) {
        // rank 1: pass each landed stage on to rank 0's MMA issuer
        const uint32_t pfull_peer = cluster_addr(smem_u32(pfull), 0);
        RingPos<STAGES> rp;
        bool ok = true;
        for (int u = pair; u < nunits && ok; u += npairs) {
          const Unit w = unit_of(p, u);
          const int n = pairs_per_part * (w.kb1 - w.kb0);
          for (int q = 0; q < n; ++q, rp.next()) {
            if (!mbar_wait<true>(&full[rp.s], rp.ph, abortf, p.wait_ns)) {
              ok = false;
              break;
            }
            mbar_arrive_cluster_release(pfull_peer + (uint32_t)(rp.s * sizeof(uint64_t)));
          }
        }
      }
    } else {
      // whole warp (the waits by every lane, the instructions by an elected one)
      bool ok = true;
      uint32_t gc = 0;
      RingPos<STAGES> rp;
      const uint64_t adesc0 = sdesc_sw128(smem_u32(smem));
      for (int u = pair; u < nunits && ok; u += npairs) {
        const Unit w = unit_of(p, u);
        const int nch = pairs_per_part * ((w.kb1 - w.kb0) / KCH);
        for (int c = 0; c < nch && ok; ++c, ++gc) {
          const uint32_t b = gc & 1u;
          ok = __all_sync(0xffffffffu, mbar_wait<true>(&tempty[b], ((gc >> 1) & 1u) ^ 1u, abortf,
                                                      p.wait_ns));
          if (!ok) break;
          tc_fence_after();
          const uint32_t dtm = tmem + b * BN;
#pragma unroll 1
          for (int kb = 0; kb < KCH; ++kb, rp.next()) {
            ok = __all_sync(0xffffffffu, mbar_wait<false>(&full[rp.s], rp.ph, abortf, p.wait_ns) &&
                                             mbar_wait<true>(&pfull[rp.s], rp.ph, abortf, p.wait_ns));
            if (!ok) break;
            tc_fence_after();
            const uint64_t adesc = adesc0 + (uint64_t)(rp.s * (G::STAGE_BYTES >> 4));
            const uint64_t bdesc = adesc + (uint64_t)(G::A_BYTES >> 4);
            umma_kblock<2>(dtm, adesc, bdesc, G::IDESC, kb > 0 ? 1u : 0u);
            umma_commit_both(&empty[rp.s]);
          }
          if (ok) umma_commit_both(&tfull[b]);
        }
      }
      if (!ok) {
        umma_commit<2>(mdone);
        mbar_wait_drain(mdone, 0, DRAIN_NS);
      }
    }
  } else {
    // warp w reads TMEM lanes 32 (w % 4) .. +31 and the columns of group (w - 2) / 4
    constexpr int TC = G::TCOLS;
    const int q = warp & 3;
    const int grp = (warp - 2) >> 2;
    const int r = (int)rank * BM + q * 32 + lane;
    const uint32_t trow = tmem + ((uint32_t)(q * 32) << 16) + (uint32_t)(grp * TC);
    const uint32_t tempty_peer = !issuer ? cluster_addr(smem_u32(tempty), 0) : 0u;
    bool ok = true;
    uint32_t gc = 0;   // chunk counter: buffer gc & 1, phase (gc >> 1) & 1
    for (int u = pair; u < nunits && ok; u += npairs) {
      uint32_t mask;
      int kch;
      int* dst;
      {
        const Unit w = unit_of(p, u);
        mask = w.mask;
        kch = (w.kb1 - w.kb0) / KCH;
        dst = p.G + ((int64_t)w.ks * kGroups * p.np + w.t.col0 + grp * TC) * p.rows +
              (int64_t)w.t.row0 + r;
      }
#pragma unroll 1
      for (int s = kGroups - 1; s >= 0; --s) {
        if (!((mask >> s) & 1u)) continue;
        // sums of the chunks' bits after the addition of 1.5 2^23, modulo 2^32
        const int nch = (s + 1) * kch;
        uint32_t acc[TC];
#pragma unroll
        for (int j = 0; j < TC; ++j) acc[j] = 0u;
#pragma unroll 1
        for (int c = nch; c > 0; --c, ++gc) {
          const uint32_t b = gc & 1u;
          const bool wt = mbar_wait<true>(&tfull[b], (gc >> 1) & 1u, abortf, p.wait_ns);
          ok = __all_sync(0xffffffffu, wt);
          if (!ok) break;
          tc_fence_after();
#pragma unroll
          for (int c0 = 0; c0 < TC; c0 += 16) {
            uint32_t v[16];
            tmem_ld16(trow + b * BN + (uint32_t)c0, v);
#pragma unroll
            for (int j = 0; j < 16; ++j)
              acc[c0 + j] += __float_as_uint(__uint_as_float(v[j]) + 12582912.0f);
          }
          tc_fence_before();
          __syncwarp();
          if (lane == 0) {
            if (!issuer)
              mbar_arrive_cluster(tempty_peer + b * (uint32_t)sizeof(uint64_t));
            else
              mbar_arrive(&tempty[b]);
          }
        }
        if (!ok) break;
        const uint32_t off = (uint32_t)nch * 0x4b400000u;   // the bits of 1.5 2^23
        int* d = dst + (int64_t)s * p.np * p.rows;
#pragma unroll
        for (int j = 0; j < TC; ++j) {
          __stcg(d, (int)(acc[j] - off));
          d += p.rows;
        }
      }
    }
  }

  tc_fence_before();
  __syncthreads();
  cluster_sync();
  if (warp == 1) {
    __syncwarp();
    tc_fence_after();
    asm volatile("tcgen05.dealloc.cta_group::2.sync.aligned.b32 %0, %1;" ::"r"(tmem),
                 "r"(G::TMEM_COLS)
                 : "memory");
  }
}

__device__ __forceinline__ bool halted_dig(const DevState* st, int step) {
  const int m = *((volatile const int*)&st->stop_at);
  return m != 0 && step > m;
}

// ------------------------------------------------------------ digits
// One block per row (of two stacked matrices): the row's power-of-two scale 2^ex >= its 2-norm, then the
// eight digit planes (plane d of the stack at d * rows * np). Integer arithmetic
// throughout (FP64 conversions run at the slow FP64 rate); the norm in FP32 from the entries' leading 20 bits, relative to the
// row's largest entry, with a margin above its rounding. HBM-bound at large N: 8
// bytes read, 16 written per entry.
constexpr int kDigThreads = 128;

template <bool TWO>   // (the choice of the source costs a single matrix's pass registers and time)
__global__ void __launch_bounds__(kDigThreads)
k_digits(const double* __restrict__ src, int64_t rows1, const double* __restrict__ src2,
         int64_t rows, int64_t np, uint16_t* __restrict__ dig, int* __restrict__ ex,
         const DevState* st, int step) {
  dep_sync();
  if (halted_dig(st, step)) return;
  __shared__ uint32_t smax[kDigThreads / 32];
  __shared__ float ssum[kDigThreads / 32];
  const int64_t row = blockIdx.x;
  const double2* x2 = reinterpret_cast<const double2*>(
      !TWO || row < rows1 ? src + row * np : src2 + (row - rows1) * np);
  const int n4 = (int)(np / 4);
  const int lane = threadIdx.x & 31, warp = threadIdx.x >> 5;
  uint32_t m = 0;
  for (int c = threadIdx.x; c < n4; c += kDigThreads) {
    const double2 a = x2[2 * c], b = x2[2 * c + 1];
    m = max(m, max(max((uint32_t)__double2hiint(a.x) & 0x7fffffffu,
                       (uint32_t)__double2hiint(a.y) & 0x7fffffffu),
                   max((uint32_t)__double2hiint(b.x) & 0x7fffffffu,
                       (uint32_t)__double2hiint(b.y) & 0x7fffffffu)));
  }
  m = __reduce_max_sync(0xffffffffu, m);
  if (lane == 0) smax[warp] = m;
  __syncthreads();
  m = smax[0];
#pragma unroll
  for (int w = 1; w < kDigThreads / 32; ++w) m = max(m, smax[w]);
  const int em = (int)(m >> 20);
  const bool bad = em == 0x7ff;
  float ss = 0.0f;
  for (int c = threadIdx.x; c < n4; c += kDigThreads) {
    const double2 a = x2[2 * c], b = x2[2 * c + 1];
    const double v[4] = {a.x, a.y, b.x, b.y};
#pragma unroll
    for (int k = 0; k < 4; ++k) {
      const uint32_t h = (uint32_t)__double2hiint(v[k]) & 0x7fffffffu;
      const int fe = (int)(h >> 20) - em;   // <= 0
      // |x| / 2^(em - 1023), truncated to 20 bits; below 2^-60 covered by the margin
      const float f = fe > -60 ? __uint_as_float((uint32_t)((127 + fe) << 23) | ((h & 0xfffffu) << 3))
                               : 0.0f;
      ss = fmaf(f, f, ss);
    }
  }
  for (int o = 16; o > 0; o >>= 1) ss += __shfl_xor_sync(0xffffffffu, ss, o);
  if (lane == 0) ssum[warp] = ss;
  __syncthreads();
  ss = 0.0f;
#pragma unroll
  for (int w = 0; w < kDigThreads / 32; ++w) ss += ssum[w];
  // sums of at most 2^14 positive FP32 terms per thread: 1 + 2^-5 covers their
  // rounding and the truncation of the entries, and keeps the fixed-point entries (and
  // the biased ones below) within 63 bits
  ss = ss * (1.0f + 0.03125f) + (float)np * 1e-17f;
  int k2;
  frexpf(ss, &k2);                      // ss < 2^k2
  const int q = (k2 + 1) >> 1;          // sqrt(ss) < 2^q
  const int e = bad ? kBadRow : (m == 0 ? 0 : em - 1023 + q);
  if (threadIdx.x == 0) ex[row] = e;
  const int64_t plane = rows * np;
  constexpr unsigned long long kBias = 0x0080808080808080ull;   // 128 in every digit below the first
  for (int c = threadIdx.x; c < n4; c += kDigThreads) {
    const double2 a = x2[2 * c], b = x2[2 * c + 1];
    const double v[4] = {a.x, a.y, b.x, b.y};
    uint32_t f[4][kDigits];
#pragma unroll
    for (int k = 0; k < 4; ++k) {
      const long long bits = __double_as_longlong(v[k]);
      const int eb = (int)((bits >> 52) & 0x7ff);
      unsigned long long mant = (unsigned long long)bits & 0xfffffffffffffull;
      if (eb) mant |= 1ull << 52;
      const int sh = (eb ? eb : 1) - (1075 - kFixBits) - e;   // at most 11
      long long I;
      if (sh >= 0) I = (long long)(mant << sh);
      else if (sh > -55) I = (long long)((mant + (1ull << (-sh - 1))) >> -sh);
      else I = 0;
      if (bits < 0) I = -I;
      if (bad || m == 0) I = 0;
      const long long B = I + (long long)kBias;
      f[k][0] = (uint32_t)((int)(B >> 56) + 128);
#pragma unroll
      for (int d = 1; d < kDigits; ++d) f[k][d] = (uint32_t)((unsigned long long)B >> (56 - 8 * d)) & 255u;
    }
#pragma unroll
    for (int d = 0; d < kDigits; ++d) {
      uint32_t h[4];
#pragma unroll
      for (int k = 0; k < 4; ++k)   // field - 128 as an FP32 integer; its upper half is the bfloat16
        h[k] = __float_as_uint(__uint_as_float(0x4B000000u + f[k][d]) - 8388736.0f);
      uint2 o;
      o.x = __byte_perm(h[0], h[1], 0x7632);
      o.y = __byte_perm(h[2], h[3], 0x7632);
      reinterpret_cast<uint2*>(dig + d * plane + row * np)[c] = o;
    }
  }
}

// A product's sums: planes of `ksplit` K parts x kGroups weights, `plane` entries each.
struct Sums {
  const int* g;
  int64_t plane;
  int ksplit;
};

// T of four consecutive entries at o: weight s counts 2^(112 - 8 s) over
// 2^(2 kFixBits - kTBits) = 2^64, that is 2^(48 - 8 s), the last one rounded
__device__ __forceinline__ void load_t(const Sums& q, int64_t o, long long (&t)[4]) {
#pragma unroll
  for (int k = 0; k < 4; ++k) t[k] = 0;
  // the last weight's sum over the K parts, x = 256 hi + lo, rounded once
  int hi[4] = {0, 0, 0, 0}, lo[4] = {0, 0, 0, 0};
  for (int ks = 0; ks < q.ksplit; ++ks) {
    int4 v[kGroups];
#pragma unroll
    for (int s = 0; s < kGroups; ++s)
      v[s] = __ldcs(reinterpret_cast<const int4*>(q.g + (int64_t)(ks * kGroups + s) * q.plane + o));
#pragma unroll
    for (int s = 0; s < kGroups; ++s) {
      const int x[4] = {v[s].x, v[s].y, v[s].z, v[s].w};
      const int sh = 2 * 56 - 8 * s - (2 * kFixBits - kTBits);
#pragma unroll
      for (int k = 0; k < 4; ++k) {
        if (sh >= 0) t[k] += (long long)x[k] << (sh > 0 ? sh : 0);
        else hi[k] += x[k] >> 8, lo[k] += x[k] & 255;
      }
    }
  }
#pragma unroll
  for (int k = 0; k < 4; ++k) t[k] += hi[k] + ((lo[k] + (1 << 7)) >> 8);
}

// T's value as FP64 (one rounding), times 2^e. The conversion by magic constants
// (two FP64 additions) and the scaling by the exponent field keep to FP32-rate
// integer work otherwise.
__device__ __forceinline__ double from_fixed(long long t, int ei, int ej) {
  const int hi = (int)(t >> 32);
  const uint32_t lo = (uint32_t)t;
  // 2^84 + 2^63 + hi 2^32, 2^52 + lo
  const double dh = __hiloint2double(0x45300000, (int)((uint32_t)hi ^ 0x80000000u));
  const double dl = __hiloint2double(0x43300000, (int)lo);
  const double off = __hiloint2double(0x45300000, (int)0x80100000u);   // 2^84 + 2^63 + 2^52
  const double v = (dh - off) + dl;
  if (ei == kBadRow || ej == kBadRow) return __longlong_as_double(0x7ff8000000000000ll);
  const int e = ei + ej - kTBits;
  const int vh = __double2hiint(v);
  const int ve = (vh >> 20) & 0x7ff;
  if (ve == 0) return v;   // zero
  const int ne = ve + e;
  if (ne > 0 && ne < 0x7ff) return __hiloint2double(vh + e * (1 << 20), __double2loint(v));
  return scalbn(v, e);
}

constexpr int TE = 32;            // tile edge of the passes over T
constexpr int kPassThreads = 256;

__device__ __forceinline__ void tri_ij(int64_t t, int64_t& I, int64_t& J) {
  J = (int64_t)((sqrtf(8.0f * (float)t + 1.0f) - 1.0f) * 0.5f);
  while (J * (J + 1) / 2 > t) --J;
  while ((J + 1) * (J + 2) / 2 <= t) ++J;
  I = t - J * (J + 1) / 2;
}

__device__ __forceinline__ void ld4d(const double* p, double (&v)[4]) {
  const double2 a = reinterpret_cast<const double2*>(p)[0];
  const double2 b = reinterpret_cast<const double2*>(p)[1];
  v[0] = a.x, v[1] = a.y, v[2] = b.x, v[3] = b.y;
}
__device__ __forceinline__ void st4d(double* p, const double (&v)[4]) {
  reinterpret_cast<double2*>(p)[0] = make_double2(v[0], v[1]);
  reinterpret_cast<double2*>(p)[1] = make_double2(v[2], v[3]);
}

// X_{n+1} = sigma > 0 ? C : 2 X_n - C from T (C = X_n^2, upper entries), mirrored;
// partials of Tr, ||.||_F^2 and ||X_n - X_n^2||_F^2 in FP64, and the step decision
// in the last block. G has leading dimension ld. Blocks walk pairs of TE x TE tiles (I <= J); T's tile (J, I)
// holds entries (i, j) of the upper tile with i along its rows. Bound by its 6 FP64
// operations per upper entry (an FP64 instruction of a warp takes 64 clocks), so
// the reductions come once per block, not per tile, ||.||_F^2 and f sharing them.
struct SquareArgs {
  Sums q;
  int64_t ld;
  const int* ex;
  const double* X;
  double* out;
  int ntiles, nblocks;
  Part3* part;
  SimtDecide dec;
};
using PassTile = double[2][TE][TE + 1];

__device__ __forceinline__ void square_pass(const SquareArgs& a, int block, int64_t np, DevState* st,
                                            int step, PassTile& sm) {
  const Sums& q = a.q;
  const int64_t ld = a.ld;
  const int* __restrict__ ex = a.ex;
  const double* __restrict__ X = a.X;
  double* __restrict__ out = a.out;
  __shared__ double red[3][kPassThreads / 32];
  const int r = threadIdx.x >> 3, c4 = (threadIdx.x & 7) * 4;
  const int lane = threadIdx.x & 31, warp = threadIdx.x >> 5;
  const int sg = st->sigma[step];
  double t1 = 0.0, t2 = 0.0, f = 0.0;   // t2, f: off-diagonal entries (counted twice below)
  double e2 = 0.0, ef = 0.0;            // their diagonal entries
  int buf = 0;
  for (int64_t tix = block; tix < a.ntiles; tix += a.nblocks, buf ^= 1) {
    int64_t I, J;
    tri_ij(tix, I, J);
    const int64_t gj = J * TE + r, gi0 = I * TE + c4;
    double y[4];
    {
      long long t[4];
      double x[4];
      load_t(q, gj * ld + gi0, t);
      ld4d(X + gj * np + gi0, x);   // X_n is symmetric
      const int ej = ex[gj];
#pragma unroll
      for (int k = 0; k < 4; ++k) {
        const int64_t gi = gi0 + k;
        if (gi > gj) continue;      // below the diagonal of a diagonal tile
        const double c = from_fixed(t[k], ex[gi], ej);
        const double v = sg > 0 ? c : 2.0 * x[k] - c;
        const double d = x[k] - c;
        y[k] = v;
        sm[buf][r][c4 + k] = v;
        if (gi == gj) {
          t1 += v;
          e2 += v * v;
          ef += d * d;
        } else {
          t2 += v * v;
          f += d * d;
        }
      }
    }
    __syncthreads();   // (the other buffer's readers are two tiles back)
    if (I == J) {
#pragma unroll
      for (int k = 0; k < 4; ++k)
        if (gi0 + k > gj) y[k] = sm[buf][c4 + k][r];
      st4d(out + gj * np + gi0, y);
    } else {
      st4d(out + gj * np + gi0, y);
      double w[4];
#pragma unroll
      for (int k = 0; k < 4; ++k) w[k] = sm[buf][c4 + k][r];   // entry (i, j), i = I TE + r
      st4d(out + (I * TE + r) * np + J * TE + c4, w);
    }
  }
  t2 = 2.0 * t2 + e2;
  f = 2.0 * f + ef;
  const bool up = lane >= 16;
  double s = (up ? f : t2) + __shfl_xor_sync(0xffffffffu, up ? t2 : f, 16);
  for (int o = 8; o > 0; o >>= 1) s += __shfl_xor_sync(0xffffffffu, s, o);
  for (int o = 16; o > 0; o >>= 1) t1 += __shfl_xor_sync(0xffffffffu, t1, o);
  if (lane == 0) red[0][warp] = t1, red[1][warp] = s;
  if (lane == 16) red[2][warp] = s;
  __syncthreads();
  if (warp == 0) {
    constexpr int NW = kPassThreads / 32;
    double v = lane < 3 * NW ? red[lane / NW][lane % NW] : 0.0;
    for (int o = NW / 2; o > 0; o >>= 1) v += __shfl_xor_sync(0xffffffffu, v, o);
    const double a2 = __shfl_sync(0xffffffffu, v, NW), af = __shfl_sync(0xffffffffu, v, 2 * NW);
    if (lane == 0) a.part[block] = Part3{v, a2, af};
  }
  if (a.dec.done) last_block_decides(a.part, a.dec, (unsigned)a.nblocks);
}

__global__ void __launch_bounds__(kPassThreads)
k_dig_square(const __grid_constant__ SquareArgs a, int64_t np, DevState* st, int step) {
  dep_sync();
  if (halted_dig(st, step)) return;
  __shared__ PassTile sm;
  square_pass(a, (int)blockIdx.x, np, st, step, sm);
}

// Y_{n+1} = sigma > 0 ? Z + Z^T : 2 Y_n - (Z + Z^T) for a batch, Z = Y_n X_n from T
// (ey: exponents of the stacked rows of Y_n, ex: of X_n; rows: G's leading dimension).
// One block per tile pair
// and batch entry.
struct SymmArgs {
  Sums q;
  int64_t rows;
  const int *ey, *ex;
  const double* yin;
  double* yout;
};

__device__ __forceinline__ void symm_pass(const SymmArgs& a, int64_t tile, int64_t entry, int64_t np,
                                          const DevState* st, int step, PassTile& sm) {
  const Sums& q = a.q;
  const int64_t rows = a.rows;
  const int *__restrict__ ey = a.ey, *__restrict__ ex = a.ex;
  const double* __restrict__ yin = a.yin;
  double* __restrict__ yout = a.yout;
  double(&za)[TE][TE + 1] = sm[0];
  double(&zb)[TE][TE + 1] = sm[1];
  int64_t I, J;
  tri_ij(tile, I, J);
  const int64_t b0 = entry * np, base = b0 * np;
  const int r = threadIdx.x >> 3, c4 = (threadIdx.x & 7) * 4;
  const int sg = st->sigma[step];
  {
    long long ta[4], tb[4];
    const int64_t gj = J * TE + r, gi = I * TE + r;
    load_t(q, gj * rows + b0 + I * TE + c4, ta);   // z(i, j): j = gj, i along c4
    load_t(q, gi * rows + b0 + J * TE + c4, tb);   // z(j, i): i = gi, j along c4
    const int xj = ex[gj], xi = ex[gi];
#pragma unroll
    for (int k = 0; k < 4; ++k) {
      za[r][c4 + k] = from_fixed(ta[k], ey[b0 + I * TE + c4 + k], xj);
      zb[r][c4 + k] = from_fixed(tb[k], ey[b0 + J * TE + c4 + k], xi);
    }
  }
  __syncthreads();
  const int64_t idx = base + (I * TE + r) * np + J * TE + c4;   // entries (I TE + r, J TE + c4 ..)
  double y[4], yo[4];
  if (sg < 0) ld4d(yin + idx, yo);
#pragma unroll
  for (int k = 0; k < 4; ++k) {
    const double sum = za[c4 + k][r] + zb[r][c4 + k];
    y[k] = sg > 0 ? sum : 2.0 * yo[k] - sum;
  }
  st4d(yout + idx, y);
  if (I == J) return;
#pragma unroll
  for (int k = 0; k < 4; ++k) zb[r][c4 + k] = y[k];   // only this thread reads zb[r][c4..] above
  __syncthreads();
  double w[4];
#pragma unroll
  for (int k = 0; k < 4; ++k) w[k] = zb[c4 + k][r];
  st4d(yout + base + (J * TE + r) * np + I * TE + c4, w);
}

__global__ void __launch_bounds__(kPassThreads)
k_dig_symm(const __grid_constant__ SymmArgs a, int64_t np, const DevState* st, int step) {
  dep_sync();
  if (halted_dig(st, step)) return;
  __shared__ PassTile sm;
  symm_pass(a, blockIdx.x, blockIdx.y, np, st, step, sm);
}

// Both of a step whose products ran together. The square's blocks come first: they end in
// the decision, a chain of latencies that the response's blocks cover (SCF of 16 fields at
// N = 256, whose square has 36 blocks: 21.4 -> 19.0 ms).
__global__ void __launch_bounds__(kPassThreads)
k_dig_step(const __grid_constant__ SquareArgs a, const __grid_constant__ SymmArgs y, int tiles,
           int64_t np, DevState* st, int step) {
  dep_sync();
  if (halted_dig(st, step)) return;
  __shared__ PassTile sm;
  const int b = (int)blockIdx.x - a.nblocks;
  if (b < 0) square_pass(a, (int)blockIdx.x, np, st, step, sm);
  else symm_pass(y, b % tiles, b / tiles, np, st, step, sm);
}

// C = T's value, row-major rows x np
__global__ void __launch_bounds__(kPassThreads)
k_dig_plain(const Sums q, int64_t rows, const int* __restrict__ ea,
            const int* __restrict__ ex, double* __restrict__ out, int64_t np, const DevState* st,
            int step) {
  dep_sync();
  if (halted_dig(st, step)) return;
  __shared__ double sm[TE][TE + 1];
  const int64_t i0 = (int64_t)blockIdx.y * TE, j0 = (int64_t)blockIdx.x * TE;
  const int r = threadIdx.x >> 3, c4 = (threadIdx.x & 7) * 4;
  long long t[4];
  load_t(q, (j0 + r) * rows + i0 + c4, t);
  const int xj = ex[j0 + r];
#pragma unroll
  for (int k = 0; k < 4; ++k) sm[r][c4 + k] = from_fixed(t[k], ea[i0 + c4 + k], xj);
  __syncthreads();
  double w[4];
#pragma unroll
  for (int k = 0; k < 4; ++k) w[k] = sm[c4 + k][r];
  st4d(out + (i0 + r) * np + j0 + c4, w);
}

// CTA pairs of k_gemm_dig<BN> resident at a time on the current device, whose
// shared-memory limit for the kernel is set with it.
template <int BN>
cudaError_t resident_pairs(int* n) {
  static PerDevice kept;
  int dev = 0;
  cudaError_t e = cudaGetDevice(&dev);
  if (e != cudaSuccess) return e;
  return kept.get(dev, cudaErrorInvalidDevice, n, [&](int* pairs) {
    auto kern = k_gemm_dig<BN>;
    int nsm = 0;
    cudaError_t r = cudaFuncSetAttribute(kern, cudaFuncAttributeMaxDynamicSharedMemorySize,
                                         Geo<BN>::SMEM_BYTES);
    if (r == cudaSuccess) r = cudaDeviceGetAttribute(&nsm, cudaDevAttrMultiProcessorCount, dev);
    if (r != cudaSuccess) return r;
    cudaLaunchConfig_t cfg = {};
    cudaLaunchAttribute at[1];
    at[0].id = cudaLaunchAttributeClusterDimension;
    at[0].val.clusterDim.x = 2;
    at[0].val.clusterDim.y = 1;
    at[0].val.clusterDim.z = 1;
    cfg.gridDim = dim3((unsigned)(2 * (nsm / 2)));
    cfg.blockDim = dim3(NUM_THREADS);
    cfg.dynamicSmemBytes = Geo<BN>::SMEM_BYTES;
    cfg.attrs = at;
    cfg.numAttrs = 1;
    r = cudaOccupancyMaxActiveClusters(pairs, kern, &cfg);
    return r == cudaSuccess && *pairs < 1 ? cudaErrorNotSupported : r;
  });
}

template <int BN>
cudaError_t launch_bn(const CUtensorMap& am, const CUtensorMap& bm, const DParams& p,
                      cudaStream_t s) {
  int res = 0;
  const cudaError_t e = resident_pairs<BN>(&res);
  if (e != cudaSuccess) return e;
  cudaLaunchConfig_t cfg = {};
  cudaLaunchAttribute at[2];
  at[1].id = cudaLaunchAttributeProgrammaticStreamSerialization;
  at[1].val.programmaticStreamSerializationAllowed = 1;
  at[0].id = cudaLaunchAttributeClusterDimension;
  at[0].val.clusterDim.x = 2;
  at[0].val.clusterDim.y = 1;
  at[0].val.clusterDim.z = 1;
  cfg.gridDim = dim3((unsigned)(2 * (p.nunits < res ? p.nunits : res)));
  cfg.blockDim = dim3(NUM_THREADS);
  cfg.dynamicSmemBytes = Geo<BN>::SMEM_BYTES;
  cfg.stream = s;
  cfg.attrs = at;
  cfg.numAttrs = 2;
  return cudaLaunchKernelEx(&cfg, k_gemm_dig<BN>, am, bm, p);
}

}  // namespace

int64_t dig_tiles(int64_t rows, int64_t np, int bn, bool upper) {
  if (!upper) return rows / 256 * (np / bn);
  int64_t n = 0;   // tiles whose first row is at most their last column
  for (int64_t r0 = 0; r0 < np; r0 += 256) n += (np - r0 / bn * bn) / bn;
  return n;
}

// Tile width and cut of one product: the fewest clocks of the busiest CTA pair by the
// estimate below, which only has to order the candidates: 2500 or 1700 clocks for four
// k-blocks of a 256- or 128-wide tile and their drain, 6000 or 3000 to store one weight's
// sums, 3000 bytes a clock to read the sums again, 76 pairs on 152 SMs. (The square at N =
// 1001, 40 units of 36 chunks and two weights: 102000 clocks; 47 to 51 us by ncu.)
DigPlan dig_plan(int64_t rows, int64_t np, bool upper, bool with_x) {
  const int nkb = (int)(np / BK);
  const int resident = 76;
  DigPlan best;
  double tbest = 0.0;
  for (int bn = 256; bn >= 128; bn -= 128) {
    const int64_t nt = dig_tiles(rows, np, bn, upper) + (with_x ? dig_tiles(np, np, bn, true) : 0);
    const double sums = ((upper ? 0.5 : 1.0) * (double)rows + (with_x ? 0.5 * (double)np : 0.0)) * (double)np;
    const double chunk = bn == 256 ? 2500.0 : 1700.0, fold = bn == 256 ? 6000.0 : 3000.0;
    for (int parts = 1; parts <= 4; parts *= 2)
      for (int ks = (nkb + KSEG_MAX - 1) / KSEG_MAX; ks <= nkb / KCH; ++ks) {
        const int kseg = ((nkb + ks - 1) / ks + KCH - 1) / KCH * KCH;
        if ((nkb + kseg - 1) / kseg != ks) continue;
        const int64_t units = nt * parts * ks;
        const int64_t waves = (units + resident - 1) / resident;
        const int folds = parts == 1 ? 8 : (parts == 2 ? 5 : 2);
        // clocks: the waves, and the pass that reads the sums' planes
        const double t = (double)waves * ((double)kPairs / parts * (kseg / KCH) * chunk + folds * fold) +
                         (double)ks * sums * 32.0 / 3000.0;
        if (tbest == 0.0 || t < tbest) {
          tbest = t;
          best.bn = bn;
          best.parts = parts;
          best.ksplit = ks;
          best.kseg = kseg;
        }
      }
  }
  return best;
}

cudaError_t launch_digits(const double* src, int64_t rows, const double* src2, int64_t rows2,
                          int64_t np, const DigOperand& o, const DevState* st, int step,
                          cudaStream_t s) {
  auto go = [&](auto kern) {
    launch_dep(kern, (unsigned)(rows + rows2), kDigThreads, 0, s, src, rows, src2, rows + rows2, np, o.dig,
               o.ex, st, step);
  };
  if (rows2 > 0) go(k_digits<true>);
  else go(k_digits<false>);
  return cudaGetLastError();
}

cudaError_t launch_gemm_dig(const DigOperand& A, int64_t rows, const DigOperand& X, int64_t np,
                            int* G, const Tile* tiles, int ntiles, const DigPlan& plan,
                            DevState* st, int step, const TcTuning& tune,
                            cudaStream_t s) {
  if (np % 256 != 0 || rows % 256 != 0 || X.rows < X.off + np || X.off % 256 != 0 ||
      kDigits * rows > (int64_t)1 << 30 || kDigits * X.rows > (int64_t)1 << 30)
    return cudaErrorInvalidValue;
  CUtensorMap am, bm;
  if (!make_map(&am, A.dig, kDigits * rows, np, BM, false) ||
      !make_map(&bm, X.dig, kDigits * X.rows, np, plan.bn / 2, false))
    return cudaErrorInvalidValue;
  DParams p;
  p.nkb = (int)(np / BK);
  p.kseg = plan.kseg;
  p.ksplit = plan.ksplit;
  p.parts = plan.parts;
  p.rows = rows;
  p.np = np;
  p.xrows = X.rows;
  p.xoff = (int)X.off;
  p.G = G;
  p.tiles = tiles;
  p.nunits = ntiles * plan.parts * plan.ksplit;
  p.st = st;
  p.step = step;
  p.wait_ns = tune.wait_ns;
  p.withhold = tune.withhold;
  return plan.bn == 256 ? launch_bn<256>(am, bm, p, s) : launch_bn<128>(am, bm, p, s);
}

static int64_t tri_tiles(int64_t np) { return (np / TE) * (np / TE + 1) / 2; }

// blocks (and partials) of the square's pass: three per SM
int64_t dig_square_nparts(int64_t np) {
  const int64_t n = tri_tiles(np);
  return n < 456 ? n : 456;
}

static SquareArgs square_args(const int* G, int ksplit, int64_t ld, int64_t off, const int* ex,
                              const double* X, double* out, int64_t np, Part3* part,
                              const SimtDecide* dec) {
  SquareArgs a{Sums{G + off, np * ld, ksplit}, ld, ex, X, out, (int)tri_tiles(np),
               (int)dig_square_nparts(np), part, SimtDecide()};
  if (dec) a.dec = *dec;
  return a;
}

cudaError_t launch_dig_square(const int* G, int ksplit, const int* ex, const double* X, double* out,
                              int64_t np, DevState* st, int step, Part3* part,
                              const SimtDecide* dec, cudaStream_t s) {
  const SquareArgs a = square_args(G, ksplit, np, 0, ex, X, out, np, part, dec);
  launch_dep(k_dig_square, (unsigned)a.nblocks, kPassThreads, 0, s, a, np, st, step);
  return cudaGetLastError();
}

cudaError_t launch_dig_symm(const int* G, int ksplit, int64_t rows, const int* ey, const int* ex,
                            const double* yin, double* yout, int64_t np, const DevState* st,
                            int step, cudaStream_t s) {
  const dim3 grid((unsigned)tri_tiles(np), (unsigned)(rows / np));
  launch_dep(k_dig_symm, grid, kPassThreads, 0, s,
             SymmArgs{Sums{G, rows * np, ksplit}, rows, ey, ex, yin, yout}, np, st, step);
  return cudaGetLastError();
}

cudaError_t launch_dig_step(const int* G, int ksplit, int64_t batch, const int* ex, const double* yin,
                            double* yout, const double* X, double* out, int64_t np, DevState* st,
                            int step, Part3* part, const SimtDecide* dec, cudaStream_t s) {
  const int64_t rows = batch * np, ld = rows + np;
  const SquareArgs a = square_args(G, ksplit, ld, rows, ex + rows, X, out, np, part, dec);
  const SymmArgs y{Sums{G, ld * np, ksplit}, ld, ex, ex + rows, yin, yout};
  const int tiles = (int)tri_tiles(np);
  launch_dep(k_dig_step, (unsigned)(a.nblocks + tiles * batch), kPassThreads, 0, s, a, y, tiles, np, st,
             step);
  return cudaGetLastError();
}

cudaError_t launch_dig_plain(const int* G, int ksplit, int64_t rows, const int* ea,
                             const int* ex, double* out, int64_t np, const DevState* st, int step,
                             cudaStream_t s) {
  const dim3 grid((unsigned)(np / TE), (unsigned)(rows / TE));
  launch_dep(k_dig_plain, grid, kPassThreads, 0, s, Sums{G, rows * np, ksplit}, rows, ea, ex, out, np, st, step);
  return cudaGetLastError();
}

}  // namespace sp2
