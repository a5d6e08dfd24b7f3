// CUDA-core product kernels for the plain FP64 and FP32 forms of the SP2 path
// (the "GPU FP32" arithmetic of Sec. VI.C and an FP64 form for small matrices).
//
// C = A * X with A a stack of row-major (np x np) matrices and X symmetric, so
// X is read row-major as the B operand. Epilogues:
//   EPI_SQUARE  X_{n+1} = sigma>0 ? X_n^2 : 2 X_n - X_n^2 (Eq. DM0) on the tiles
//               meeting the upper triangle; element (i,j), i<j, is written to
//               both (i,j) and (j,i), i>j is skipped, so the result is exactly
//               symmetric. Per-block FP64 partials of Tr[X] and ||X||_F^2.
//   EPI_PLAIN   Z = A X for the response update of Eqs. DM1-DM3.
#include "sp2_internal.h"
#include "decide.cuh"

namespace sp2 {

namespace {

__device__ __forceinline__ bool halted_simt(const DevState* st, int step) {
  const int m = *((volatile const int*)&st->stop_at);
  return m != 0 && step > m;
}

template <typename T> struct Vec;
template <> struct Vec<double> { using type = double2; static constexpr int n = 2; };

template <typename T, int BM, int BN, int BK, int TM, int TN>
__global__ void __launch_bounds__(256)
k_gemm_simt(const T* __restrict__ A, const T* __restrict__ X, int64_t np, int epi,
            T* __restrict__ out, const T* __restrict__ xprev, Part3* __restrict__ part,
            const Tile* __restrict__ tiles, const DevState* st, int step, SimtDecide dec) {
  static_assert((BM / TM) * (BN / TN) == 256, "256 threads");
  using V = typename Vec<T>::type;
  constexpr int VN = Vec<T>::n;
  static_assert(BM * BK == 256 * VN && BN * BK == 256 * VN, "one vector per thread per tile");
  if (halted_simt(st, step)) return;

  __shared__ __align__(16) T As[BK][BM];
  __shared__ __align__(16) T Bs[BK][BN];
  const Tile t = tiles[blockIdx.x];
  const int tid = threadIdx.x;
  const int tx = tid % (BN / TN), ty = tid / (BN / TN);

  // global -> register staging indices
  const int a_r = tid / (BK / VN), a_k = (tid % (BK / VN)) * VN;
  const int b_k = tid / (BN / VN), b_c = (tid % (BN / VN)) * VN;
  const T* a_ptr = A + (int64_t)(t.row0 + a_r) * np + a_k;
  const T* b_ptr = X + (int64_t)b_k * np + t.col0 + b_c;

  T acc[TM][TN];
#pragma unroll
  for (int i = 0; i < TM; ++i)
#pragma unroll
    for (int j = 0; j < TN; ++j) acc[i][j] = (T)0;

  V ra = *reinterpret_cast<const V*>(a_ptr);
  V rb = *reinterpret_cast<const V*>(b_ptr);
  for (int64_t k0 = 0; k0 < np; k0 += BK) {
    {
      const T* pa = reinterpret_cast<const T*>(&ra);
#pragma unroll
      for (int v = 0; v < VN; ++v) As[a_k + v][a_r] = pa[v];
      *reinterpret_cast<V*>(&Bs[b_k][b_c]) = rb;
    }
    __syncthreads();
    if (k0 + BK < np) {  // prefetch the next K slice while this one is consumed
      ra = *reinterpret_cast<const V*>(a_ptr + k0 + BK);
      rb = *reinterpret_cast<const V*>(b_ptr + (k0 + BK) * np);
    }
#pragma unroll
    for (int kk = 0; kk < BK; ++kk) {
      T a[TM], b[TN];
#pragma unroll
      for (int i = 0; i < TM; ++i) a[i] = As[kk][ty + i * (BM / TM)];
#pragma unroll
      for (int j = 0; j < TN; ++j) b[j] = Bs[kk][tx + j * (BN / TN)];
#pragma unroll
      for (int i = 0; i < TM; ++i)
#pragma unroll
        for (int j = 0; j < TN; ++j) acc[i][j] = fma(a[i], b[j], acc[i][j]);
    }
    __syncthreads();
  }

  if (epi == EPI_PLAIN) {
#pragma unroll
    for (int i = 0; i < TM; ++i)
#pragma unroll
      for (int j = 0; j < TN; ++j) {
        const int64_t gi = t.row0 + ty + i * (BM / TM), gj = t.col0 + tx + j * (BN / TN);
        out[gi * np + gj] = acc[i][j];
      }
    return;
  }

  const int sg = st->sigma[step];
  double t1 = 0.0, t2 = 0.0, f = 0.0;
#pragma unroll
  for (int i = 0; i < TM; ++i)
#pragma unroll
    for (int j = 0; j < TN; ++j) {
      const int64_t gi = t.row0 + ty + i * (BM / TM), gj = t.col0 + tx + j * (BN / TN);
      if (gi > gj) continue;
      const T c = acc[i][j];
      const T x = xprev[gi * np + gj];
      const T v = sg > 0 ? c : (T)2 * x - c;
      out[gi * np + gj] = v;
      const double d = (double)v;
      const double r = (double)x - (double)c;  // (X_n - X_n^2)_ij
      if (gi == gj) {
        t1 += d;
        t2 += d * d;
        f += r * r;
      } else {
        out[gj * np + gi] = v;
        t2 += 2.0 * d * d;
        f += 2.0 * r * r;
      }
    }
  // block reduction of the partials (fixed order)
  __shared__ double r1[8], r2[8], r3[8];
  for (int o = 16; o > 0; o >>= 1) {
    t1 += __shfl_xor_sync(0xffffffffu, t1, o);
    t2 += __shfl_xor_sync(0xffffffffu, t2, o);
    f += __shfl_xor_sync(0xffffffffu, f, o);
  }
  if ((tid & 31) == 0) { r1[tid >> 5] = t1; r2[tid >> 5] = t2; r3[tid >> 5] = f; }
  __syncthreads();
  if (tid == 0) {
    double s1 = 0.0, s2 = 0.0, s3 = 0.0;
    for (int w = 0; w < 8; ++w) { s1 += r1[w]; s2 += r2[w]; s3 += r3[w]; }
    part[blockIdx.x] = Part3{s1, s2, s3};
  }
  if (dec.done) last_block_decides(part, dec);   // (partials in fixed order, as the decision kernel)
}

// ------------------------------------------------------------ small FP64
// 8 x 8 tiles for matrices whose 16 x 16 tiles would leave most SMs idle (36 tiles at
// np = 128), with the K axis halved between two groups of 64 threads: one warp per
// scheduler, each np / 2 fused multiply-adds long (64 clocks a warp and instruction on
// the FP64 pipe bound it: 4100 clocks at np = 128, where the 16 x 16 tile takes 16400).
// The whole K panel of both factors sits in shared memory.
constexpr int kSmallMaxN = 192;

__global__ void __launch_bounds__(128)
k_gemm_f64_small(const double* __restrict__ A, const double* __restrict__ X, int64_t np, int epi,
                 double* __restrict__ out, const double* __restrict__ xprev,
                 Part3* __restrict__ part, const Tile* __restrict__ tiles, const DevState* st,
                 int step, SimtDecide dec) {
  if (halted_simt(st, step)) return;
  __shared__ __align__(16) double As[8][kSmallMaxN + 2];   // rows of the left factor
  __shared__ __align__(16) double Bs[kSmallMaxN][8];
  __shared__ double half[64], r3[3][2];
  const Tile t = tiles[blockIdx.x];
  const int n = (int)np, tid = threadIdx.x;
  for (int e = tid; e < 4 * n; e += 128) {   // 16 bytes at a time: 8 rows of n, n rows of 8
    const int r = e / (n / 2), k = (e - r * (n / 2)) * 2;
    const double2 v = *reinterpret_cast<const double2*>(A + (int64_t)(t.row0 + r) * np + k);
    *reinterpret_cast<double2*>(&As[r][k]) = v;
    const int kb = e >> 2, c = (e & 3) * 2;
    *reinterpret_cast<double2*>(&Bs[kb][c]) =
        *reinterpret_cast<const double2*>(X + (int64_t)kb * np + t.col0 + c);
  }
  __syncthreads();
  const int g = tid >> 6, i = (tid & 63) >> 3, j = tid & 7;
  double acc = 0.0;
  const int k1 = (g + 1) * (n / 2);
#pragma unroll 8
  for (int k = g * (n / 2); k < k1; ++k) acc = fma(As[i][k], Bs[k][j], acc);
  if (g == 1) half[tid & 63] = acc;
  __syncthreads();
  const int64_t gi = t.row0 + i, gj = t.col0 + j;
  double t1 = 0.0, t2 = 0.0, f = 0.0;
  if (g == 0) {
    const double c = acc + half[tid];
    if (epi == EPI_PLAIN) {
      out[gi * np + gj] = c;
    } else if (gi <= gj) {
      const int sg = st->sigma[step];
      const double x = xprev[gi * np + gj];
      const double v = sg > 0 ? c : 2.0 * x - c;
      const double r = x - c, w = gi == gj ? 1.0 : 2.0;
      out[gi * np + gj] = v;
      if (gi != gj) out[gj * np + gi] = v;
      t1 = gi == gj ? v : 0.0;
      t2 = w * v * v;
      f = w * r * r;
    }
  }
  if (epi == EPI_PLAIN) return;
  if (g == 0) {
    for (int o = 16; o > 0; o >>= 1) {
      t1 += __shfl_xor_sync(0xffffffffu, t1, o);
      t2 += __shfl_xor_sync(0xffffffffu, t2, o);
      f += __shfl_xor_sync(0xffffffffu, f, o);
    }
    if ((tid & 31) == 0) r3[0][tid >> 5] = t1, r3[1][tid >> 5] = t2, r3[2][tid >> 5] = f;
  }
  __syncthreads();
  if (tid == 0)
    part[blockIdx.x] = Part3{r3[0][0] + r3[0][1], r3[1][0] + r3[1][1], r3[2][0] + r3[2][1]};
  if (dec.done) last_block_decides<true>(part, dec);
}

// ------------------------------------------------------------ FP32
// BM x BN tile, 8 x TN entries per thread (4 x 4 blocks, so that shared memory is read
// 16 bytes at a time; TN = 4 for the smaller tiles, where a tile's warps alone hide the
// latencies), K steps of BK through two shared-memory buffers with the next step's
// global loads in registers. The products are packed pairs (fma.rn.f32x2: each half
// rounds as fmaf): the same rate as scalar ones at half the instructions. Shared-memory
// reads (four wavefronts for 16 bytes a lane) and the FMA pipe bound it about equally;
// the left factor's entries are doubled in registers, since pairs stored in shared
// memory made its reads the bound (N = 1000 square 63 us). Each entry's terms are added
// in the order of k, as by the scalar form.
__device__ __forceinline__ uint64_t ffma2(uint64_t a, uint64_t b, uint64_t c) {
  uint64_t r;
  asm("fma.rn.f32x2 %0, %1, %2, %3;" : "=l"(r) : "l"(a), "l"(b), "l"(c));
  return r;
}
__device__ __forceinline__ uint64_t twice(float x) {
  uint64_t r;
  asm("mov.b64 %0, {%1, %1};" : "=l"(r) : "f"(x));
  return r;
}
__device__ __forceinline__ float2 unpack2(uint64_t v) {
  float2 r;
  asm("mov.b64 {%0, %1}, %2;" : "=f"(r.x), "=f"(r.y) : "l"(v));
  return r;
}

// s + c += x exactly up to the rounding of c (Knuth's TwoSum; the _rn forms are never
// contracted), and the square of r + er
struct SumF32 {
  float s = 0.0f, c = 0.0f;
  __device__ __forceinline__ void add(float x) {
    const float t = __fadd_rn(s, x), bp = __fsub_rn(t, s);
    c = __fadd_rn(c, __fadd_rn(__fsub_rn(s, __fsub_rn(t, bp)), __fsub_rn(x, bp)));
    s = t;
  }
  __device__ __forceinline__ void add_sq(float r, float er = 0.0f) {
    const float p = __fmul_rn(r, r);
    add(p);
    c = __fadd_rn(c, fmaf(2.0f * r, er, fmaf(r, r, -p)));
  }
  __device__ __forceinline__ double value() const { return (double)s + (double)c; }
};

template <int BM, int BN, int BK, int TN>
__global__ void __launch_bounds__(BM / 8 * BN / TN, BM * BN == 128 * 128 ? 2 : (BM == 128 ? 2 : 4))
k_gemm_f32(const float* __restrict__ A, const float* __restrict__ X, int64_t np, int epi,
           float* __restrict__ out, const float* __restrict__ xprev, Part3* __restrict__ part,
           const Tile* __restrict__ tiles, const DevState* st, int step, SimtDecide dec) {
  constexpr int TX = BN / TN, NT = BM / 8 * TX, NH = TN / 4;   // column blocks per thread
  constexpr int AS = BM + 4;                       // entries per k row of the left buffer
  constexpr int A4 = BM * BK / 4 / NT, B4 = BN * BK / 4 / NT;   // 16-byte loads per thread
  if (halted_simt(st, step)) return;
  __shared__ __align__(16) float As[2][BK][AS];
  __shared__ __align__(16) float Bs[2][BK][BN];
  const Tile t = tiles[blockIdx.x];
  const int tid = threadIdx.x, tx = tid % TX, ty = tid / TX;
  const float* ap = A + (int64_t)t.row0 * np;
  const float* bp = X + t.col0;
  float4 ra[A4], rb[B4];
  auto load = [&](int64_t k0) {
#pragma unroll
    for (int i = 0; i < A4; ++i) {
      const int e = tid + i * NT;
      ra[i] = *reinterpret_cast<const float4*>(ap + (int64_t)(e / (BK / 4)) * np + k0 +
                                               (e % (BK / 4)) * 4);
    }
#pragma unroll
    for (int i = 0; i < B4; ++i) {
      const int e = tid + i * NT;
      rb[i] = *reinterpret_cast<const float4*>(bp + (k0 + e / (BN / 4)) * np + (e % (BN / 4)) * 4);
    }
  };
  auto store = [&](int b) {
#pragma unroll
    for (int i = 0; i < A4; ++i) {
      const int e = tid + i * NT, r = e / (BK / 4), k = (e % (BK / 4)) * 4;
      As[b][k + 0][r] = ra[i].x;
      As[b][k + 1][r] = ra[i].y;
      As[b][k + 2][r] = ra[i].z;
      As[b][k + 3][r] = ra[i].w;
    }
#pragma unroll
    for (int i = 0; i < B4; ++i) {
      const int e = tid + i * NT;
      *reinterpret_cast<float4*>(&Bs[b][e / (BN / 4)][(e % (BN / 4)) * 4]) = rb[i];
    }
  };
  uint64_t acc[8][2 * NH];
#pragma unroll
  for (int i = 0; i < 8; ++i)
#pragma unroll
    for (int j = 0; j < 2 * NH; ++j) acc[i][j] = 0ull;
  load(0);
  store(0);
  __syncthreads();
  int buf = 0;
  for (int64_t k0 = 0; k0 < np; k0 += BK, buf ^= 1) {
    const bool more = k0 + BK < np;
    if (more) load(k0 + BK);
#pragma unroll
    for (int kk = 0; kk < BK; ++kk) {
      uint64_t a[8], b[2 * NH];
#pragma unroll
      for (int h = 0; h < 2; ++h) {
        const float4 v = *reinterpret_cast<const float4*>(&As[buf][kk][h * (BM / 2) + ty * 4]);
        a[4 * h] = twice(v.x), a[4 * h + 1] = twice(v.y);
        a[4 * h + 2] = twice(v.z), a[4 * h + 3] = twice(v.w);
      }
#pragma unroll
      for (int h = 0; h < NH; ++h) {
        const ulonglong2 bv =
            *reinterpret_cast<const ulonglong2*>(&Bs[buf][kk][h * (BN / 2) + tx * 4]);
        b[2 * h] = bv.x, b[2 * h + 1] = bv.y;
      }
#pragma unroll
      for (int i = 0; i < 8; ++i)
#pragma unroll
        for (int j = 0; j < 2 * NH; ++j) acc[i][j] = ffma2(a[i], b[j], acc[i][j]);
    }
    if (more) store(buf ^ 1);   // (its readers passed the barrier of the step before)
    __syncthreads();
  }
  // entry (i, j) of this thread: row (i / 4) BM/2 + ty 4 + i % 4, columns likewise
  const int64_t r0 = t.row0 + ty * 4, c0 = t.col0 + tx * 4;
  if (epi == EPI_PLAIN) {
#pragma unroll
    for (int i = 0; i < 8; ++i)
#pragma unroll
      for (int h = 0; h < NH; ++h) {
        const float2 u = unpack2(acc[i][2 * h]), v = unpack2(acc[i][2 * h + 1]);
        *reinterpret_cast<float4*>(out + (r0 + (i >> 2) * (BM / 2) + (i & 3)) * np + c0 +
                                   h * (BN / 2)) = make_float4(u.x, u.y, v.x, v.y);
      }
    return;
  }
  const int sg = st->sigma[step];
  // sums of this thread's entries in FP32 with their rounding errors (FP64
  // instructions on all 64 entries took 34 us of a tile): entries above the diagonal
  // (counted twice) and on it. Tr X - ||X||_F^2 comes within 6 units in the last place of
  // the sums (N = 100 to 4096); a third word per sum would make it 1, and a step of N = 96 to
  // 2000 5 to 18 % longer.
  SumF32 t1, t2, f, e2, ef;
#pragma unroll
  for (int ih = 0; ih < 2; ++ih)
#pragma unroll
    for (int jh = 0; jh < NH; ++jh) {
      const int64_t gi0 = r0 + ih * (BM / 2), gj0 = c0 + jh * (BN / 2);
      if (gi0 > gj0 + 3) continue;   // the 4 x 4 block lies below the diagonal
      const bool above = gi0 + 3 < gj0;
      float v[4][4];
#pragma unroll
      for (int i = 0; i < 4; ++i) {
        const float2 u0 = unpack2(acc[4 * ih + i][2 * jh]), u1 = unpack2(acc[4 * ih + i][2 * jh + 1]);
        const float c[4] = {u0.x, u0.y, u1.x, u1.y};
        const float4 xv = *reinterpret_cast<const float4*>(xprev + (gi0 + i) * np + gj0);
        const float x[4] = {xv.x, xv.y, xv.z, xv.w};
#pragma unroll
        for (int j = 0; j < 4; ++j) {
          v[i][j] = sg > 0 ? c[j] : 2.0f * x[j] - c[j];
          // x - c = r + er exactly
          const float r = __fsub_rn(x[j], c[j]), bb = __fsub_rn(r, x[j]);
          const float er = __fsub_rn(__fsub_rn(x[j], __fsub_rn(r, bb)), __fadd_rn(c[j], bb));
          if (gi0 + i < gj0 + j) {
            t2.add_sq(v[i][j]);
            f.add_sq(r, er);
          } else if (gi0 + i == gj0 + j) {
            t1.add(v[i][j]);
            e2.add_sq(v[i][j]);
            ef.add_sq(r, er);
          }
        }
      }
      if (above) {
#pragma unroll
        for (int i = 0; i < 4; ++i) {
          *reinterpret_cast<float4*>(out + (gi0 + i) * np + gj0) =
              make_float4(v[i][0], v[i][1], v[i][2], v[i][3]);
          *reinterpret_cast<float4*>(out + (gj0 + i) * np + gi0) =
              make_float4(v[0][i], v[1][i], v[2][i], v[3][i]);
        }
      } else {
#pragma unroll
        for (int i = 0; i < 4; ++i)
#pragma unroll
          for (int j = 0; j < 4; ++j) {
            if (gi0 + i > gj0 + j) continue;
            out[(gi0 + i) * np + gj0 + j] = v[i][j];
            if (gi0 + i < gj0 + j) out[(gj0 + j) * np + gi0 + i] = v[i][j];
          }
      }
    }
  double d1 = t1.value(), d2 = 2.0 * t2.value() + e2.value(), d3 = 2.0 * f.value() + ef.value();
  constexpr int NW = NT / 32;
  __shared__ double red[3][NW];
  for (int o = 16; o > 0; o >>= 1) {
    d1 += __shfl_xor_sync(0xffffffffu, d1, o);
    d2 += __shfl_xor_sync(0xffffffffu, d2, o);
    d3 += __shfl_xor_sync(0xffffffffu, d3, o);
  }
  if ((tid & 31) == 0) red[0][tid >> 5] = d1, red[1][tid >> 5] = d2, red[2][tid >> 5] = d3;
  __syncthreads();
  if (tid == 0) {
    double s1 = 0.0, s2 = 0.0, s3 = 0.0;
    for (int w = 0; w < NW; ++w) s1 += red[0][w], s2 += red[1][w], s3 += red[2][w];
    part[blockIdx.x] = Part3{s1, s2, s3};
  }
  if (dec.done) last_block_decides(part, dec);
}

// Tile of an FP32 product: the least work of the busiest SM, a tile's work weighed by
// how well the SM's resident warps hide latency (eight or more: fully).
void f32_tile(int64_t rows, int64_t np, bool upper, int* bm, int* bn) {
  constexpr int kShapes[3][2] = {{128, 128}, {128, 64}, {64, 64}};
  double best = 0.0;
  for (const auto& s : kShapes) {
    const int64_t m = rows / s[0], n = np / s[1];
    int64_t nt = m * n;
    if (upper) {
      nt = 0;
      for (int64_t i = 0; i < m; ++i) nt += (np - i * s[0]) / s[1];
    }
    const int64_t per = (nt + 151) / 152;
    const int warps = s[0] * s[1] / (s[1] == 128 ? 64 : 32) / 32;
    const double w = (double)(per * warps < 8 ? per * warps : 8);
    // (the narrow tiles read more shared memory per multiply-add)
    const double c = (double)per * s[0] * s[1] / (0.55 + 0.45 * w / 8.0) / (s[1] == 128 ? 1.0 : 0.85);
    if (best == 0.0 || c < 0.97 * best) {
      best = c;
      *bm = s[0];
      *bn = s[1];
    }
  }
}

}  // namespace

// FP64 runs at a small fraction of the FP32 rate on GB300, so an FP64 product
// takes as long as its busiest SM: 8 x 8 tiles up to np = 192 for a square or a
// single product (at np = 128 16 x 16 tiles keep 36 SMs busy), 16 x 16 up to
// np = 1024 (136 upper tiles at np = 256, where 64 x 64 would keep 10 SMs busy),
// above that 64 x 64.
void simt_tile_shape(int mode, int64_t rows, int64_t np, bool upper, int* bm, int* bn) {
  if (mode == SP2_MODE_FP64) {
    const int t = np <= kSmallMaxN && rows == np ? 8 : (np <= 1024 ? 16 : 64);
    *bm = t;
    *bn = t;
  } else {
    f32_tile(rows, np, upper, bm, bn);
  }
}

// Plain launches: as programmatic dependents their blocks shared SMs unevenly with the
// blocks before them (FP32 forward chi at N = 1500 11.0 -> 19.4 ms).
cudaError_t launch_gemm_simt(int mode, int epi, const void* A, int64_t a_rows, const void* X,
                             int64_t np, void* out, const void* x_prev, Part3* part,
                             const Tile* tiles, int ntiles, int bm, int bn, const DevState* st,
                             int step, cudaStream_t s, const SimtDecide* dec) {
  (void)a_rows;
  if (ntiles <= 0) return cudaSuccess;
  SimtDecide sd;
  if (dec && epi == EPI_SQUARE) sd = *dec;
  if (mode == SP2_MODE_FP64 && bm == 8) {
    k_gemm_f64_small<<<ntiles, 128, 0, s>>>(
        static_cast<const double*>(A), static_cast<const double*>(X), np, epi,
        static_cast<double*>(out), static_cast<const double*>(x_prev), part, tiles, st, step, sd);
  } else if (mode == SP2_MODE_FP64 && bm == 16) {
    k_gemm_simt<double, 16, 16, 32, 1, 1><<<ntiles, 256, 0, s>>>(static_cast<const double*>(A), static_cast<const double*>(X), np, epi,
        static_cast<double*>(out), static_cast<const double*>(x_prev), part, tiles, st, step, sd);
  } else if (mode == SP2_MODE_FP64) {
    k_gemm_simt<double, 64, 64, 8, 4, 4><<<ntiles, 256, 0, s>>>(static_cast<const double*>(A), static_cast<const double*>(X), np, epi,
        static_cast<double*>(out), static_cast<const double*>(x_prev), part, tiles, st, step, sd);
  } else {
    const float *a = static_cast<const float*>(A), *x = static_cast<const float*>(X);
    const float* xp = static_cast<const float*>(x_prev);
    float* o = static_cast<float*>(out);
    if (bm == 128 && bn == 128)
      k_gemm_f32<128, 128, 8, 8><<<ntiles, 256, 0, s>>>(a, x, np, epi, o, xp, part, tiles, st, step, sd);
    else if (bm == 128)
      k_gemm_f32<128, 64, 16, 4><<<ntiles, 256, 0, s>>>(a, x, np, epi, o, xp, part, tiles, st, step, sd);
    else
      k_gemm_f32<64, 64, 16, 4><<<ntiles, 128, 0, s>>>(a, x, np, epi, o, xp, part, tiles, st, step, sd);
  }
  return cudaGetLastError();
}

}  // namespace sp2
