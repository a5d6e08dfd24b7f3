// Internal declarations shared by the translation units of libsp2.so.
// Not part of the public ABI (that is include/sp2.h).
#pragma once

#include <cuda_runtime.h>
#include <cuda_bf16.h>
#include <cuda_fp16.h>
#include <stddef.h>
#include <stdint.h>

#include "../../include/sp2.h"

namespace sp2 {

// Internal matrices are padded to a multiple of the largest tile edge of their
// arithmetic mode, zero outside the caller's N x N block: 256 for the split
// modes (the tensor-core tiles and the TMA row pitch), 128 for FP32 (its
// CUDA-core tiles), 64 for FP64 (its tiles; GB300's FP64 rate makes every padded
// row count). Zero padding is invariant under all recursions (X -> X^2,
// 2X - X^2, Y -> YX + XY), so it never touches results.
constexpr int kPad = 256;

// Above this N FP64 products run by digits on the tensor cores and matrices are
// padded to kPad (per SP2 step at N = 300: 75 us by digits at np = 512 against 86 us
// on the CUDA cores at np = 320; at N = 200, 72 against 60).
constexpr int64_t kDigMinN = 257;

inline int64_t pad_n(int64_t n, int mode) {
  const int64_t q = mode == SP2_MODE_FP64 && n < kDigMinN ? 64 : (mode == SP2_MODE_FP32 ? 128 : kPad);
  return (n + q - 1) / q * q;
}

// Device-resident SP2 control state: traces of every X_n, the branch signs
// and the stop decision. Written by the step decisions (decide.cuh: k_decide, or the last
// block of a square), the kernels that start a recursion (bounds, given branches) and the
// block-sparse plan, and by products whose wait runs out; read by the step kernels
// (which become no-ops once the recursion has stopped) and by the host.
struct DevState {
  double t1[SP2_MAX_ITER + 2];   // Tr[X_n], index n = 1..M+1
  double t2[SP2_MAX_ITER + 2];   // ||X_n||_F^2
  double f[SP2_MAX_ITER + 2];    // ||X_n - X_n^2||_F^2, known after step n
  int sigma[SP2_MAX_ITER + 2];   // sigma_n, the branch taken by step n (X_n -> X_{n+1})
  int plane1[SP2_MAX_ITER + 2];  // split-tail mode: 1 if step n uses the hi planes alone
  double fill[SP2_MAX_ITER + 2]; // block-sparse: share of the upper blocks step n formed
  int stop_at;                   // M once a stop rule fired, else 0
  int nonfinite;                 // a trace was NaN/Inf
  int abort_flag;                // a device wait timed out (kernel bailed out)
  int pad_;
  double bounds[2];              // Gershgorin eps_min, eps_max
  double fbest;                  // smallest f among the floor candidates (f <= floor_gate)
  int nbest;                     // its iterate index n (X_n), 0 if none yet
  int keep_step;                 // step whose input X_n (and Y_n) is to be kept now
  int backtracked;               // the floor stop returned X_nbest, not the last iterate
  int stop_step;                 // the step after which the stop test fired
  double alpha, beta;            // X_1 = alpha I + beta H, from the (widened) bounds
  double work_kblocks;           // block-sparse: 256-wide K blocks the squares ran, all tiles
  double fold;                   // min f_1..f_{s-kStall} after step s (the stall floor's older part)
};

// What the host learns of a step, in a slot of a pinned host ring written by the step
// decision. A copy of the state on the stream after every step (and an event behind
// it) cost more than a small step's kernels.
struct HostSnap {
  unsigned long long word;       // 2 x token (call and step) + 1 when the recursion ends
                                 // there and the other fields are valid
  int stop_at, nonfinite, abort_flag, backtracked, stop_step, pad_;
  double bounds[2], alpha, beta, work_kblocks;
};

// Storage of one padded matrix (or a batch of them) in a given mode.
struct MatBuf {
  void* master = nullptr;        // double (FP64 mode) or float, rows x np, unscaled
  uint16_t* hi = nullptr;        // split modes: hi plane (bf16 or fp16 bits)
  uint16_t* lo = nullptr;        // split modes: lo plane
  uint16_t* mid = nullptr;       // BF16X3: the middle plane
};

inline bool split_mode(int mode) {
  return mode == SP2_MODE_BF16X2 || mode == SP2_MODE_FP16X2 || mode == SP2_MODE_BF16X3;
}
inline int n_planes(int mode) { return mode == SP2_MODE_BF16X3 ? 3 : (split_mode(mode) ? 2 : 0); }

// Eq. doubleHalf with bfloat16: hi = bf16(v), lo = bf16(v - hi).
__device__ __forceinline__ void split_bf16(float v, uint16_t& h, uint16_t& l) {
  const __nv_bfloat16 hb = __float2bfloat16_rn(v);
  const __nv_bfloat16 lb = __float2bfloat16_rn(v - __bfloat162float(hb));
  h = __bfloat16_as_ushort(hb);
  l = __bfloat16_as_ushort(lb);
}

// Three bfloat16 planes of v: hi = bf16(v), mid = bf16(v - hi), lo = bf16(v - hi - mid).
// Both residuals are exact in FP32, so hi + mid + lo = v for normal v.
__device__ __forceinline__ void split_bf16x3(float v, uint16_t& h, uint16_t& m, uint16_t& l) {
  const __nv_bfloat16 hb = __float2bfloat16_rn(v);
  const float r1 = v - __bfloat162float(hb);
  const __nv_bfloat16 mb = __float2bfloat16_rn(r1);
  const __nv_bfloat16 lb = __float2bfloat16_rn(r1 - __bfloat162float(mb));
  h = __bfloat16_as_ushort(hb);
  m = __bfloat16_as_ushort(mb);
  l = __bfloat16_as_ushort(lb);
}

// The fp16 lo plane holds the residual times 2^11 (one fp16 significand), so
// it stays out of the subnormal range; products with it are scaled back by
// 2^-11 from a separate accumulator.
constexpr float kLoScale = 2048.0f;

// Eq. doubleHalf with fp16 on s * v (s a power of two chosen per matrix so
// that |s v| <= 2^14 < 65504): hi = fp16(s v), lo = fp16((s v - hi) * 2^11).
__device__ __forceinline__ void split_fp16(float v, float s, uint16_t& h, uint16_t& l) {
  const float vs = v * s;
  const __half hh = __float2half_rn(vs);
  const __half ll = __float2half_rn((vs - __half2float(hh)) * kLoScale);
  h = __half_as_ushort(hh);
  l = __half_as_ushort(ll);
}

// Power-of-two plane scale for a matrix whose entries are bounded by `bound`:
// 2^(14 - e) with bound <= 2^e, so every scaled entry is at most 2^14.
__device__ __forceinline__ float pow2_scale(float bound) {
  if (!(bound > 0.0f) || !isfinite(bound)) return 1.0f;
  int e;
  frexpf(bound, &e);
  int k = 14 - e;
  k = k < -120 ? -120 : (k > 120 ? 120 : k);
  return ldexpf(1.0f, k);
}

// four consecutive entries of a matrix (idx a multiple of 4): master and, in the split
// modes, the planes as one 8-byte store each
template <typename ZT, int MODE>
__device__ __forceinline__ void store_y4(MatBuf y, int64_t idx, const ZT (&v)[4], float s) {
  if constexpr (sizeof(ZT) == 4) {
    *reinterpret_cast<float4*>(static_cast<float*>(y.master) + idx) =
        make_float4((float)v[0], (float)v[1], (float)v[2], (float)v[3]);
  } else {
    double2* d = reinterpret_cast<double2*>(static_cast<double*>(y.master) + idx);
    d[0] = make_double2((double)v[0], (double)v[1]);
    d[1] = make_double2((double)v[2], (double)v[3]);
  }
  if (MODE == SP2_MODE_BF16X3) {
    uint16_t h[4], m[4], l[4];
#pragma unroll
    for (int j = 0; j < 4; ++j) split_bf16x3((float)v[j], h[j], m[j], l[j]);
    *reinterpret_cast<uint2*>(y.hi + idx) =
        make_uint2(h[0] | ((uint32_t)h[1] << 16), h[2] | ((uint32_t)h[3] << 16));
    *reinterpret_cast<uint2*>(y.mid + idx) =
        make_uint2(m[0] | ((uint32_t)m[1] << 16), m[2] | ((uint32_t)m[3] << 16));
    *reinterpret_cast<uint2*>(y.lo + idx) =
        make_uint2(l[0] | ((uint32_t)l[1] << 16), l[2] | ((uint32_t)l[3] << 16));
  }
  if (MODE == SP2_MODE_BF16X2 || MODE == SP2_MODE_FP16X2) {
    uint16_t h[4], l[4];
#pragma unroll
    for (int j = 0; j < 4; ++j) {
      if (MODE == SP2_MODE_BF16X2) split_bf16((float)v[j], h[j], l[j]);
      else split_fp16((float)v[j], s, h[j], l[j]);
    }
    *reinterpret_cast<uint2*>(y.hi + idx) =
        make_uint2(h[0] | ((uint32_t)h[1] << 16), h[2] | ((uint32_t)h[3] << 16));
    *reinterpret_cast<uint2*>(y.lo + idx) =
        make_uint2(l[0] | ((uint32_t)l[1] << 16), l[2] | ((uint32_t)l[3] << 16));
  }
}

// Per-matrix scale state of a batch of B response matrices (FP16X2 only).
struct ScaleBuf {
  float* ymax = nullptr;    // [2][B] max |Y| of the matrix in each ping-pong slot
  float* yscale = nullptr;  // [2][B] power-of-two scale of each slot's fp16 planes
  float* zmax = nullptr;    // [2][B] max |Z| of a step's product Z = Y X, by step parity
  int64_t B = 0;
};

enum Epi : int {
  EPI_SQUARE = 0,   // out = sigma>0 ? C : 2 X - C, symmetric (upper tiles, mirrored), traces
  EPI_PLAIN = 1,    // out = C (fp32/fp64 Z), all tiles
  EPI_SYMM = 2,     // out = sigma>0 ? YX+XY : 2Y - (YX+XY), symmetric batch (upper tiles, mirrored)
};

// Per-block partial sums written by the kernels that produce an X_{n+1}:
// t1 = Tr[X_{n+1}], t2 = ||X_{n+1}||_F^2, f = ||X_n - X_n^2||_F^2.
struct Part3 {
  double t1, t2, f;
};

struct Tile {       // one output tile of a product kernel
  int row0;         // first output row (within the stacked A operand)
  int col0;         // first output column
};

// Packed pairs of FP32 values (add / mul / fma.rn.f32x2: each half rounds as the
// scalar operation does, in half the instructions).
__device__ __forceinline__ uint64_t pk2(float x, float y) {
  uint64_t r;
  asm("mov.b64 %0, {%1, %2};" : "=l"(r) : "f"(x), "f"(y));
  return r;
}
__device__ __forceinline__ void upk2(uint64_t v, float& x, float& y) {
  asm("mov.b64 {%0, %1}, %2;" : "=f"(x), "=f"(y) : "l"(v));
}
__device__ __forceinline__ uint64_t add2(uint64_t a, uint64_t b) {
  uint64_t r;
  asm("add.rn.f32x2 %0, %1, %2;" : "=l"(r) : "l"(a), "l"(b));
  return r;
}
__device__ __forceinline__ uint64_t mul2(uint64_t a, uint64_t b) {
  uint64_t r;
  asm("mul.rn.f32x2 %0, %1, %2;" : "=l"(r) : "l"(a), "l"(b));
  return r;
}
__device__ __forceinline__ uint64_t fma2(uint64_t a, uint64_t b, uint64_t c) {
  uint64_t r;
  asm("fma.rn.f32x2 %0, %1, %2, %3;" : "=l"(r) : "l"(a), "l"(b), "l"(c));
  return r;
}
constexpr uint64_t kMinus1x2 = 0xbf800000bf800000ull;   // {-1, -1}
__device__ __forceinline__ uint64_t sub2(uint64_t a, uint64_t b) { return fma2(b, kMinus1x2, a); }

// ---------------------------------------------------------------- dependent launches
// The kernels of a step follow one another within microseconds. Launched as
// programmatic dependents, a kernel's blocks become resident while the one before
// still runs, and wait in dep_sync (first thing in every kernel, before any early
// exit) until it has completed and its writes are visible; as every kernel waits for
// the one before it, all earlier ones are then complete too.
__device__ __forceinline__ void dep_sync() {
  asm volatile("griddepcontrol.launch_dependents;\n\tgriddepcontrol.wait;" ::: "memory");
}

template <typename... P, typename... A>
inline cudaError_t launch_dep(void (*kern)(P...), dim3 grid, dim3 block, size_t smem,
                              cudaStream_t s, A&&... args) {
  cudaLaunchConfig_t cfg = {};
  cudaLaunchAttribute at[1];
  at[0].id = cudaLaunchAttributeProgrammaticStreamSerialization;
  at[0].val.programmaticStreamSerializationAllowed = 1;
  cfg.gridDim = grid;
  cfg.blockDim = block;
  cfg.dynamicSmemBytes = smem;
  cfg.stream = s;
  cfg.attrs = at;
  cfg.numAttrs = 1;
  return cudaLaunchKernelEx(&cfg, kern, static_cast<P>(args)...);
}

// ---------------------------------------------------------------- launchers
// elementwise / reduction kernels (kernels_elem.cu)
// Gershgorin bounds of H into st->bounds (widened for a point spectrum) and the
// coefficients st->alpha, st->beta of X_1 = alpha I + beta H; NaN/Inf bounds set
// st->nonfinite and stop the recursion before its first step (stop_at = -1).
cudaError_t launch_bounds(const void* H, int64_t n, int dtype, double2* part, int nparts,
                          DevState* st, cudaStream_t s);
int bounds_nparts(int64_t n);
// the same from given bounds
cudaError_t launch_set_bounds(DevState* st, double eps_min, double eps_max, cudaStream_t s);
// preset branch signs sigma_1..sigma_m (m <= SP2_MAX_ITER), passed by value
cudaError_t launch_set_sigma(DevState* st, const int8_t* sigma, int m, cudaStream_t s);

// X_1 = alpha I + beta H (or Y_1 = beta B for a batch), caller layout -> padded mode layout.
// diag_only: B given as diagonals (batch x n). symmetrize: use (B + B^T)/2.
// part (nullable): trace partials, one per block.
// FP16X2: planes are written with scale 1 when ymax is null (X), otherwise only
// the master is written and max|entry| per batch entry is accumulated into
// ymax (planes follow from launch_split_scaled).
// coef: INIT_ARGS uses (alpha, beta); INIT_STATE takes alpha, beta from st;
// INIT_STATE_BETA takes (0, st->beta).
enum InitCoef : int { INIT_ARGS = 0, INIT_STATE = 1, INIT_STATE_BETA = 2 };
cudaError_t launch_init(const void* src, int64_t n, int64_t np, int64_t batch, int dtype,
                        int diag_only, int symmetrize, double alpha, double beta, int mode,
                        MatBuf dst, Part3* part, int nparts, float* ymax, cudaStream_t s,
                        int coef = INIT_ARGS, const DevState* st = nullptr);
int init_nparts(int64_t np);

// reduce trace partials of X_n, decide stop/sigma (see DevState)
struct DecideParams {
  int n;             // index of the X just produced (X_n)
  int nparts;
  double nocc, idem_tol, floor_gate;
  int min_iter, max_iter;
  int fixed_m;       // > 0: sigma preset, stop when n - 1 == fixed_m
  double tail_f;     // > 0: single-plane products while f of the last iterate exceeds it
  int ratio_floor = 0;  // block-sparse recursion: the threshold-floor test as well
  HostSnap* snap = nullptr;  // pinned host slot of this step (nullable) and its token
  unsigned long long token = 0;
  const void* keep_src = nullptr;    // small FP64 X_s: the block that takes the decision
  void* keep_dst = nullptr;          // keeps a floor candidate, keep_n vectors of 16 bytes
  int keep_n = 0;
};
constexpr size_t kKeepSmall = (size_t)128 << 10;   // FP64 matrices up to np = 128
constexpr double kRatioGate = 1e-4;   // f from which a pair of opposite steps must cut f 600-fold
cudaError_t launch_decide(const Part3* part, DevState* st, DecideParams p, cudaStream_t s);
// copy `count` entries of the master src -> dst when st->keep_step == step (the
// floor candidate with the smallest f so far), else nothing
cudaError_t launch_keep_best(const void* src, void* dst, int64_t count, int mode, const DevState* st,
                             int step, cudaStream_t s);

// Y_{n+1} = sigma>0 ? Z + Z^T : 2 Y - (Z + Z^T) for a batch; step n reads sigma_n.
// FP16X2: the planes of Y_{n+1} use the scale bounded by 2 max|Z| (+ 2 max|Y_n|
// when sigma<0) from sc (slots slot_in -> slot_out); max|Y_{n+1}| is recorded.
cudaError_t launch_symm_update(const void* Z, MatBuf y_in, MatBuf y_out, int64_t np, int64_t batch,
                               int mode, const DevState* st, int step, ScaleBuf sc, int slot_in,
                               int slot_out, cudaStream_t s);

// padded mode layout -> caller layout (N x N per batch entry), times `scale`
// (times st->beta as well when beta_state is given)
cudaError_t launch_copy_out(MatBuf src, int64_t n, int64_t np, int64_t batch, int mode,
                            double scale, void* dst, int dtype, cudaStream_t s,
                            const DevState* beta_state = nullptr);
// reset of the fields an adjoint recursion does not use (stop, keep, abort, nonfinite)
cudaError_t launch_adjoint_state(DevState* st, cudaStream_t s);

// regenerate hi/lo planes from the FP32 master, rows x np (plane scale 1)
cudaError_t launch_split(MatBuf m, int64_t rows, int64_t np, int mode, cudaStream_t s);
// FP16X2 batch of B matrices: scale of slot `slot` from its ymax, then planes
cudaError_t launch_split_scaled(MatBuf m, int64_t np, ScaleBuf sc, int slot, cudaStream_t s);

// response_contract
cudaError_t launch_contract(const void* P, int64_t L, const void* Q, int64_t K, int64_t n,
                            int dtype, int q_diag, double* part, int nparts, double* out,
                            cudaStream_t s);
int contract_nparts(int64_t n, int q_diag);

// product kernels
// The step decision taken by the last block of a CUDA-core square (one launch
// fewer per step): its parameters, the state it writes, and a completion counter
// that is zero between launches (the last block resets it).
struct SimtDecide {
  DecideParams p;
  DevState* st = nullptr;
  unsigned* done = nullptr;
};
// SIMT (FP64 / FP32): C = A * X with A rows x np (stacked), X np x np symmetric.
// dec (squares only, may be null): take the step decision in the last block.
cudaError_t launch_gemm_simt(int mode, int epi, const void* A, int64_t a_rows, const void* X,
                             int64_t np, void* out, const void* x_prev, Part3* part,
                             const Tile* tiles, int ntiles, int bm, int bn, const DevState* st,
                             int step, cudaStream_t s, const SimtDecide* dec = nullptr);
// output tile of a square (upper) or plain product of a rows x np left factor
void simt_tile_shape(int mode, int64_t rows, int64_t np, bool upper, int* bm, int* bn);

// tcgen05 split-precision (BF16X2 / FP16X2 / BF16X3)
struct TcOperand {   // hi/lo (and BF16X3 mid) planes of a stacked operand, rows x np
  const uint16_t* hi = nullptr;
  const uint16_t* lo = nullptr;
  int64_t rows = 0;
  const uint16_t* mid = nullptr;
};
// Launch settings of the product kernel that are not part of the arithmetic.
struct TcTuning {
  unsigned long long wait_ns = 2000000000ull;  // limit of every mbarrier wait
  int withhold = 0;    // test hook: the first TMA load of CTA 0 is never issued
  int fused_response = 0;  // response step as one EPI_SYMM launch (else EPI_PLAIN + transpose-add)
  int pair = 1;        // 256 x 256 tiles on CTA pairs (tcgen05 cta_group::2), else 128 x 256
};
// (TcLaunch.tail: the split-tail mode; the kernel reads st->plane1[step] and uses
// the hi planes alone, one product per segment pair, where it is set.)
// One product launch: C = P Q (EPI_SQUARE: P = Q = X; EPI_PLAIN: P = stacked A,
// Q = symmetric B; EPI_SYMM: P = stacked symmetric Y, Q = X, C = Y X + X Y).
struct TcLaunch {
  int mode = 0;
  int epi = 0;
  TcOperand P, Q;
  int64_t np = 0;
  MatBuf out;                      // master + planes (planes only for the symmetric epilogues)
  const float* prev = nullptr;     // EPI_SQUARE: X_n master; EPI_SYMM: Y_n master
  Part3* part = nullptr;           // per-tile partials (>= ntiles)
  const Tile* tiles = nullptr;
  int ntiles = 0;
  DevState* st = nullptr;
  int step = 0;
  const float* p_scale = nullptr;  // FP16X2: per batch entry of P, the plane scale to divide out
  const float* q_scale = nullptr;  // FP16X2: the plane scale of Q (nullable)
  const float* o_scale = nullptr;  // FP16X2 EPI_SYMM: per batch entry, scale of the output planes
  float* zmax = nullptr;           // FP16X2 EPI_PLAIN: per batch entry, receives max |C|
  float* zero = nullptr;           // EPI_PLAIN: nzero floats the launch clears
  int nzero = 0;
  int trans = 0;                   // EPI_PLAIN: store each batch entry of C transposed
  int tail = 0;                    // split-tail mode (st->plane1 decides per step)
  TcTuning tune;
  // block-sparse square (CTA pairs): tiles, their count and their K-block lists
  // are written on the device by the plan kernel; ntiles is then the upper bound
  const int* dyn_ntiles = nullptr;
  const int* kcnt = nullptr;
  const uint16_t* klist = nullptr;
  int nbk = 0;                     // K blocks of 256 (np / 256): the stride of klist
  int bn = 256;                    // tile columns: 256, or 128 / 64 (squares and plain products on pairs)
  const SimtDecide* dec = nullptr; // squares with bn < 256: take the step decision in the last CTA
};
cudaError_t launch_gemm_tc(const TcLaunch& L, cudaStream_t s, char* errbuf, size_t errlen);

// ---- block-sparse recursion (sparse_kernels.cu): 256 x 256 blocks, N <= 65536
constexpr int kMaxSparseBlocks = 256;
struct SparseBufs {
  int nb = 0;                      // blocks per dimension (np / 256)
  double tau2 = 0.0;               // a block stays when its norm^2 > tau2 (or it is diagonal)
  uint8_t* mask[2] = {};           // content mask of X[0], X[1] (nb x nb, symmetric)
  Tile* tiles[2] = {};             // tile lists, by step parity (step n squares tiles[n % 2])
  int* ntiles[2] = {};
  int* kcnt[2] = {};
  uint16_t* klist[2] = {};         // nb K blocks per tile
  uint32_t* zero = nullptr;        // blocks to zero: (I << 16) | J, I <= J
  int* nzero = nullptr;
  double* nrm2 = nullptr;          // nb x nb scratch: block norms^2
  Part3* psum = nullptr;           // the decision's one partial: traces of X~, and f
};
// ||block||_F^2 of the upper blocks of a master into nrm2
cudaError_t launch_block_norms(const float* master, int64_t np, int nb, double* nrm2,
                               cudaStream_t s);
// threshold the iterate just formed (init: X_1 from nrm2 and the init partials;
// else the square of `step`, from its two partials per tile), list the blocks to
// zero in buffer xo, reduce the decision's partial, and write the next square's
// tiles and K lists into tiles[tl_out]. No-op after the stop (but for init).
cudaError_t launch_sparse_plan(const SparseBufs& B, int init, int xo, int tl_in, int tl_out,
                               const Part3* part, int nparts_init, DevState* st, int step,
                               cudaStream_t s);
// zero the listed blocks (and mirrors) of x's master and planes
cudaError_t launch_zero_blocks(const SparseBufs& B, MatBuf x, int64_t np, int mode,
                               const DevState* st, int step, int init, cudaStream_t s);
void tc_tile_shape(int pair, int* bm, int* bn);   // output tile of one CTA (pair)
// Tile columns of a product on CTA pairs: narrower tiles where 256-wide ones would
// leave most pairs idle.
int tc_tile_width(int64_t rows, int64_t np, bool upper);

// ---- FP64 products by digits on the tensor cores (gemm_dig.cu), np % 256 == 0
constexpr int kDigPlanes = 8;
struct DigOperand {        // digit planes of a rows x np factor and its rows' exponents
  uint16_t* dig = nullptr; // kDigPlanes x rows x np, bfloat16 integers
  int* ex = nullptr;       // rows
  int64_t rows = 0, off = 0;   // rows of a plane, and the operand's first (a right factor
                               // may be the last matrix of a stacked left one)
};
struct DigPlan {           // tile width of a CTA pair and the cut of a tile's work
  int bn = 256, parts = 1, ksplit = 1, kseg = 4;
};
// with_x: np more rows, of which only the upper tiles are formed
DigPlan dig_plan(int64_t rows, int64_t np, bool upper, bool with_x = false);
int64_t dig_square_nparts(int64_t np);   // partials of launch_dig_square
// digits of src (rows x np) and, below it, of src2 (rows2 x np; rows2 may be 0)
cudaError_t launch_digits(const double* src, int64_t rows, const double* src2, int64_t rows2,
                          int64_t np, const DigOperand& o, const DevState* st, int step,
                          cudaStream_t s);
// G: kDigPlanes x plan.ksplit planes of np x rows 32-bit sums, [j * rows + i] for entry
// (i, j) of A X, over the listed 256 x plan.bn tiles
cudaError_t launch_gemm_dig(const DigOperand& A, int64_t rows, const DigOperand& X, int64_t np,
                            int* G, const Tile* tiles, int ntiles, const DigPlan& plan,
                            DevState* st, int step, const TcTuning& tune, cudaStream_t s);
// the passes from G: the square step with its partials (and, with dec, the step
// decision), the symmetrised response update of a batch, both from one G of the batch's
// rows and X's below them (ex: the exponents likewise), C = A X
cudaError_t launch_dig_square(const int* G, int ksplit, const int* ex, const double* X, double* out,
                              int64_t np, DevState* st, int step, Part3* part,
                              const SimtDecide* dec, cudaStream_t s);
cudaError_t launch_dig_symm(const int* G, int ksplit, int64_t rows, const int* ey, const int* ex,
                            const double* yin, double* yout, int64_t np, const DevState* st,
                            int step, cudaStream_t s);
cudaError_t launch_dig_step(const int* G, int ksplit, int64_t batch, const int* ex, const double* yin,
                            double* yout, const double* X, double* out, int64_t np, DevState* st,
                            int step, Part3* part, const SimtDecide* dec, cudaStream_t s);
cudaError_t launch_dig_plain(const int* G, int ksplit, int64_t rows, const int* ea, const int* ex,
                             double* out, int64_t np, const DevState* st, int step, cudaStream_t s);

// FP16X2 scale of the next symmetric response step: per batch entry, the sum of
// the EPI_SYMM tile partials (||Y_{n+1}||_F^2) and the plane scale of Y_{n+2},
// pow2_scale(2 ||Y_{n+1}||_F) (|Y_{n+2}|_max <= ||Y_{n+2}||_2 <= 2 ||Y_{n+1}||_2).
// No-op when the recursion stopped before `step`.
cudaError_t launch_sym_scale(const Part3* part, int ppt, const Tile* tiles, int ntiles, int64_t np,
                             int64_t batch, const DevState* st, int step, float* scale_out,
                             cudaStream_t s);
// FP16X2: the same bound from a batch's masters (the first response step)
cudaError_t launch_fro_scale(const float* master, int64_t np, int64_t batch, double* part,
                             int nparts, float* scale_out, cudaStream_t s);
int fro_nparts();

// finite temperature (fermi_kernels.cu)
// Max magnitudes of the operands (per batch entry) that fix the FP16X2 plane scale of a
// combination, and where that scale and the result's own max go; null elsewhere.
struct CombineScale {
  const float* z1max = nullptr;
  const float* z2max = nullptr;
  const float* amax = nullptr;
  float* scale = nullptr;
  float* omax = nullptr;     // (must start at 0)
};
// out = z1 (Z1 + Z1^T) + z2 (Z2 + Z2^T) + a A + id I for a batch of padded np x np
// matrices (null operands skipped, I only on the caller's n x n block), with its
// planes when `planes`.
cudaError_t launch_combine(int mode, MatBuf out, int64_t np, int64_t n, int64_t batch,
                           const void* Z1, double z1, const void* Z2, double z2, const void* A,
                           double a, double id, bool planes, const CombineScale& cs,
                           cudaStream_t s);
// out[b] = Tr of the caller's n x n block of batch entry b, FP64
cudaError_t launch_trace(int mode, const void* M, int64_t np, int64_t n, int64_t batch, double* out,
                         cudaStream_t s);

// self-consistent response and MLP (scf_kernels.cu)
cudaError_t launch_sgemm(int64_t M, int64_t N, int64_t K, float alpha, const float* A, int64_t lda,
                         int ta, const float* B, int64_t ldb, int tb, float beta, float* C,
                         int64_t ldc, int relu, int bf16, cudaStream_t s);
cudaError_t launch_site_potential(const double* V, const double* K, const double* q, int64_t F,
                                  int64_t ns, double* u, cudaStream_t s);
cudaError_t launch_expand_sites(const double* u, int64_t F, int64_t ns, int norb, void* out,
                                int dtype, cudaStream_t s);
cudaError_t launch_site_charges(const void* Y, int mode, int64_t F, int64_t ns, int norb,
                                int64_t np, double* q, cudaStream_t s);
cudaError_t launch_residual(const double* qout, const double* q, int64_t total, double* r,
                            double* out2, cudaStream_t s);
cudaError_t launch_axpy_d(double* y, double a, const double* x, int64_t total, cudaStream_t s);
cudaError_t launch_gram(const double* R, int m, int64_t F, int64_t ns, int64_t stride, double* G,
                        cudaStream_t s);
cudaError_t launch_anderson_combine(const double* Qh, const double* Rh, const double* c, int m,
                                    int64_t F, int64_t ns, int64_t stride, double alpha, double* q,
                                    cudaStream_t s);
cudaError_t launch_normalise_rows(const double* r, int64_t F, int64_t ns, float* x, double* nr,
                                  cudaStream_t s);
cudaError_t launch_apply_update(double* q, const float* y, const double* nr, int64_t F, int64_t ns,
                                cudaStream_t s);
cudaError_t launch_mse_grad(const float* Y, const float* T, int64_t total, float scale, float* dY,
                            double* loss, cudaStream_t s);
cudaError_t launch_relu_mask(float* dH, const float* Hr, int64_t total, cudaStream_t s);
cudaError_t launch_adam(float* w, const float* g, float* m, float* v, int64_t total, float lr,
                        float b1, float b2, float eps, int t, cudaStream_t s);

}  // namespace sp2
