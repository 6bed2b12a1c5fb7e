// CP fitting by alternating least squares (Sec. 2.3, eq. cp_als) and its
// skew-preserving variant ALS-skew (Sec. 3.3, eq. skew_abc_struct,
// eq. cp_als_quad), with the MTTKRP of every subproblem on the tensor cores.
//
// Each least-squares subproblem is solved through its normal equations,
//   A_m = MTTKRP_m * (Hadamard product of the other two Gram matrices)^-1,
// where MTTKRP_m = X_(m) (P kr Q) is the K2 contraction with the Khatri-Rao
// operand built from the two other factors.  The tensor is kept in three
// BF16 layouts, one per matricization, each in the K2 row format (rows of
// round_up(n, 64) values):
//   X1[i][j][k]  (rows i: P = A2 over j, Q = A3 over k)
//   X2[j][i][k]  (rows j: P = A1 over i, Q = A3 over k)
//   X3[k][i][j]  (rows k: P = A1 over i, Q = A2 over j)
// Everything after the upload stays on the device: the factors, their FP64
// Gram matrices, and the rank x rank SPD solves (a blocked FP64 Cholesky of
// the normal matrix, then one warp per row for the two triangular solves;
// rank^3/3 + 2 n rank^2 flops per update).  Only the Cholesky breakdown flag,
// the residual's two sums and the final factors come back to the host.
#include <algorithm>
#include <cmath>
#include <cstring>
#include <new>
#include <vector>

#include "ds_arith.cuh"
#include "grom_internal.h"
#include "ptx.cuh"

using namespace grom;

constexpr int ALS_PARTS = 256;  // blocks of the residual's reductions

// Of one solve, written by its kernels: whether a pivot broke down, and device
// clock values in ns at the start and end of the factorisation, of the triangular
// solves.  (Events around them cost a small fit 2 %: three more records an update
// on its chain of dependent launches.)
struct AlsSolve {
  int bad, pad;
  unsigned long long f0, f1, s0, s1;
};

struct grom_als {
  int64_t n = 0, np = 0;
  cudaStream_t stream = nullptr;
  int sm_count = 0;
  uint8_t* x[3] = {nullptr, nullptr, nullptr};  // BF16 layouts X1, X2, X3
  CUtensorMap tmap[3];
  double xnorm2 = 0.0;  // ||X||_F^2 of the BF16 tensor the fit sees
  int* err = nullptr;
  // per-fit buffers (grown on demand), FP64 on the device
  int64_t rcap = 0;
  double* f[3] = {nullptr, nullptr, nullptr};     // factors, n x rank
  double* anew = nullptr;                         // a least-squares update, n x rank
  double* b1 = nullptr;                           // ALS-skew's shared factor, n x rank/2
  double* mt = nullptr;                           // MTTKRP output, rank x n
  double* gram[3] = {nullptr, nullptr, nullptr};  // Gram matrices of the factors, rank x rank
  double* h = nullptr;                            // normal matrix, then its Cholesky factor L
  double* lt = nullptr;                           // L^T
  double* rdiag = nullptr;                        // reciprocals of L's diagonal
  double* part = nullptr;                         // 2 x ALS_PARTS reduction partials
  AlsSolve* solve = nullptr;                      // on the device: the last solve's flag and times
  void* k2s = nullptr;
  size_t k2s_bytes = 0;
  // timing since the last grom_als_stats: device times of the tensor-core
  // launches (CUDA events) and of the SPD solves (each factorisation, whatever
  // runs beside it, and the triangular solves)
  cudaEvent_t ev0 = nullptr, ev1 = nullptr;
  cudaStream_t side = nullptr;                    // the factorisations' stream
  cudaEvent_t fork = nullptr, join = nullptr;
  double mttkrp_ms = 0.0, solve_ms = 0.0;
  int64_t mttkrp_calls = 0;
};

namespace {

// X1 and X2 rows of a slab of test indices [i0, i0 + cnt) (FP64 input rows
// (i, j) of n values), rounded once to BF16.
__global__ void k_als_x12(const double* __restrict__ src, int64_t cnt, int64_t n, int64_t np, int64_t i0,
                          __nv_bfloat16* __restrict__ x1, __nv_bfloat16* __restrict__ x2) {
  const int64_t total = cnt * n * n;
  for (int64_t t = (int64_t)blockIdx.x * blockDim.x + threadIdx.x; t < total; t += (int64_t)gridDim.x * blockDim.x) {
    const int64_t il = t / (n * n), rem = t - il * n * n, j = rem / n, k = rem - j * n;
    const int64_t i = i0 + il;
    const __nv_bfloat16 v = __double2bfloat16(src[t]);
    x1[(i * n + j) * np + k] = v;
    x2[(j * n + i) * np + k] = v;
  }
}

// X3[k][i][j] = X[i][j][k]: a 32 x 32 tile of (j, k) per block through shared
// memory, coalesced on both sides.
__global__ void k_als_x3(const double* __restrict__ src, int64_t n, int64_t np, int64_t i0,
                         __nv_bfloat16* __restrict__ x3) {
  __shared__ double tile[32][33];
  const int64_t il = blockIdx.z;
  const int64_t jb = (int64_t)blockIdx.x * 32, kb = (int64_t)blockIdx.y * 32;
  const double* s = src + il * n * n;
  for (int r = threadIdx.y; r < 32; r += blockDim.y) {
    const int64_t j = jb + r, k = kb + threadIdx.x;
    tile[r][threadIdx.x] = (j < n && k < n) ? s[j * n + k] : 0.0;
  }
  __syncthreads();
  const int64_t i = i0 + il;
  for (int r = threadIdx.y; r < 32; r += blockDim.y) {
    const int64_t k = kb + r, j = jb + threadIdx.x;
    if (j < n && k < n) x3[(k * n + i) * np + j] = __double2bfloat16(tile[threadIdx.x][r]);
  }
}

// Per-block partial sums of x^2 over the BF16-rounded values, the tensor the
// fit sees (summed on the host in block order).
__global__ void k_als_norm(const double* __restrict__ src, int64_t total, double* part) {
  __shared__ double sh[256];
  double s = 0.0;
  for (int64_t t = (int64_t)blockIdx.x * blockDim.x + threadIdx.x; t < total; t += (int64_t)gridDim.x * blockDim.x) {
    const double x = (double)__bfloat162float(__double2bfloat16(src[t]));
    s = fma(x, x, s);
  }
  sh[threadIdx.x] = s;
  __syncthreads();
  for (int w = 128; w > 0; w >>= 1) {
    if ((int)threadIdx.x < w) sh[threadIdx.x] += sh[threadIdx.x + w];
    __syncthreads();
  }
  if (threadIdx.x == 0) part[blockIdx.x] = sh[0];
}

// The tile (row tj <= column ti) at place x of a triangle taken row by row.
__device__ __forceinline__ void triangle_tile(int64_t x, int64_t& ti, int64_t& tj) {
  ti = (int64_t)((sqrt((double)(8 * x + 1)) - 1.0) / 2.0);
  while ((ti + 1) * (ti + 2) / 2 <= x) ++ti;
  while (ti * (ti + 1) / 2 > x) --ti;
  tj = x - ti * (ti + 1) / 2;
}

// G = F^T F for F (n x r, row-major FP64), 16 x 16 output tiles; G is
// symmetric, so only the tiles on and above the diagonal are computed (FP64
// runs at about two operations per clock per SM here) and mirrored.  Chunks
// of 64 rows with the next one in flight, so that two warps per FP64 pipe
// keep it busy.  A CTA per tile of the triangle and none beside it: in a
// square grid the CTAs that leave at once take places of the first wave, and
// the working ones pair up on SMs while others idle (n = 512, r = 256, 136
// tiles: 37.9 us against 68.0; the pipe's own time is 32 us).
constexpr int GR_K = 64;
__global__ void __launch_bounds__(256) k_gram(const double* __restrict__ F, int64_t n, int64_t r,
                                              double* __restrict__ G) {
  __shared__ double a[GR_K][17], b[GR_K][17];
  int64_t ti, tj;
  triangle_tile(blockIdx.x, ti, tj);
  const int tx = threadIdx.x, ty = threadIdx.y;
  const int64_t ra = tj * 16 + tx, col = ti * 16 + tx;
  double na[GR_K / 16], nb[GR_K / 16];
  auto fetch = [&](int64_t i0) {
#pragma unroll
    for (int k = 0; k < GR_K / 16; ++k) {
      const int64_t i = i0 + 16 * k + ty;
      na[k] = i < n && ra < r ? F[i * r + ra] : 0.0;
      nb[k] = i < n && col < r ? F[i * r + col] : 0.0;
    }
  };
  fetch(0);
  double s = 0.0;
  for (int64_t i0 = 0; i0 < n; i0 += GR_K) {
#pragma unroll
    for (int k = 0; k < GR_K / 16; ++k) {
      a[16 * k + ty][tx] = na[k];
      b[16 * k + ty][tx] = nb[k];
    }
    __syncthreads();
    if (i0 + GR_K < n) fetch(i0 + GR_K);
#pragma unroll 16
    for (int q = 0; q < GR_K; ++q) s = fma(a[q][ty], b[q][tx], s);
    __syncthreads();
  }
  const int64_t row = tj * 16 + ty;
  if (row < r && col < r) {
    G[row * r + col] = s;
    G[col * r + row] = s;
  }
}

// ------------------------------------------------ SPD solves on the device
// The normal equations A = M H^-1 with H = Ga o Gb + (ridge + mu) max diag(Ga o Gb) I.

// H, with the diagonal maximum found by every block (r entries).
__global__ void k_als_normal(const double* __restrict__ Ga, const double* __restrict__ Gb, int64_t r, double rel,
                             double* __restrict__ H, AlsSolve* solve) {
  if (blockIdx.x == 0 && threadIdx.x == 0) solve->f0 = ptx::globaltimer();
  __shared__ double wm[32];
  double m = 0.0;
  for (int64_t a = threadIdx.x; a < r; a += blockDim.x) m = fmax(m, Ga[a * r + a] * Gb[a * r + a]);
  for (int o = 16; o; o >>= 1) m = fmax(m, __shfl_xor_sync(0xffffffffu, m, o));
  if ((threadIdx.x & 31) == 0) wm[threadIdx.x >> 5] = m;
  __syncthreads();
  m = 0.0;
  for (int w = 0; w < (int)(blockDim.x >> 5); ++w) m = fmax(m, wm[w]);
  const double add = rel * m;
  for (int64_t t = (int64_t)blockIdx.x * blockDim.x + threadIdx.x; t < r * r; t += (int64_t)gridDim.x * blockDim.x) {
    const int64_t a = t / r;
    H[t] = Ga[t] * Gb[t] + (t == a * r + a ? add : 0.0);
  }
}

constexpr int CH = 32;  // Cholesky block
constexpr int UT = 16;  // trailing-update tile

// 1/sqrt(d) for a positive finite d: the exponent is split off so that the
// mantissa part m in [1, 4) takes an FP32 estimate, which two Newton-Raphson
// steps for the reciprocal square root, y <- y (3 - m y^2) / 2, bring to FP64
// precision (each step about doubles the correct bits).  FP64 division and
// square root cost thousands of cycles on this part, a step of this a few
// hundred.  The exponents are moved as integers: only the steps' six FP64
// operations are left on the chain.
__device__ __forceinline__ double rsqrt_nr(double d) {
  int hi = __double2hiint(d), up = 0;
  int lo = __double2loint(d);
  if (hi < 0x00100000) {  // subnormal: 2^108 d first
    d *= 0x1p108;
    hi = __double2hiint(d);
    lo = __double2loint(d);
    up = 54;
  }
  const int e = ((hi >> 20) - 1023) >> 1;
  hi -= e * (1 << 21);
  const double h = __hiloint2double(hi - (1 << 20), lo);  // m / 2
  double y = f2d_int(rsqrtf(d2f_int(__hiloint2double(hi, lo))));
  y = y * (1.5 - h * y * y);
  y = y * (1.5 - h * y * y);
  return __hiloint2double(__double2hiint(y) - (e - up) * (1 << 20), __double2loint(y));
}

// Factors the diagonal block at (kb, kb) in place (lower), right-looking, and
// stores the reciprocals of its pivots in rdiag[kb ..].  A pivot that is not
// positive and finite sets *flag.  The chain of dependent FP64 operations from
// one pivot to the next bounds it (some 70 cycles each), so warp 0, alone on
// its FP64 pipe, runs only that chain: lane = row, it holds column c, takes
// the pivot's reciprocal root, scales the column and brings column c + 1 up to
// date.  Warps 1 to 3 hold the block (lane = column, rows warp - 1, + 3, ...)
// and apply column c - 1 meanwhile; what warp 0 gets of column c + 1 is
// therefore short of the columns c - 1 and c, which it applies itself.  Every
// entry sees the columns in the same order as one after the other.  One
// barrier a pivot; us a block, 32 pivots: 24.6 against 38.2 with the update
// between two pivots, 50.5 with a thread per entry.
constexpr int CD_ROWS = (CH + 2) / 3;
__global__ void __launch_bounds__(128) k_chol_diag(double* H, int64_t r, int64_t kb, double* rdiag, int* flag) {
  __shared__ double Ls[CH][CH + 1], col[2][CH], lb[2][CH];
  const int lane = threadIdx.x & 31, w = threadIdx.x >> 5;
  const int nb = (int)(r - kb < CH ? r - kb : CH);
  auto entry = [&](int i, int j) {
    return i < nb && j <= i ? H[(kb + i) * r + kb + j] : (j == i ? 1.0 : 0.0);
  };
  double a[CD_ROWS];
  double cc = 0.0, lp = 0.0;  // warp 0: column c, the scaled column c - 1
  if (w == 0) {
    cc = entry(lane, 0);
  } else {
#pragma unroll
    for (int k = 0; k < CD_ROWS; ++k) {
      const int i = w - 1 + 3 * k;
      a[k] = i < CH ? entry(i, lane) : 0.0;
      if (i < CH && lane == 1) col[1][i] = a[k];
    }
  }
  __syncthreads();
  for (int c = 0; c < nb; ++c) {
    int bad = 0;
    if (w == 0) {
      const double d = __shfl_sync(0xffffffffu, cc, c);
      const long long bits = __double_as_longlong(d);
      if (bits <= 0 || bits >= 0x7ff0000000000000ll) {  // not positive and finite; the same in every lane
        if (lane == 0) atomicExch(flag, 1);
        bad = 1;
      } else {
        double x = col[(c + 1) & 1][lane];
        if (c > 0) x = fma(-__shfl_sync(0xffffffffu, lp, (c + 1) & 31), lp, x);
        const double y = rsqrt_nr(d);
        const double l = cc * y;  // L[lane][c] for lane > c
        Ls[lane][c] = lane > c ? l : lane == c ? d * y : 0.0;
        lb[c & 1][lane] = l;
        if (lane == 0) rdiag[kb + c] = y;
        cc = fma(-__shfl_sync(0xffffffffu, l, (c + 1) & 31), l, x);
        lp = l;
      }
    } else {
      const double l = c > 0 ? lb[(c - 1) & 1][lane] : 0.0;
#pragma unroll
      for (int k = 0; k < CD_ROWS; ++k) {
        const int i = w - 1 + 3 * k;
        if (i < c || i >= CH) continue;  // warp-uniform
        if (c > 0) a[k] = fma(-__shfl_sync(0xffffffffu, l, i), l, a[k]);
        if (lane == c + 2) col[c & 1][i] = a[k];
      }
    }
    if (__syncthreads_or(bad)) return;
  }
  for (int x = threadIdx.x; x < nb * CH; x += 128)
    if (x % CH < nb) H[(kb + x / CH) * r + kb + x % CH] = Ls[x / CH][x % CH];
}

// Rows i >= kb + CH: H[i][kb .. kb+CH) <- H[i][kb .. kb+CH) L11^-T (one warp
// per row, forward substitution with lane = column).
__global__ void k_chol_panel(double* H, int64_t r, int64_t kb, const double* __restrict__ rdiag) {
  __shared__ double L11[CH][CH + 1];  // column CH: reciprocals of the pivots
  const int lane = threadIdx.x & 31;
  for (int t = threadIdx.x >> 5; t < CH; t += blockDim.x >> 5) L11[t][lane] = H[(kb + t) * r + kb + lane];
  if (threadIdx.x < CH) L11[threadIdx.x][CH] = rdiag[kb + threadIdx.x];
  __syncthreads();
  const int64_t i = kb + CH + (int64_t)blockIdx.x * (blockDim.x >> 5) + (threadIdx.x >> 5);
  if (i >= r) return;
  double v = H[i * r + kb + lane];
  for (int c = 0; c < CH; ++c) {
    const double xc = __shfl_sync(0xffffffffu, v, c) * L11[c][CH];
    if (lane == c) v = xc;
    else if (lane > c) v -= L11[lane][c] * xc;
  }
  H[i * r + kb + lane] = v;
}

// H[i][j] -= sum_t L[i][kb+t] L[j][kb+t] for kb + CH <= j <= i < r, one CTA
// (one thread per entry) per UT x UT tile of the lower trailing matrix.
__global__ void __launch_bounds__(UT * UT) k_chol_update(double* H, int64_t r, int64_t kb) {
  __shared__ double Pi[UT][CH + 1], Pj[UT][CH + 1];
  int64_t ti, tj;
  triangle_tile(blockIdx.x, ti, tj);
  const int64_t i0 = kb + CH + ti * UT, j0 = kb + CH + tj * UT;
  const int tx = threadIdx.x % UT, ty = threadIdx.x / UT;
  for (int e = threadIdx.x; e < UT * CH; e += UT * UT) {
    const int q = e / CH, t = e % CH;
    Pi[q][t] = i0 + q < r ? H[(i0 + q) * r + kb + t] : 0.0;
    Pj[q][t] = j0 + q < r ? H[(j0 + q) * r + kb + t] : 0.0;
  }
  __syncthreads();
  const int64_t i = i0 + ty, j = j0 + tx;
  if (i < r && j <= i) {
    double acc = 0.0;
#pragma unroll 8
    for (int t = 0; t < CH; ++t) acc = fma(Pi[ty][t], Pj[tx][t], acc);
    H[i * r + j] -= acc;
  }
}

__global__ void k_transpose(const double* __restrict__ L, int64_t r, double* __restrict__ Lt, AlsSolve* solve) {
  for (int64_t t = (int64_t)blockIdx.x * blockDim.x + threadIdx.x; t < r * r; t += (int64_t)gridDim.x * blockDim.x) {
    const int64_t a = t / r, b = t - a * r;
    Lt[t] = L[b * r + a];
  }
  if (threadIdx.x == 0) atomicMax(&solve->f1, (unsigned long long)ptx::globaltimer());
}

// A[i][:] = M[i][:] H^-1 (M given transposed, r x n; H = L L^T): forward
// L z = m_i, backward L^T a_i = z, 32 unknowns at a time, SV_ROWS rows per CTA
// and four warps per row.  Per block the solved unknowns' contribution is
// summed with lanes over the contracted index (coalesced rows of L or L^T,
// eight unknowns a warp, a butterfly across the lanes), then one warp of the
// row (each row's on another FP64 pipe; the rows of a CTA run at their own
// pace) solves the 32 x 32 triangle, staged in shared memory with the
// reciprocals of its pivots, with shuffles.
// n r^2 multiply-adds (53 us of the FP64 pipe at n = 512, r = 256) and the
// triangles' chains of 2 r shuffle-multiply-add steps bound it: 154 us
// there (192 with the triangle loaded when its turn comes); one warp per row,
// with 32 sums of its own, took 400.
constexpr int SV_ROWS = 4, SV_WARPS = 4, SV_T = CH / SV_WARPS;
constexpr int SV_FETCH = (CH * CH + 32 * (SV_WARPS - 1) - 1) / (32 * (SV_WARPS - 1));

// Butterfly sums over the 32 lanes of v[0 .. 8): every pair of partial sums
// is added in the order 16, 8, 4, 2, 1, and lane l ends with v[(l >> 2) & 7]
// of the order below (bit 4 of the lane picks the upper four, and so on).
__device__ __forceinline__ double warp_sum8(double (&v)[SV_T], int lane) {
#pragma unroll
  for (int h = SV_T / 2, s = 16; h >= 1; h >>= 1, s >>= 1) {
    const bool up = (lane & s) != 0;
#pragma unroll
    for (int c = 0; c < h; ++c) {
      const double send = up ? v[c] : v[c + h];
      const double keep = up ? v[c + h] : v[c];
      v[c] = keep + __shfl_xor_sync(0xffffffffu, send, s);
    }
  }
  double x = v[0];
  x += __shfl_xor_sync(0xffffffffu, x, 2);
  x += __shfl_xor_sync(0xffffffffu, x, 1);
  return x;
}

__global__ void __launch_bounds__(32 * SV_ROWS * SV_WARPS)
    k_als_rowsolve(const double* __restrict__ L, const double* __restrict__ Lt, const double* __restrict__ rdiag,
                   const double* __restrict__ Mt, int64_t n, int64_t r, double* __restrict__ A, AlsSolve* solve) {
  if (blockIdx.x == 0 && threadIdx.x == 0) solve->s0 = ptx::globaltimer();
  extern __shared__ double ybuf[];
  __shared__ double Bs[SV_ROWS][CH][CH + 1];
  const int lane = threadIdx.x & 31, w = threadIdx.x >> 5, row = w / SV_WARPS, sub = w % SV_WARPS;
  const int64_t i0 = (int64_t)blockIdx.x * SV_ROWS, i = i0 + row;
  double* y = ybuf + (size_t)row * r;
  double(*B)[CH + 1] = Bs[row];
  auto row_sync = [&] { asm volatile("bar.sync %0, %1;" ::"r"(row + 1), "r"(32 * SV_WARPS) : "memory"); };
  for (int64_t t = threadIdx.x; t < SV_ROWS * r; t += blockDim.x) {
    const int64_t c = t / SV_ROWS, q = t % SV_ROWS;
    ybuf[q * r + c] = i0 + q < n ? Mt[c * n + i0 + q] : 0.0;
  }
  __syncthreads();
  const int64_t last = (r - 1) / CH * CH;
  // the triangle of the next block, on its way while the row's solver works:
  // by the row's other warps, in their registers
  const int solver = row % SV_WARPS;
  const int ft = (sub + SV_WARPS - 1 - solver) % SV_WARPS * 32 + lane;  // 0 .. 95 in them
  double bn[SV_FETCH], rn = 0.0;
  auto fetch = [&](const double* M, int64_t a0, int nb) {
#pragma unroll
    for (int k = 0; k < SV_FETCH; ++k) {
      const int t = ft + k * 32 * (SV_WARPS - 1);
      bn[k] = t < CH * CH && t / CH < nb && t % CH < nb ? M[(a0 + t / CH) * r + a0 + t % CH] : 0.0;
    }
    if (ft < nb) rn = rdiag[a0 + ft];
  };
  if (sub != solver) fetch(L, 0, (int)(r < CH ? r : CH));
  for (int pass = 0; pass < 2; ++pass) {
    const double* M = pass ? Lt : L;
    for (int64_t x = 0; x <= last; x += CH) {
      const int64_t a0 = pass ? last - x : x;
      const int nb = (int)(r - a0 < CH ? r - a0 : CH);
      const int64_t q0 = pass ? a0 + nb : 0, q1 = pass ? r : a0;  // the solved unknowns
      if (sub != solver) {
#pragma unroll
        for (int k = 0; k < SV_FETCH; ++k) {
          const int t = ft + k * 32 * (SV_WARPS - 1);
          if (t < CH * CH) B[t / CH][t % CH] = bn[k];
        }
        if (ft < CH) B[ft][CH] = rn;
      }
      double acc[SV_T];
#pragma unroll
      for (int t = 0; t < SV_T; ++t) acc[t] = 0.0;
      const double* Mr = M + (a0 + sub * SV_T) * r;
#pragma unroll 2
      for (int64_t q = q0 + lane; q < q1; q += 32) {
        const double yq = y[q];
#pragma unroll
        for (int t = 0; t < SV_T; ++t)
          if (sub * SV_T + t < nb) acc[t] = fma(Mr[t * r + q], yq, acc[t]);
      }
      const double v8 = warp_sum8(acc, lane);
      if ((lane & 3) == 0 && sub * SV_T + (lane >> 2) < nb) y[a0 + sub * SV_T + (lane >> 2)] -= v8;
      row_sync();
      if (sub == solver) {
        double v = lane < nb ? y[a0 + lane] : 0.0;
        for (int k = 0; k < nb; ++k) {
          const int c = pass ? nb - 1 - k : k;
          const double xc = __shfl_sync(0xffffffffu, v, c) * B[c][CH];
          const bool open = pass ? lane < c : lane > c && lane < nb;
          if (lane == c)
            v = xc;
          else if (open)
            v -= B[lane][c] * xc;
        }
        if (lane < nb) {
          y[a0 + lane] = v;
          if (pass && i < n) A[i * r + a0 + lane] = v;
        }
      } else if (x < last || pass == 0) {
        const int64_t a1 = pass ? a0 - CH : x < last ? a0 + CH : last;
        fetch(x < last ? M : Lt, a1, (int)(r - a1 < CH ? r - a1 : CH));
      }
      row_sync();
    }
  }
  __syncthreads();
  if (threadIdx.x == 0) atomicMax(&solve->s1, (unsigned long long)ptx::globaltimer());
}

// Block b of ALS_PARTS: partial sums of <A, M> (A n x r, M^T r x n) into
// part[b] and of sum G0 o G1 o G2 (r x r) into part[ALS_PARTS + b], each in a
// fixed order.
__device__ __forceinline__ double block_sum(double v, double* sh) {
  for (int o = 16; o; o >>= 1) v += __shfl_xor_sync(0xffffffffu, v, o);
  if ((threadIdx.x & 31) == 0) sh[threadIdx.x >> 5] = v;
  __syncthreads();
  double t = 0.0;
  for (int w = 0; w < (int)(blockDim.x >> 5); ++w) t += sh[w];
  return t;
}

__global__ void k_als_residual_parts(const double* __restrict__ A, const double* __restrict__ Mt, int64_t n, int64_t r,
                                     const double* __restrict__ G0, const double* __restrict__ G1,
                                     const double* __restrict__ G2, double* part) {
  __shared__ double sh[32];
  double ip = 0.0, kk = 0.0;
  const int64_t stride = (int64_t)gridDim.x * blockDim.x;
  for (int64_t t = (int64_t)blockIdx.x * blockDim.x + threadIdx.x; t < n * r; t += stride) {
    const int64_t i = t / r, a = t - i * r;
    ip = fma(A[t], Mt[a * n + i], ip);
  }
  for (int64_t t = (int64_t)blockIdx.x * blockDim.x + threadIdx.x; t < r * r; t += stride) kk += G0[t] * G1[t] * G2[t];
  const double s1 = block_sum(ip, sh);
  __syncthreads();
  const double s2 = block_sum(kk, sh);
  if (threadIdx.x == 0) {
    part[blockIdx.x] = s1;
    part[ALS_PARTS + blockIdx.x] = s2;
  }
}

// ALS-skew factors from A1 = [A1_1 A1_2] (n x r) and B1 (n x h):
// A2 = [B1 B1], A3 = [A1_2, -A1_1].
__global__ void k_skew_derive(const double* __restrict__ A1, const double* __restrict__ B1, int64_t n, int64_t h,
                              double* __restrict__ A2, double* __restrict__ A3) {
  for (int64_t t = (int64_t)blockIdx.x * blockDim.x + threadIdx.x; t < n * h; t += (int64_t)gridDim.x * blockDim.x) {
    const int64_t i = t / h, a = t - i * h, r = 2 * h;
    if (A2) A2[i * r + a] = A2[i * r + h + a] = B1[t];
    if (A3) {
      A3[i * r + a] = A1[i * r + h + a];
      A3[i * r + h + a] = -A1[i * r + a];
    }
  }
}

// B1 = mean of the two halves of a fresh A2 update.
__global__ void k_skew_halves(const double* __restrict__ An, int64_t n, int64_t h, double* __restrict__ B1) {
  for (int64_t t = (int64_t)blockIdx.x * blockDim.x + threadIdx.x; t < n * h; t += (int64_t)gridDim.x * blockDim.x) {
    const int64_t i = t / h, a = t - i * h;
    B1[t] = 0.5 * (An[i * 2 * h + a] + An[i * 2 * h + h + a]);
  }
}

// A1 = lambda A1 + (1 - lambda) An.
__global__ void k_momentum(double* __restrict__ A1, const double* __restrict__ An, int64_t cnt, double lambda) {
  for (int64_t t = (int64_t)blockIdx.x * blockDim.x + threadIdx.x; t < cnt; t += (int64_t)gridDim.x * blockDim.x)
    A1[t] = lambda * A1[t] + (1.0 - lambda) * An[t];
}

unsigned grid_for(int64_t cnt) {
  const int64_t b = (cnt + 255) / 256;
  return (unsigned)(b < 1 ? 1 : b > 4096 ? 4096 : b);
}

void als_free_fit(grom_als* s) {
  for (double*& p : s->f)
    if (p) cudaFree(p), p = nullptr;
  for (double*& p : s->gram)
    if (p) cudaFree(p), p = nullptr;
  for (double** p : {&s->anew, &s->b1, &s->mt, &s->h, &s->lt, &s->rdiag, &s->part})
    if (*p) cudaFree(*p), *p = nullptr;
  if (s->solve) cudaFree(s->solve), s->solve = nullptr;
  if (s->k2s) cudaFree(s->k2s), s->k2s = nullptr;
  s->rcap = 0;
  s->k2s_bytes = 0;
}

grom_status als_grow(grom_als* s, int64_t r) {
  // the split-K scratch of the MTTKRP is not monotonic in the rank: size it per fit
  const size_t need = k2_scratch_bytes(k2_plan(s->n, (int)r, s->sm_count));
  if (r <= s->rcap && need > s->k2s_bytes) {
    if (s->k2s) cudaFree(s->k2s);
    s->k2s = nullptr;
    if (cudaMalloc(&s->k2s, need) != cudaSuccess) {
      cudaGetLastError();
      als_free_fit(s);
      return fail(GROM_ERR_OOM, "grom_als_fit: device allocation");
    }
    s->k2s_bytes = need;
  }
  if (r <= s->rcap) return GROM_OK;
  als_free_fit(s);
  const size_t fb = (size_t)(s->n * r) * sizeof(double), gb = (size_t)(r * r) * sizeof(double);
  cudaError_t e = cudaSuccess;
  for (double*& p : s->f)
    if (e == cudaSuccess) e = cudaMalloc(&p, fb);
  for (double*& p : s->gram)
    if (e == cudaSuccess) e = cudaMalloc(&p, gb);
  if (e == cudaSuccess) e = cudaMalloc(&s->anew, fb);
  if (e == cudaSuccess) e = cudaMalloc(&s->b1, fb);
  if (e == cudaSuccess) e = cudaMalloc(&s->mt, fb);
  if (e == cudaSuccess) e = cudaMalloc(&s->h, gb);
  if (e == cudaSuccess) e = cudaMalloc(&s->lt, gb);
  if (e == cudaSuccess) e = cudaMalloc(&s->rdiag, (size_t)r * sizeof(double));
  if (e == cudaSuccess) e = cudaMalloc(&s->part, 2 * ALS_PARTS * sizeof(double));
  if (e == cudaSuccess) e = cudaMalloc(&s->solve, sizeof(AlsSolve));
  if (e == cudaSuccess) e = cudaMalloc(&s->k2s, need);
  if (e != cudaSuccess) {
    cudaGetLastError();
    als_free_fit(s);
    return fail(e == cudaErrorMemoryAllocation ? GROM_ERR_OOM : GROM_ERR_CUDA, "grom_als_fit: device allocation");
  }
  s->k2s_bytes = need;
  s->rcap = r;
  return GROM_OK;
}

// Gram matrix of factor q (on the device).
grom_status gram_of(grom_als* s, int q, int64_t r) {
  const int64_t t = (r + 15) / 16;
  k_gram<<<(unsigned)(t * (t + 1) / 2), dim3(16, 16), 0, s->stream>>>(s->f[q], s->n, r, s->gram[q]);
  GROM_CUDA_TRY(cudaGetLastError());
  return GROM_OK;
}

// MTTKRP of layout m (0, 1, 2) with factors P (middle index) and Q (inner
// index) into s->mt (r x n), enqueued; als_wait collects its time and errors.
grom_status mttkrp(grom_als* s, int m, int fp, int fq, int64_t r) {
  const K2Plan pl = k2_plan(s->n, (int)r, s->sm_count);
  K2Args a{};
  a.fp = s->f[fp];
  a.fq = s->f[fq];
  a.f_stride = r;
  a.batch = (int)r;
  a.c = s->mt;
  a.c_stride = s->n;
  a.scratch = s->k2s;
  a.err = s->err;
  a.ev0 = s->ev0;
  a.ev1 = s->ev1;
  GROM_CUDA_TRY(k2_launch(pl, &s->tmap[m], a, s->stream));
  return GROM_OK;
}

// Waits for the stream; after an MTTKRP its time and the device error word,
// after a solve (ok != nullptr) its times and whether every pivot was positive.
grom_status als_wait(grom_als* s, bool mttkrp_ran, bool* ok) {
  int flags = 0;
  AlsSolve v{};
  GROM_CUDA_TRY(cudaMemcpyAsync(&flags, s->err, sizeof(int), cudaMemcpyDeviceToHost, s->stream));
  if (ok) GROM_CUDA_TRY(cudaMemcpyAsync(&v, s->solve, sizeof(v), cudaMemcpyDeviceToHost, s->stream));
  GROM_CUDA_TRY(cudaStreamSynchronize(s->stream));
  float ms = 0.f;
  if (mttkrp_ran) {
    GROM_CUDA_TRY(cudaEventElapsedTime(&ms, s->ev0, s->ev1));
    s->mttkrp_ms += ms;
    ++s->mttkrp_calls;
  }
  if (flags & DEV_ERR_TIMEOUT) {
    cudaMemset(s->err, 0, sizeof(int));
    return fail(GROM_ERR_TIMEOUT, "grom_als_fit: a device-side wait timed out");
  }
  if (ok) {
    *ok = v.bad == 0;
    s->solve_ms += 1e-6 * ((double)(v.f1 - v.f0) + (double)(v.s1 - v.s0));
  }
  return GROM_OK;
}

// H = Ga o Gb + rel max diag(Ga o Gb) I and its Cholesky factor L (s->h) and
// L^T (s->lt), on stream st.
grom_status factorise(grom_als* s, const double* Ga, const double* Gb, int64_t r, double rel, cudaStream_t st) {
  GROM_CUDA_TRY(cudaMemsetAsync(s->solve, 0, sizeof(AlsSolve), st));
  k_als_normal<<<grid_for(r * r), 256, 0, st>>>(Ga, Gb, r, rel, s->h, s->solve);
  for (int64_t kb = 0; kb < r; kb += CH) {
    k_chol_diag<<<1, 128, 0, st>>>(s->h, r, kb, s->rdiag, &s->solve->bad);
    if (kb + CH < r) {
      const int64_t rows = r - kb - CH, m = (rows + UT - 1) / UT;
      k_chol_panel<<<(unsigned)((rows + 7) / 8), 256, 0, st>>>(s->h, r, kb, s->rdiag);
      k_chol_update<<<(unsigned)(m * (m + 1) / 2), UT * UT, 0, st>>>(s->h, r, kb);
    }
  }
  k_transpose<<<grid_for(r * r), 256, 0, st>>>(s->h, r, s->lt, s->solve);
  GROM_CUDA_TRY(cudaGetLastError());
  return GROM_OK;
}

// dst = M H^-1 (M = s->mt) with the factors in s->h and s->lt.
grom_status triangular_solves(grom_als* s, int64_t r, double* dst) {
  const size_t smem = (size_t)SV_ROWS * r * sizeof(double);
  if (smem > 12 * 1024)
    GROM_CUDA_TRY(cudaFuncSetAttribute(k_als_rowsolve, cudaFuncAttributeMaxDynamicSharedMemorySize, (int)smem));
  k_als_rowsolve<<<(unsigned)((s->n + SV_ROWS - 1) / SV_ROWS), 32 * SV_ROWS * SV_WARPS, smem, s->stream>>>(
      s->h, s->lt, s->rdiag, s->mt, s->n, r, dst, s->solve);
  GROM_CUDA_TRY(cudaGetLastError());
  return GROM_OK;
}

// One least-squares update dst = M H^-1 for mode m with the other modes'
// factors fp, fq: M by MTTKRP (unless s->mt already holds it), H = Ga o Gb +
// ridge max diag(Ga o Gb) I factorised beside it.  If H is numerically
// singular (ALS on a tensor dominated by a few components drives the factor
// columns towards each other), retry with an extra mu max diag I, mu = 1e-12
// growing 100x up to three times.
grom_status ls_update(grom_als* s, int m, int fp, int fq, int64_t r, double ridge, double* dst, bool have_m) {
  const double *Ga = s->gram[fp], *Gb = s->gram[fq];
  grom_status st;
  GROM_CUDA_TRY(cudaEventRecord(s->fork, s->stream));
  GROM_CUDA_TRY(cudaStreamWaitEvent(s->side, s->fork, 0));
  if ((st = factorise(s, Ga, Gb, r, ridge, s->side))) return st;
  GROM_CUDA_TRY(cudaEventRecord(s->join, s->side));
  if (!have_m && (st = mttkrp(s, m, fp, fq, r))) return st;
  GROM_CUDA_TRY(cudaStreamWaitEvent(s->stream, s->join, 0));
  bool ok = false, ran = !have_m;
  double mu = 0.0;
  for (int attempt = 0; attempt < 4 && !ok; ++attempt) {
    if (attempt > 0) {
      mu = mu == 0.0 ? 1e-12 : mu * 100.0;
      if ((st = factorise(s, Ga, Gb, r, ridge + mu, s->stream))) return st;
    }
    if ((st = triangular_solves(s, r, s->anew))) return st;
    if ((st = als_wait(s, ran, &ok))) return st;
    ran = false;
  }
  if (!ok) return fail(GROM_ERR_INVALID_ARG, "grom_als_fit: a Gram matrix is not positive definite");
  if (dst != s->anew)
    GROM_CUDA_TRY(cudaMemcpyAsync(dst, s->anew, (size_t)(s->n * r) * sizeof(double), cudaMemcpyDeviceToDevice, s->stream));
  return GROM_OK;
}

// Relative residual ||X - [[A1, A2, A3]]|| / ||X|| from <X, K> = <A1, M_1>
// (s->mt holds the mode-1 MTTKRP of the current factors) and
// ||K||^2 = sum G1 o G2 o G3.
grom_status residual_of(grom_als* s, int64_t r, double* out) {
  k_als_residual_parts<<<ALS_PARTS, 256, 0, s->stream>>>(s->f[0], s->mt, s->n, r, s->gram[0], s->gram[1], s->gram[2],
                                                        s->part);
  GROM_CUDA_TRY(cudaGetLastError());
  double ph[2 * ALS_PARTS];
  GROM_CUDA_TRY(cudaMemcpyAsync(ph, s->part, sizeof(ph), cudaMemcpyDeviceToHost, s->stream));
  if (const grom_status st = als_wait(s, true, nullptr)) return st;
  double ip = 0.0, kk = 0.0;
  for (int q = 0; q < ALS_PARTS; ++q) {
    ip += ph[q];
    kk += ph[ALS_PARTS + q];
  }
  const double r2 = s->xnorm2 - 2.0 * ip + kk;
  *out = std::sqrt(std::max(r2, 0.0) / s->xnorm2);
  return GROM_OK;
}

grom_status copy(grom_als* s, void* dst, const void* src, size_t bytes) {
  GROM_CUDA_TRY(cudaMemcpyAsync(dst, src, bytes, cudaMemcpyDefault, s->stream));
  GROM_CUDA_TRY(cudaStreamSynchronize(s->stream));
  return GROM_OK;
}

}  // namespace

extern "C" {

grom_status grom_als_create(int32_t n, const double* tensor, void* stream, grom_als** out) {
  if (!tensor || !out || n < 1) return fail(GROM_ERR_INVALID_ARG, "grom_als_create: bad argument");
  *out = nullptr;
  if (n > grom_max_n(GROM_FORM_FULL, GROM_BF16))
    return fail(GROM_ERR_UNSUPPORTED, "grom_als_create: n exceeds the BF16 row limit");
  grom_als* s = new (std::nothrow) grom_als();
  if (!s) return fail(GROM_ERR_OOM, "grom_als_create: host allocation");
  s->n = n;
  s->np = padded_n(n);
  s->stream = static_cast<cudaStream_t>(stream);
  int dev = 0;
  auto bail = [&](grom_status st) {
    grom_als_destroy(s);
    return st;
  };
  if (cudaGetDevice(&dev) != cudaSuccess ||
      cudaDeviceGetAttribute(&s->sm_count, cudaDevAttrMultiProcessorCount, dev) != cudaSuccess) {
    cudaGetLastError();
    return bail(fail(GROM_ERR_CUDA, "grom_als_create: no usable CUDA device"));
  }
  const size_t lbytes = (size_t)n * n * s->np * sizeof(__nv_bfloat16);
  for (auto& x : s->x) {
    if (cudaMalloc(&x, lbytes) != cudaSuccess || cudaMemsetAsync(x, 0, lbytes, s->stream) != cudaSuccess) {
      cudaGetLastError();
      return bail(fail(GROM_ERR_OOM, "grom_als_create: device allocation"));
    }
  }
  if (cudaMalloc(&s->err, sizeof(int)) != cudaSuccess || cudaMemsetAsync(s->err, 0, sizeof(int), s->stream) != cudaSuccess)
    return bail(fail(GROM_ERR_OOM, "grom_als_create: device allocation"));
  if (cudaEventCreate(&s->ev0) != cudaSuccess || cudaEventCreate(&s->ev1) != cudaSuccess ||
      cudaEventCreateWithFlags(&s->fork, cudaEventDisableTiming) != cudaSuccess ||
      cudaEventCreateWithFlags(&s->join, cudaEventDisableTiming) != cudaSuccess ||
      cudaStreamCreateWithFlags(&s->side, cudaStreamNonBlocking) != cudaSuccess)
    return bail(cuda_fail(cudaGetLastError(), "grom_als_create: events"));
  // stream the FP64 tensor through a staging buffer by test index
  const int64_t per_i = (int64_t)n * n;
  const int64_t si = std::min<int64_t>(n, std::max<int64_t>(1, (int64_t)(256ll << 20) / (per_i * 8)));
  double *stage = nullptr, *part = nullptr;
  constexpr int NB = 1024;
  if (cudaMalloc(&stage, (size_t)(si * per_i * 8)) != cudaSuccess || cudaMalloc(&part, NB * sizeof(double)) != cudaSuccess) {
    cudaGetLastError();
    if (stage) cudaFree(stage);
    return bail(fail(GROM_ERR_OOM, "grom_als_create: staging allocation"));
  }
  std::vector<double> ph(NB);
  double norm2 = 0.0;
  cudaError_t e = cudaSuccess;
  for (int64_t a = 0; e == cudaSuccess && a < n; a += si) {
    const int64_t cnt = std::min(si, (int64_t)n - a);
    e = cudaMemcpyAsync(stage, tensor + a * per_i, (size_t)(cnt * per_i * 8), cudaMemcpyDefault, s->stream);
    if (e != cudaSuccess) break;
    int64_t blocks = std::min<int64_t>(65536, (cnt * per_i + 255) / 256);
    k_als_x12<<<(unsigned)blocks, 256, 0, s->stream>>>(stage, cnt, n, s->np, a, reinterpret_cast<__nv_bfloat16*>(s->x[0]),
                                                       reinterpret_cast<__nv_bfloat16*>(s->x[1]));
    dim3 g3((unsigned)((n + 31) / 32), (unsigned)((n + 31) / 32), (unsigned)cnt);
    k_als_x3<<<g3, dim3(32, 8), 0, s->stream>>>(stage, n, s->np, a, reinterpret_cast<__nv_bfloat16*>(s->x[2]));
    k_als_norm<<<NB, 256, 0, s->stream>>>(stage, cnt * per_i, part);
    e = cudaGetLastError();
    if (e == cudaSuccess) e = cudaMemcpyAsync(ph.data(), part, NB * sizeof(double), cudaMemcpyDeviceToHost, s->stream);
    if (e == cudaSuccess) e = cudaStreamSynchronize(s->stream);
    for (int q = 0; q < NB; ++q) norm2 += ph[q];
  }
  cudaFree(stage);
  cudaFree(part);
  if (e != cudaSuccess) return bail(cuda_fail(e, "grom_als_create: tensor upload"));
  s->xnorm2 = norm2;
  for (int q = 0; q < 3; ++q)
    if (!k2_make_tmap(&s->tmap[q], s->x[q], n, s->np))
      return bail(fail(GROM_ERR_UNSUPPORTED, "grom_als_create: tensor map encoding failed"));
  *out = s;
  return GROM_OK;
}

grom_status grom_als_fit(grom_als* s, int32_t rank, int32_t method, int32_t iters, double lambda, int32_t subiters,
                         double ridge, double* fa, double* fb, double* fc, double* residual) {
  TraceRange trace("grom_als_fit");
  if (!s || !fa || !fb || rank < 1 || iters < 0 || !(ridge >= 0.0))
    return fail(GROM_ERR_INVALID_ARG, "grom_als_fit: bad argument");
  if (method != GROM_ALS_PLAIN && method != GROM_ALS_SKEW) return fail(GROM_ERR_INVALID_ARG, "grom_als_fit: bad method");
  if (method == GROM_ALS_PLAIN && !fc) return fail(GROM_ERR_INVALID_ARG, "grom_als_fit: fc is NULL");
  if (method == GROM_ALS_SKEW && (rank % 2 || subiters < 1 || !(lambda >= 0.0 && lambda < 1.0)))
    return fail(GROM_ERR_INVALID_ARG, "grom_als_fit: ALS-skew needs an even rank, subiters >= 1, 0 <= lambda < 1");
  const int64_t n = s->n, r = rank, h = r / 2;
  grom_status st = als_grow(s, r);
  if (st) return st;
  const size_t fbytes = (size_t)(n * r) * sizeof(double);
  if (method == GROM_ALS_PLAIN) {
    if ((st = copy(s, s->f[0], fa, fbytes)) || (st = copy(s, s->f[1], fb, fbytes)) ||
        (st = copy(s, s->f[2], fc, fbytes)))
      return st;
    for (int q = 0; q < 3; ++q)
      if ((st = gram_of(s, q, r))) return st;
    for (int it = 0; it < iters; ++it) {
      for (int m = 0; m < 3; ++m) {
        // layout m: rows of mode m; P, Q = the factors of its middle and inner index
        const int fp = m == 0 ? 1 : 0, fq = m == 2 ? 1 : 2;
        // the residual's MTTKRP of the last iteration is this iteration's first
        const bool have_m = m == 0 && it > 0 && residual;
        if ((st = ls_update(s, m, fp, fq, r, ridge, s->f[m], have_m)) || (st = gram_of(s, m, r))) return st;
      }
      // <X, K> from a fresh mode-1 MTTKRP with the final factors: the M the
      // last update used carries the noise that update amplified along the
      // near-null directions of its normal matrix, and would hide it
      if (residual && ((st = mttkrp(s, 0, 1, 2, r)) || (st = residual_of(s, r, &residual[it])))) return st;
    }
    if ((st = copy(s, fa, s->f[0], fbytes)) || (st = copy(s, fb, s->f[1], fbytes)) || (st = copy(s, fc, s->f[2], fbytes)))
      return st;
    return GROM_OK;
  }
  // ALS-skew: A1 = [A1_1 A1_2] (factor 0), A2 = [B1 B1], A3 = [A1_2, -A1_1]
  const unsigned gh = grid_for(n * h);
  if ((st = copy(s, s->f[0], fa, fbytes)) || (st = copy(s, s->b1, fb, (size_t)(n * h) * sizeof(double)))) return st;
  k_skew_derive<<<gh, 256, 0, s->stream>>>(s->f[0], s->b1, n, h, s->f[1], s->f[2]);
  GROM_CUDA_TRY(cudaGetLastError());
  for (int q = 0; q < 3; ++q)
    if ((st = gram_of(s, q, r))) return st;
  for (int it = 0; it < iters; ++it) {
    // A2 as in ALS (layout X2: P = A1, Q = A3), halves averaged
    if ((st = ls_update(s, 1, 0, 2, r, ridge, s->anew, false))) return st;
    k_skew_halves<<<gh, 256, 0, s->stream>>>(s->anew, n, h, s->b1);
    k_skew_derive<<<gh, 256, 0, s->stream>>>(s->f[0], s->b1, n, h, s->f[1], nullptr);
    GROM_CUDA_TRY(cudaGetLastError());
    if ((st = gram_of(s, 1, r))) return st;
    for (int sub = 0; sub < subiters; ++sub) {
      // A1_next with A2, A3 fixed (layout X1: P = A2, Q = A3), then momentum
      if ((st = ls_update(s, 0, 1, 2, r, ridge, s->anew, false))) return st;
      k_momentum<<<grid_for(n * r), 256, 0, s->stream>>>(s->f[0], s->anew, n * r, lambda);
      k_skew_derive<<<gh, 256, 0, s->stream>>>(s->f[0], s->b1, n, h, nullptr, s->f[2]);
      GROM_CUDA_TRY(cudaGetLastError());
      if ((st = gram_of(s, 0, r)) || (st = gram_of(s, 2, r))) return st;
    }
    if (residual && ((st = mttkrp(s, 0, 1, 2, r)) || (st = residual_of(s, r, &residual[it])))) return st;
  }
  if ((st = copy(s, fa, s->f[0], fbytes)) || (st = copy(s, fb, s->b1, (size_t)(n * h) * sizeof(double)))) return st;
  return GROM_OK;
}

grom_status grom_als_stats(grom_als* s, double* mttkrp_ms, int64_t* mttkrp_calls, double* solve_ms) {
  if (!s || !mttkrp_ms || !mttkrp_calls || !solve_ms) return fail(GROM_ERR_INVALID_ARG, "grom_als_stats: null argument");
  *mttkrp_ms = s->mttkrp_ms;
  *mttkrp_calls = s->mttkrp_calls;
  *solve_ms = s->solve_ms;
  s->mttkrp_ms = s->solve_ms = 0.0;
  s->mttkrp_calls = 0;
  return GROM_OK;
}

grom_status grom_als_destroy(grom_als* s) {
  if (!s) return GROM_OK;
  if (s->side) cudaStreamSynchronize(s->side);
  if (s->stream) cudaStreamSynchronize(s->stream);
  for (cudaEvent_t e : {s->ev0, s->ev1, s->fork, s->join})
    if (e) cudaEventDestroy(e);
  if (s->side) cudaStreamDestroy(s->side);
  for (auto p : s->x)
    if (p) cudaFree(p);
  als_free_fit(s);
  if (s->err) cudaFree(s->err);
  delete s;
  return GROM_OK;
}

}  // extern "C"
