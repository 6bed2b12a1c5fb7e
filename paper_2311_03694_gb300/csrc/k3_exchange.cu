// Persistent CPD-ROM stepper for one to four trajectories (F64: one or two)
// whose factors fit the shared memory of the chip twice over: every step of a
// grom_step call in one cooperative launch, without grid barriers.
//
// CTA g keeps its rank columns of the projected factors and its rows of the
// expansion factors in shared memory.  A step:
//   1  u^l of every test index, in the factors' arithmetic;
//   2  a warp per owned column: p = V^T u, q = W^T u (s = U^T u), and the
//      Hadamard products h1 = p o q (h2 = p o s), published;
//   3  h1, h2 of every column;
//   4  a warp per owned row: c_i = sum_r U_ir h1_r - W_ir h2_r and the diagonal
//      BDFk/EXTk step of the row; u^{l+1}_i is published.
// What bounds a step is not the arithmetic (some 5 n r multiply-adds over the
// whole chip) but the two exchanges.  A published value is an eight-byte word
// (value, step number), stored and loaded as one: a CTA polls the words it
// needs, so that an exchange costs one store and one load through L2 where a
// grid barrier took a fence, an atomic, a poll and then the loads, and rows
// need no sums over the CTAs' partial results.  No word is overwritten before
// it has been read: u^{l+1} is published after its CTA has read every h of step l,
// and h of step l + 1 needs every u^{l+1}.  The step numbers go on from launch
// to launch (the base word), so what an earlier call left never matches.
// n = r = 1024 BF16, one trajectory: 6.4 us a step against 15.5 with two
// barriers and partial sums (k3_persistent.cu, which keeps the larger ROMs);
// n = r = 512 F64: 12.4 against 20.0; n = 256 F64, two trajectories: 14.2
// against 40.1.  Of the 6.4 us the exchanges take 3.0 and the dependent
// arithmetic (FP64 operations some 70 cycles apart) most of the rest.
// The sums of FP32 products are carried in three floats (ts_add) across
// vectors and lanes, in place of the FP64 sums over the CTAs' partials.
#include <algorithm>

#include "ds_arith.cuh"
#include "cp_async.cuh"
#include "grom_internal.h"
#include "ptx.cuh"
#include "step_elem.cuh"

namespace grom {

constexpr int KX_THREADS = 256;
constexpr int KX_WARPS = KX_THREADS / 32;

template <int ST>
struct KXT;  // acc_t; EV elements of a 16-byte vector; WORDS a published value takes
template <>
struct KXT<GROM_F64> {
  using acc_t = double;
  using el = double;
  static constexpr int EV = 2, WORDS = 2;
  static __device__ __forceinline__ void load(const el* p, double (&x)[EV]) {
    const double2 v = *reinterpret_cast<const double2*>(p);
    x[0] = v.x;
    x[1] = v.y;
  }
};
template <>
struct KXT<GROM_F32> {
  using acc_t = float;
  using el = float;
  static constexpr int EV = 4, WORDS = 1;
  static __device__ __forceinline__ void load(const el* p, float (&x)[EV]) {
    const float4 v = *reinterpret_cast<const float4*>(p);
    x[0] = v.x;
    x[1] = v.y;
    x[2] = v.z;
    x[3] = v.w;
  }
};
template <>
struct KXT<GROM_BF16> {
  using acc_t = float;
  using el = uint16_t;
  static constexpr int EV = 8, WORDS = 1;
  static __device__ __forceinline__ void load(const el* p, float (&x)[EV]) {
    const uint4 v = *reinterpret_cast<const uint4*>(p);
    const uint32_t w[4] = {v.x, v.y, v.z, v.w};
#pragma unroll
    for (int q = 0; q < 4; ++q) {
      x[2 * q] = __uint_as_float(w[q] << 16);
      x[2 * q + 1] = __uint_as_float(w[q] & 0xffff0000u);
    }
  }
};

// Place of element i of a padded vector in shared memory: the 16-byte pieces
// that a lane reads for one vector of factors lie pad / H apart, so that the
// lanes of a piece are contiguous.
template <int ST>
__device__ __forceinline__ int kx_pos(int i, int pad) {
  if constexpr (ST == GROM_BF16) return ((i >> 2) & 1) * (pad / 2) + (i >> 3) * 4 + (i & 3);
  return i;
}
// The EV values that go with the factors' vector at element v.
template <int ST>
__device__ __forceinline__ void kx_vec(const typename KXT<ST>::acc_t* a, int v, int pad,
                                       typename KXT<ST>::acc_t (&x)[KXT<ST>::EV]) {
  if constexpr (ST == GROM_F64) {
    const double2 t = *reinterpret_cast<const double2*>(a + v);
    x[0] = t.x;
    x[1] = t.y;
  } else {
#pragma unroll
    for (int h = 0; h < KXT<ST>::EV / 4; ++h) {
      const float4 t = *reinterpret_cast<const float4*>(a + h * (pad / 2) + v / (KXT<ST>::EV / 4));
      x[4 * h] = t.x;
      x[4 * h + 1] = t.y;
      x[4 * h + 2] = t.z;
      x[4 * h + 3] = t.w;
    }
  }
}

struct KXArgs {
  const uint8_t *fa, *fb, *fc;  // stored factors, n x rp
  int nf;                       // 3 skew, 2 general
  int n, rp, npad, rpad;        // padded to 32 vectors
  int cols, rows;               // most columns and rows of a CTA
  int batch, nsteps;
  unsigned int* base;           // step number of the last word published
  unsigned long long* uw;       // WORDS x NB x n
  unsigned long long* hw;       // WORDS x 2 x NB x rp
  unsigned long long* rw;       // 2 (step parity) x grid x NB x 4: energy and invariant partials
  StepArgs st;
};

__device__ __forceinline__ void kx_store(unsigned long long* w, uint32_t bits, uint32_t tag) {
  asm volatile("st.relaxed.gpu.global.u64 [%0], %1;" ::"l"(w), "l"((unsigned long long)tag << 32 | bits) : "memory");
}
__device__ __forceinline__ unsigned long long kx_load(const unsigned long long* w) {
  unsigned long long v;
  asm volatile("ld.relaxed.gpu.global.u64 %0, [%1];" : "=l"(v) : "l"(w) : "memory");
  return v;
}
// Value x as word(s) `plane` words apart.
__device__ __forceinline__ void kx_publish(unsigned long long* w, int64_t, float x, uint32_t tag) {
  kx_store(w, __float_as_uint(x), tag);
}
__device__ __forceinline__ void kx_publish(unsigned long long* w, int64_t plane, double x, uint32_t tag) {
  kx_store(w, (uint32_t)__double2loint(x), tag);
  kx_store(w + plane, (uint32_t)__double2hiint(x), tag);
}

// Waits for the words t, t + stride, ... < count to carry `tag` and hands
// each value on; false after the time limit (or another thread's).  SPREAD:
// the threads of a CTA share the words, and a warp waits for one of its words
// before it asks for them all: what every CTA polls lies in a few lines, whose
// slices of the L2 the failed rounds of 128 CTAs kept busy (8.7K cycles for
// the 2048 words of n = r = 1024, 4.2K this way).
template <bool SPREAD, typename F>
__device__ __forceinline__ bool kx_poll(const unsigned long long* w, int count, uint32_t tag, int t, int stride,
                                        volatile int* abort_flag, F take) {
  constexpr int B = 8;  // words in flight: every round loads all that are missing
  for (int i0 = t; i0 < count; i0 += B * stride) {
    uint32_t missing = 0;
#pragma unroll
    for (int k = 0; k < B; ++k)
      if (i0 + k * stride < count) missing |= 1u << k;
    uint64_t t0 = 0;
    if constexpr (SPREAD) {
      const int x = i0 & ~31;  // the warp's first word: one address, one request
      for (uint32_t spin = 0; (uint32_t)(kx_load(w + x) >> 32) != tag; ++spin)
        if ((spin & 63u) == 63u) {
          const uint64_t now = ptx::globaltimer();
          if (t0 == 0) t0 = now;
          if (*abort_flag || now - t0 > ptx::WAIT_LIMIT_NS) return false;
        }
    }
    for (uint32_t spin = 0; missing; ++spin) {
      unsigned long long v[B];
#pragma unroll
      for (int k = 0; k < B; ++k)
        if (missing >> k & 1u) v[k] = kx_load(w + i0 + k * stride);
#pragma unroll
      for (int k = 0; k < B; ++k)
        if ((missing >> k & 1u) && (uint32_t)(v[k] >> 32) == tag) {
          missing &= ~(1u << k);
          take(i0 + k * stride, (uint32_t)v[k]);
        }
      if ((spin & 63u) == 63u && missing) {
        const uint64_t now = ptx::globaltimer();
        if (t0 == 0) t0 = now;
        if (*abort_flag || now - t0 > ptx::WAIT_LIMIT_NS) return false;
      }
    }
  }
  return true;
}

// A wait that ran out.  The base goes on as after a whole launch, so that the
// words this one did publish are not taken for a later launch's.
__device__ __forceinline__ void kx_abort(volatile int* abort_flag, int* err, unsigned int* base, uint32_t next) {
  *abort_flag = 1;
  *reinterpret_cast<volatile unsigned int*>(base) = next;
  atomicOr(err, DEV_ERR_TIMEOUT);
}

template <int ST, int NB>
__global__ void __launch_bounds__(KX_THREADS, 1) k3x_kernel(const KXArgs p) {
  using T = KXT<ST>;
  using acc_t = typename T::acc_t;
  using el = typename T::el;
  constexpr int EV = T::EV;
  constexpr bool F64 = ST == GROM_F64;
  extern __shared__ __align__(16) uint8_t kx_smem[];
  __shared__ int abort_sh;
  __shared__ double se[2][KX_WARPS][NB];
  const int tid = threadIdx.x, warp = tid >> 5, lane = tid & 31;
  const int G = gridDim.x, g = blockIdx.x;
  const int n = p.n, rp = p.rp, npad = p.npad, rpad = p.rpad;
  const StepArgs& st = p.st;
  const int r0 = (int)((int64_t)g * rp / G), rb = (int)((int64_t)(g + 1) * rp / G) - r0;
  const int i0 = (int)((int64_t)g * n / G), ni = (int)((int64_t)(g + 1) * n / G) - i0;
  const bool skew = p.nf == 3;
  volatile int* abort_flag = &abort_sh;
  // [factor columns nf x cols x npad][expansion rows 2 x rows x rpad][u: NB x npad][h: 2 x NB x rpad]
  // [history NB x rows x 6][K: NB x rows]
  el* colf = reinterpret_cast<el*>(kx_smem);
  el* rowe = colf + (size_t)p.nf * p.cols * npad;
  acc_t* us = reinterpret_cast<acc_t*>(rowe + (size_t)(p.nf - 1) * p.rows * rpad);
  acc_t* hs = us + (size_t)NB * npad;
  double* hist = reinterpret_cast<double*>(hs + (size_t)2 * NB * rpad);  // u^l, u^l-1, u^l-2, n^l, n^l-1, n^l-2
  double* kk = hist + (size_t)NB * p.rows * 6;

  if (tid == 0) abort_sh = 0;
  const uint32_t tag0 = *reinterpret_cast<volatile unsigned int*>(p.base);
  {
    // zeros first (padding), then the columns eight loads at a time, the rows in 16-byte pieces
    uint4* z = reinterpret_cast<uint4*>(kx_smem);
    const int nz = (int)(reinterpret_cast<uint8_t*>(us) - kx_smem) / 16;
    for (int t = tid; t < nz; t += KX_THREADS) z[t] = make_uint4(0, 0, 0, 0);
    __syncthreads();
    const el* F[3] = {reinterpret_cast<const el*>(p.fb), reinterpret_cast<const el*>(p.fc),
                      reinterpret_cast<const el*>(p.fa)};
    for (int f = 0; f < p.nf; ++f)
      for (int ib = tid; ib < n; ib += KX_THREADS) {  // a thread per row of the factor
        const el* src = F[f] + (int64_t)ib * rp + r0;
        el* dst = colf + (size_t)f * p.cols * npad + ib;
        for (int c = 0; c < rb; c += 8) {
          el x[8];
#pragma unroll
          for (int k = 0; k < 8; ++k)
            if (c + k < rb) x[k] = src[c + k];
#pragma unroll
          for (int k = 0; k < 8; ++k)
            if (c + k < rb) dst[(size_t)(c + k) * npad] = x[k];
        }
      }
    const el* E[2] = {reinterpret_cast<const el*>(p.fa), reinterpret_cast<const el*>(p.fc)};
    const int pieces = rp * (int)sizeof(el) / 16;  // rp is a multiple of 8: whole pieces
    for (int e = 0; e < p.nf - 1; ++e)
      for (int t = tid; t < ni * pieces; t += KX_THREADS) {
        const int ri = t / pieces, q = t - ri * pieces;
        reinterpret_cast<uint4*>(rowe + ((size_t)e * p.rows + ri) * rpad)[q] =
            reinterpret_cast<const uint4*>(E[e] + (int64_t)(i0 + ri) * rp)[q];
      }
    for (int t = tid; t < 2 * NB * rpad; t += KX_THREADS) hs[t] = acc_t(0);
    for (int t = tid; t < NB * npad; t += KX_THREADS) us[t] = acc_t(0);
  }
  int64_t l0[NB];
#pragma unroll
  for (int b = 0; b < NB; ++b) l0[b] = b < p.batch ? st.taken[b] : 0;
  for (int t = tid; t < NB * ni * 6; t += KX_THREADS) {
    const int q = t % 6, ri = t / 6 % ni, b = t / (6 * ni);
    double v = 0.0;
    if (b < p.batch) {
      const int64_t l = st.taken[b], m = ((l - (q % 3)) % 3 + 3) % 3;
      v = st.hist[b * st.hist_stride + ((q < 3 ? 0 : 3) + m) * n + i0 + ri];
    }
    hist[((size_t)b * p.rows + ri) * 6 + q] = v;
  }
  __syncthreads();
  // K of a row: all of the step's terms but the new advection term's,
  // u^{l+1} = -(alpha_1 c + K) / H_k, formed while the words travel
  auto form_k = [&](int b, int ri, int64_t l) {
    const int k = (int)(l + 1 < st.order ? l + 1 : st.order);
    const double* h = hist + ((size_t)b * p.rows + ri) * 6;
    const int i = i0 + ri;
    double K = 0.0, bdf = st.bdt[k - 1][0] * h[0];
    if (k >= 2) bdf = fma(st.bdt[k - 1][1], h[1], bdf);
    if (k == 3) bdf = fma(st.bdt[2][2], h[2], bdf);
    if (st.lin_diag || st.forcing) {
      const double ld = st.lin_diag ? st.lin_diag[i] : 0.0, f = st.forcing ? st.forcing[i] : 0.0;
      for (int q = 0; q < k; ++q) K = fma(c_alpha[k - 1][q], fma(ld, h[q], f), K);
    }
    if (k == 2) K -= h[4];
    if (k == 3) K += fma(-3.0, h[4], h[5]);
    kk[(size_t)b * p.rows + ri] = st.mass_diag ? fma(st.mass_diag[i], bdf, K) : K + bdf;
  };
  const bool sums = st.energy || st.invariant;
  // rows of this warp: warp, warp + 8, ...; lane b < NB steps trajectory b
  if (lane < NB && lane < p.batch)
    for (int ri = warp; ri < ni; ri += KX_WARPS) form_k(lane, ri, l0[lane]);

  // the energy / invariant of step s: warp b of CTA 0 adds the CTAs' partials
  // of trajectory b (lane q those of CTAs q, q + 32, ... in order)
  auto close_sums = [&](int s) {
    if (g != 0 || warp >= NB || warp >= p.batch) return;
    double e = 0.0, v = 0.0;
    const unsigned long long* w = p.rw + ((size_t)(s & 1) * G * NB + warp) * 4;
    for (int q = lane; q < G; q += 32) {
      uint32_t x[4];
      if (!kx_poll<false>(w + (size_t)q * NB * 4, 4, tag0 + 1u + (uint32_t)s, 0, 1, abort_flag,
                   [&](int k, uint32_t bits) { x[k] = bits; })) {
        kx_abort(abort_flag, st.err, p.base, tag0 + 1u + (uint32_t)p.nsteps);
        break;
      }
      e += __hiloint2double((int)x[1], (int)x[0]);
      v += __hiloint2double((int)x[3], (int)x[2]);
    }
    __syncwarp();
#pragma unroll
    for (int off = 16; off > 0; off >>= 1) {
      e += __shfl_xor_sync(0xffffffffu, e, off);
      v += __shfl_xor_sync(0xffffffffu, v, off);
    }
    if (lane == 0) {
      if (st.energy) st.energy[(int64_t)s * st.batch + warp] = 0.5 * e;
      if (st.invariant) st.invariant[(int64_t)s * st.batch + warp] = v;
    }
  };

  for (int s = 0; s < p.nsteps; ++s) {
    const uint32_t tag = tag0 + 1u + (uint32_t)s;
    if (sums && s > 0) close_sums(s - 1);
    // ---- 1: u^l
    bool ok = true;
    if (s == 0) {
      for (int t = tid; t < p.batch * n; t += KX_THREADS) {
        const int b = t / n, i = t - b * n;
        const double v = st.hist[b * st.hist_stride + (l0[b] % 3) * n + i];
        if constexpr (F64)
          us[b * npad + i] = v;
        else
          us[b * npad + kx_pos<ST>(i, npad)] = d2f_int(v);
      }
    } else if (rb > 0) {  // without a column the words may be overwritten before they are read
      ok = kx_poll<true>(p.uw, T::WORDS * p.batch * n, tag, tid, KX_THREADS, abort_flag, [&](int x, uint32_t bits) {
        const int half = F64 ? x / (p.batch * n) : 0, y = F64 ? x - half * p.batch * n : x;
        const int b = NB == 1 ? 0 : y / n, i = y - b * n;
        reinterpret_cast<uint32_t*>(us)[(size_t)T::WORDS * (b * npad + kx_pos<ST>(i, npad)) + half] = bits;
      });
    }
    if (!ok) kx_abort(abort_flag, st.err, p.base, tag0 + 1u + (uint32_t)p.nsteps);
    if (__syncthreads_or(*abort_flag)) return;
    // ---- 2: projections of the owned columns
    for (int c = warp; c < rb; c += KX_WARPS) {
      acc_t acc[3][NB];
#pragma unroll
      for (int f = 0; f < 3; ++f)
#pragma unroll
        for (int b = 0; b < NB; ++b) acc[f][b] = acc_t(0);
#pragma unroll 2
      for (int v = lane * EV; v < npad; v += 32 * EV) {
        acc_t x[3][EV];
        T::load(colf + (size_t)c * npad + v, x[0]);
        T::load(colf + (size_t)(p.cols + c) * npad + v, x[1]);
        if (skew) T::load(colf + (size_t)(2 * p.cols + c) * npad + v, x[2]);
#pragma unroll
        for (int b = 0; b < NB; ++b) {
          acc_t u[EV];
          kx_vec<ST>(us + b * npad, v, npad, u);
#pragma unroll
          for (int e = 0; e < EV; ++e) {
            acc[0][b] = fma(x[0][e], u[e], acc[0][b]);
            acc[1][b] = fma(x[1][e], u[e], acc[1][b]);
            if (skew) acc[2][b] = fma(x[2][e], u[e], acc[2][b]);
          }
        }
      }
#pragma unroll
      for (int off = 16; off > 0; off >>= 1)
#pragma unroll
        for (int f = 0; f < 3; ++f)
#pragma unroll
          for (int b = 0; b < NB; ++b) acc[f][b] += __shfl_xor_sync(0xffffffffu, acc[f][b], off);
#pragma unroll
      for (int b = 0; b < NB; ++b) {
        if (b >= p.batch) break;
        const int64_t plane = (int64_t)2 * p.batch * rp;
        if (lane == 0) kx_publish(p.hw + (int64_t)b * rp + r0 + c, plane, acc[0][b] * acc[1][b], tag);
        if (lane == 1 && skew)
          kx_publish(p.hw + (int64_t)(p.batch + b) * rp + r0 + c, plane, acc[0][b] * acc[2][b], tag);
      }
    }
    // ---- 3: h of every column
    if (ni > 0) {
      const int per = (skew ? 2 : 1) * p.batch * rp, plane = 2 * p.batch * rp;
#pragma unroll
      for (int half = 0; half < T::WORDS; ++half)
        ok = ok && kx_poll<true>(p.hw + (size_t)half * plane, per, tag, tid, KX_THREADS, abort_flag,
                           [&](int x, uint32_t bits) {
                             const int row = x / rp, r = x - row * rp;  // row: which * batch + b
                             const int which = row >= p.batch ? 1 : 0, b = row - which * p.batch;
                             reinterpret_cast<uint32_t*>(
                                 hs)[(size_t)T::WORDS * ((which * NB + b) * rpad + kx_pos<ST>(r, rpad)) + half] = bits;
                           });
    }
    if (!ok) kx_abort(abort_flag, st.err, p.base, tag0 + 1u + (uint32_t)p.nsteps);
    if (__syncthreads_or(*abort_flag)) return;
    // ---- 4: the owned rows
    double e_acc = 0.0, i_acc = 0.0;
    for (int ri = warp; ri < ni; ri += KX_WARPS) {
      double ch = 0.0, cl = 0.0;  // lane b: c of trajectory b as two parts
      acc_t s1[NB], s2[NB], s3[NB];
#pragma unroll
      for (int b = 0; b < NB; ++b) s1[b] = s2[b] = s3[b] = acc_t(0);
#pragma unroll 2
      for (int v = lane * EV; v < rpad; v += 32 * EV) {
        acc_t x[EV], w[EV];
        T::load(rowe + (size_t)ri * rpad + v, x);
        if (skew) T::load(rowe + (size_t)(p.rows + ri) * rpad + v, w);
#pragma unroll
        for (int b = 0; b < NB; ++b) {
          acc_t t0 = F64 ? s1[b] : acc_t(0), t1 = F64 ? s2[b] : acc_t(0), h1[EV], h2[EV];  // two chains
          kx_vec<ST>(hs + b * rpad, v, rpad, h1);
          if (skew) kx_vec<ST>(hs + (NB + b) * rpad, v, rpad, h2);
#pragma unroll
          for (int e = 0; e < EV; e += 2) {
            t0 = fma(x[e], h1[e], t0);
            t1 = fma(x[e + 1], h1[e + 1], t1);
            if (skew) {
              t0 = fma(-w[e], h2[e], t0);
              t1 = fma(-w[e + 1], h2[e + 1], t1);
            }
          }
          if constexpr (F64) {
            s1[b] = t0;
            s2[b] = t1;
          } else {
            ts_add(t0 + t1, s1[b], s2[b], s3[b]);
          }
        }
      }
#pragma unroll
      for (int b = 0; b < NB; ++b) {
        double hi, lo = 0.0;
        if constexpr (F64) {
          hi = s1[b] + s2[b];
#pragma unroll
          for (int off = 16; off > 0; off >>= 1) hi += __shfl_xor_sync(0xffffffffu, hi, off);
        } else {
#pragma unroll
          for (int off = 16; off > 0; off >>= 1) {
            const float x1 = __shfl_xor_sync(0xffffffffu, s1[b], off), x2 = __shfl_xor_sync(0xffffffffu, s2[b], off);
            const float x3 = __shfl_xor_sync(0xffffffffu, s3[b], off);
            ts_add(x1, s1[b], s2[b], s3[b]);
            ts_add(x2, s1[b], s2[b], s3[b]);
            s3[b] += x3;
          }
          hi = f2d_int(s1[b]);
          lo = f2d_int(s2[b]) + f2d_int(s3[b]);
        }
        if (lane == b) {
          ch = hi;
          cl = lo;
        }
      }
      if (lane < NB && lane < p.batch) {
        const int b = lane, i = i0 + ri;
        int64_t l = s;
#pragma unroll
        for (int q = 0; q < NB; ++q)
          if (q == b) l += l0[q];
        const int k = (int)(l + 1 < st.order ? l + 1 : st.order);
        double y = fma((double)k, ch, kk[(size_t)b * p.rows + ri]);  // alpha_1 = k
        if constexpr (!F64) y = fma((double)k, cl, y);
        const double un = -y * st.hdiag[k - 1][i];
        if constexpr (F64)
          kx_publish(p.uw + (int64_t)b * n + i, (int64_t)p.batch * n, un, tag + 1u);
        else
          kx_publish(p.uw + (int64_t)b * n + i, 0, d2f_int(un), tag + 1u);
        if (step_is_bad(un)) {
          atomicOr(st.err, DEV_ERR_NONFINITE);
          atomicMin(st.first_bad, b);
        }
        double* h = hist + ((size_t)b * p.rows + ri) * 6;
        const double cv = ch + cl;
        if (sums) {
          const double mb = st.mass_diag ? st.mass_diag[i] : 1.0;
          e_acc += mb * un * un;
          i_acc += h[0] * cv;
        }
        h[2] = h[1];
        h[1] = h[0];
        h[0] = un;
        h[5] = h[4];
        h[4] = cv;
        form_k(b, ri, l + 1);
      }
    }
    if (sums) {
      if (lane < NB) {
        se[0][warp][lane] = e_acc;
        se[1][warp][lane] = i_acc;
      }
      __syncthreads();
      if (tid < NB && tid < p.batch) {
        double e = 0.0, v = 0.0;
        for (int w = 0; w < KX_WARPS; ++w) {
          e += se[0][w][tid];
          v += se[1][w][tid];
        }
        unsigned long long* w = p.rw + ((size_t)(s & 1) * G * NB + (size_t)g * NB + tid) * 4;
        kx_publish(w, 1, e, tag);
        kx_publish(w + 2, 1, v, tag);
      }
      __syncthreads();
    }
  }
  if (sums) close_sums(p.nsteps - 1);
  // the owned rows' history back into the ring (n^l of the newest state is
  // not known yet; its slot keeps the last n)
  __syncthreads();
  for (int t = tid; t < NB * ni * 6; t += KX_THREADS) {
    const int q = t % 6, ri = t / 6 % ni, b = t / (6 * ni);
    if (b >= p.batch || q == 3) continue;
    const int64_t l = l0[b] + p.nsteps, m = ((l - (q % 3)) % 3 + 3) % 3;
    st.hist[b * st.hist_stride + ((q < 3 ? 0 : 3) + m) * n + i0 + ri] = hist[((size_t)b * p.rows + ri) * 6 + q];
  }
  if (g == 0 && !*abort_flag) {
    if (tid < NB && tid < p.batch) st.taken[tid] = l0[tid] + p.nsteps;
    if (tid == 0) *p.base = tag0 + 1u + (uint32_t)p.nsteps;
  }
}

// ------------------------------------------------------------- evaluations
// One evaluation of FP64 factors with the same exchange: the CTAs' columns
// straight from memory (a thread takes the CTA's entries of every 256th row of
// a factor; the rows of the expansion are copied to shared memory meanwhile), h published,
// then the CTAs' rows.  The two kernels of k3_cp.cu cost a second launch, the
// row slices' partial sums and their gathering; here one exchange is left, and
// the rest is latency.  us an evaluation, here against two kernels: n = 500,
// r = 129, one trajectory 8.3 against 16.4; n = r = 64 8.3 against 12.4; n = r =
// 512, general form, four trajectories 21.8 against 28.7.
// Every CTA counts itself in once it has read the base, and the last one moves
// it on, so that none can take the next evaluation's number.
struct KEArgs {
  const double *fa, *fb, *fc;  // stored factors, n x rp
  int n, rp, batch, rows;
  const double* u;
  int64_t u_stride;
  double* c;
  int64_t c_stride;
  unsigned int* base;      // step number of the last word published, arrivals
  unsigned long long* hw;  // 2 x 2 x NB x rp
  int* err;
};

// NF factors to project on, CH columns whose sums a thread carries at a time.
template <int NB, int NF, int CH>
__global__ void __launch_bounds__(KX_THREADS, 1) k3x_eval(const KEArgs p) {
  constexpr int V = NF * CH * NB;
  extern __shared__ __align__(16) double ke_smem[];
  __shared__ int abort_sh;
  __shared__ uint32_t tag_sh;
  __shared__ double tot[V];
  const int tid = threadIdx.x, warp = tid >> 5, lane = tid & 31;
  const int G = gridDim.x, g = blockIdx.x, n = p.n, rp = p.rp;
  const int r0 = (int)((int64_t)g * rp / G), rb = (int)((int64_t)(g + 1) * rp / G) - r0;
  const int i0 = (int)((int64_t)g * n / G), ni = (int)((int64_t)(g + 1) * n / G) - i0;
  volatile int* abort_flag = &abort_sh;
  // [expansion rows (NF - 1) x rows x rp][h 2 x NB x rp][partial sums V x threads]
  double* rowe = ke_smem;
  double* hs = rowe + (size_t)(NF - 1) * p.rows * rp;
  double* red = hs + (size_t)2 * NB * rp;
  const double* F[3] = {p.fb, p.fc, p.fa};
  if (tid == 0) {
    abort_sh = 0;
    tag_sh = *reinterpret_cast<volatile unsigned int*>(p.base);
  }
  const int pieces = rp / 2;  // 16-byte pieces of a row
  for (int e = 0; e < NF - 1; ++e)
    for (int t = tid; t < ni * pieces; t += KX_THREADS) {
      const int ri = t / pieces, q = t - ri * pieces;
      ptx::cp_async16(rowe + ((size_t)e * p.rows + ri) * rp + 2 * q,
                      (e == 0 ? p.fa : p.fc) + (int64_t)(i0 + ri) * rp + 2 * q);
    }
  ptx::cp_async_commit();
  // ---- projections of the owned columns
  for (int c0 = 0; c0 < rb; c0 += CH) {
    double acc[NF][CH][NB];
#pragma unroll
    for (int f = 0; f < NF; ++f)
#pragma unroll
      for (int k = 0; k < CH; ++k)
#pragma unroll
        for (int b = 0; b < NB; ++b) acc[f][k][b] = 0.0;
#pragma unroll 2
    for (int i = tid; i < n; i += KX_THREADS) {
      double x[NF][CH], u[NB];
#pragma unroll
      for (int b = 0; b < NB; ++b) u[b] = b < p.batch ? p.u[b * p.u_stride + i] : 0.0;
#pragma unroll
      for (int f = 0; f < NF; ++f)
#pragma unroll
        for (int k = 0; k < CH; ++k) x[f][k] = c0 + k < rb ? F[f][(int64_t)i * rp + r0 + c0 + k] : 0.0;
#pragma unroll
      for (int f = 0; f < NF; ++f)
#pragma unroll
        for (int k = 0; k < CH; ++k)
#pragma unroll
          for (int b = 0; b < NB; ++b) acc[f][k][b] = fma(x[f][k], u[b], acc[f][k][b]);
    }
#pragma unroll
    for (int f = 0; f < NF; ++f)
#pragma unroll
      for (int k = 0; k < CH; ++k)
#pragma unroll
        for (int b = 0; b < NB; ++b) red[((f * CH + k) * NB + b) * KX_THREADS + tid] = acc[f][k][b];
    __syncthreads();
    for (int v = warp; v < V; v += KX_WARPS) {
      const double* x = red + v * KX_THREADS + lane;
      double t = ((x[0] + x[32]) + (x[64] + x[96])) + ((x[128] + x[160]) + (x[192] + x[224]));
#pragma unroll
      for (int off = 16; off > 0; off >>= 1) t += __shfl_xor_sync(0xffffffffu, t, off);
      if (lane == 0) tot[v] = t;
    }
    __syncthreads();
    if (tid < CH * NB) {
      const int k = tid / NB, b = tid - k * NB;
      if (c0 + k < rb && b < p.batch) {
        const uint32_t tag = tag_sh + 1u;
        const int64_t plane = (int64_t)2 * p.batch * rp;
        unsigned long long* w = p.hw + (int64_t)b * rp + r0 + c0 + k;
        kx_publish(w, plane, tot[tid] * tot[CH * NB + tid], tag);
        if constexpr (NF == 3) kx_publish(w + (int64_t)p.batch * rp, plane, tot[tid] * tot[2 * CH * NB + tid], tag);
      }
    }
  }
  __syncthreads();
  const uint32_t tag = tag_sh + 1u;
  if (tid == 0) {
    __threadfence();
    if (atomicInc(p.base + 1, (unsigned)G - 1u) == (unsigned)G - 1u)
      *reinterpret_cast<volatile unsigned int*>(p.base) = tag;
  }
  // ---- h of every column
  bool ok = true;
  if (ni > 0) {
    const int per = (NF - 1) * p.batch * rp, plane = 2 * p.batch * rp;
#pragma unroll
    for (int half = 0; half < 2; ++half)
      ok = ok && kx_poll<true>(p.hw + (size_t)half * plane, per, tag, tid, KX_THREADS, abort_flag,
                               [&](int x, uint32_t bits) {
                                 const int row = x / rp, r = x - row * rp;  // row: which * batch + b
                                 const int which = row >= p.batch ? 1 : 0, b = row - which * p.batch;
                                 reinterpret_cast<uint32_t*>(hs)[(size_t)2 * ((which * NB + b) * rp + r) + half] = bits;
                               });
  }
  ptx::cp_async_wait<0>();
  if (!ok) kx_abort(abort_flag, p.err, p.base, tag);
  if (__syncthreads_or(*abort_flag)) return;
  // ---- the owned rows
  for (int ri = warp; ri < ni; ri += KX_WARPS) {
    const double* x = rowe + (size_t)ri * rp;
    const double* w = rowe + ((size_t)p.rows + ri) * rp;  // skew only
    double s1[NB], s2[NB];
#pragma unroll
    for (int b = 0; b < NB; ++b) s1[b] = s2[b] = 0.0;
#pragma unroll 4
    for (int v = lane; v < rp; v += 32) {
#pragma unroll
      for (int b = 0; b < NB; ++b) {
        if (b >= p.batch) break;
        s1[b] = fma(x[v], hs[(size_t)b * rp + v], s1[b]);
        if constexpr (NF == 3) s2[b] = fma(w[v], hs[(size_t)(NB + b) * rp + v], s2[b]);
      }
    }
#pragma unroll
    for (int b = 0; b < NB; ++b) {
      if (b >= p.batch) break;
      double t = NF == 3 ? s1[b] - s2[b] : s1[b];
#pragma unroll
      for (int off = 16; off > 0; off >>= 1) t += __shfl_xor_sync(0xffffffffu, t, off);
      if (lane == 0) p.c[b * p.c_stride + i0 + ri] = t;
    }
  }
}

// A warp per column and row: CTAs of eight of each, as many as there are SMs.
static int kx_grid(int64_t n, int64_t rp, int sm_count) {
  return (int)std::max<int64_t>(1, std::min<int64_t>(sm_count, (std::max(n, rp) + KX_WARPS - 1) / KX_WARPS));
}

struct KXShape {
  int grid, cols, rows, npad, rpad, nb;
  size_t smem;
};
static KXShape kx_shape(int64_t n, int64_t rp, int form, int storage, int batch, int sm_count) {
  KXShape s{};
  const int nf = form == GROM_FORM_CP_SKEW ? 3 : 2, el = storage_elem_bytes(storage), acc = storage == GROM_F64 ? 8 : 4;
  const int vec = 32 * 16 / el;  // elements of 32 vectors
  s.grid = kx_grid(n, rp, sm_count);
  s.cols = (int)((rp + s.grid - 1) / s.grid);
  s.rows = (int)((n + s.grid - 1) / s.grid);
  s.npad = (int)((n + vec - 1) / vec * vec);
  s.rpad = (int)((rp + vec - 1) / vec * vec);
  s.nb = batch <= 1 ? 1 : batch <= 2 ? 2 : 4;
  s.smem = (size_t)nf * s.cols * s.npad * el + (size_t)(nf - 1) * s.rows * s.rpad * el +
           ((size_t)s.nb * s.npad + 2 * (size_t)s.nb * s.rpad) * acc + (size_t)s.nb * s.rows * 7 * 8;
  return s;
}

// Trajectories of a launch; FP64 ROMs step three and four through the per-step kernels.
static constexpr int kx_max_batch(int storage) { return storage == GROM_F64 ? 2 : 4; }
bool k3x_fits(int64_t n, int64_t rp, int form, int storage, int batch, int sm_count) {
  if (batch > kx_max_batch(storage) || n > (1 << 14) || rp > (1 << 14)) return false;
  return kx_shape(n, rp, form, storage, batch, sm_count).smem <= 220 * 1024;
}

// [base and arrival words][u words][h words][energy / invariant words], for four trajectories
size_t k3x_scratch_bytes(int64_t n, int64_t rp, int sm_count) {
  return 256 + 8 * (2 * 4 * (size_t)n + 2 * 2 * 4 * (size_t)rp + 2 * (size_t)sm_count * 4 * 4);
}

template <int ST>
static cudaError_t kx_run(const KXArgs& p, const KXShape& s, cudaStream_t strm) {
  auto kern = s.nb == 1 ? k3x_kernel<ST, 1> : s.nb == 2 ? k3x_kernel<ST, 2> : k3x_kernel<ST, kx_max_batch(ST)>;
  cudaError_t e = cudaFuncSetAttribute(kern, cudaFuncAttributeMaxDynamicSharedMemorySize, (int)s.smem);
  if (e != cudaSuccess) return e;
  KXArgs a = p;
  void* args[] = {&a};
  return cudaLaunchCooperativeKernel(reinterpret_cast<const void*>(kern), dim3(s.grid), dim3(KX_THREADS), args, s.smem,
                                     strm);
}

cudaError_t k3x_launch(const uint8_t* fa, const uint8_t* fb, const uint8_t* fc, int form, int64_t n, int64_t rp,
                       int storage, int batch, int nsteps, const StepArgs& st, void* scratch, int sm_count,
                       cudaStream_t strm) {
  const KXShape s = kx_shape(n, rp, form, storage, batch, sm_count);
  KXArgs p{};
  p.fa = fa;
  p.fb = fb;
  p.fc = fc;
  p.nf = form == GROM_FORM_CP_SKEW ? 3 : 2;
  p.n = (int)n;
  p.rp = (int)rp;
  p.npad = s.npad;
  p.rpad = s.rpad;
  p.cols = s.cols;
  p.rows = s.rows;
  p.batch = batch;
  p.nsteps = nsteps;
  p.base = static_cast<unsigned int*>(scratch);
  p.uw = reinterpret_cast<unsigned long long*>(static_cast<uint8_t*>(scratch) + 256);
  p.hw = p.uw + 2 * 4 * (size_t)n;
  p.rw = p.hw + 2 * 2 * 4 * (size_t)rp;
  p.st = st;
  switch (storage) {
    case GROM_F64: return kx_run<GROM_F64>(p, s, strm);
    case GROM_F32: return kx_run<GROM_F32>(p, s, strm);
    case GROM_BF16: return kx_run<GROM_BF16>(p, s, strm);
  }
  return cudaErrorInvalidValue;
}

struct KEShape {
  int grid, rows, nb, ch;
  size_t smem;
};
static KEShape ke_shape(int64_t n, int64_t rp, int form, int batch, int sm_count) {
  KEShape s{};
  const int nf = form == GROM_FORM_CP_SKEW ? 3 : 2;
  s.grid = (int)std::max<int64_t>(1, std::min<int64_t>(sm_count, std::max(rp, (n + KX_WARPS - 1) / KX_WARPS)));
  s.rows = (int)((n + s.grid - 1) / s.grid);
  s.nb = batch <= 1 ? 1 : batch <= 2 ? 2 : 4;
  const int cols = (int)((rp + s.grid - 1) / s.grid);
  s.ch = std::min(4 / s.nb, cols <= 1 ? 1 : cols <= 2 ? 2 : 4);
  s.smem = ((size_t)(nf - 1) * s.rows * rp + 2 * (size_t)s.nb * rp + (size_t)nf * s.ch * s.nb * KX_THREADS) * 8;
  return s;
}

// Where one launch is faster: until a CTA's columns and the h that every CTA
// polls outgrow the second launch (skew form: five products an entry and two h
// a column).  us here against k3_cp.cu, n, r, trajectories: skew 256, 256, 4:
// 18.5, 26.7; 512, 512, 2: 20.5, 24.7; 512, 512, 4: 34.3, 33.9; 700, 700, 1:
// 22.6, 25.4; 700, 700, 2: 33.8, 32.9; 1024, 1024, 1: 30.8, 27.3; 2048, 512,
// 2: 36.4, 44.0; general 1024, 1024, 4: 46.9, 53.3; 2048, 512, 4: 45.4, 55.4.
bool k3x_eval_faster(int64_t n, int64_t rp, int form, int batch, int sm_count) {
  if (batch > 4 || n > 2048) return false;
  const KEShape s = ke_shape(n, rp, form, batch, sm_count);
  if (s.smem > 220 * 1024) return false;
  return form == GROM_FORM_CP_SKEW ? s.nb * rp <= 1024 && rp <= 5 * s.grid : s.nb * rp <= 4096 && rp <= 1024;
}

template <int NF>
static void (*ke_kernel(const KEShape& s))(const KEArgs) {
  if (s.nb == 4) return k3x_eval<4, NF, 1>;
  if (s.nb == 2) return s.ch == 1 ? k3x_eval<2, NF, 1> : k3x_eval<2, NF, 2>;
  return s.ch == 1 ? k3x_eval<1, NF, 1> : s.ch == 2 ? k3x_eval<1, NF, 2> : k3x_eval<1, NF, 4>;
}

cudaError_t k3x_eval_launch(const K3Args& a, int64_t n, int64_t rp, int batch, void* scratch, int* err, int sm_count,
                            cudaStream_t strm) {
  const KEShape s = ke_shape(n, rp, a.form, batch, sm_count);
  KEArgs p{};
  p.fa = reinterpret_cast<const double*>(a.fa);
  p.fb = reinterpret_cast<const double*>(a.fb);
  p.fc = reinterpret_cast<const double*>(a.fc);
  p.n = (int)n;
  p.rp = (int)rp;
  p.batch = batch;
  p.rows = s.rows;
  p.u = a.u;
  p.u_stride = a.u_stride;
  p.c = a.c;
  p.c_stride = a.c_stride;
  p.base = static_cast<unsigned int*>(scratch);
  p.hw = reinterpret_cast<unsigned long long*>(static_cast<uint8_t*>(scratch) + 256) + 2 * 4 * (size_t)n;
  p.err = err;
  auto kern = a.form == GROM_FORM_CP_SKEW ? ke_kernel<3>(s) : ke_kernel<2>(s);
  cudaError_t e = cudaFuncSetAttribute(kern, cudaFuncAttributeMaxDynamicSharedMemorySize, (int)s.smem);
  if (e != cudaSuccess) return e;
  void* args[] = {&p};
  return cudaLaunchCooperativeKernel(reinterpret_cast<const void*>(kern), dim3(s.grid), dim3(KX_THREADS), args, s.smem,
                                     strm);
}

}  // namespace grom
