// The skew-packed advection term of the FP64-tolerance storages (F64, F32X2),
// HBM streaming: the folded layout of a skew tensor.
//
// c_i = sum_jk C_ijk u_j u_k depends on C_ijk + C_ikj only, and C_ijk = -C_kji
// ties those sums over the three roles of an index triple to zero, so n^3 / 3
// of the n^3 entries fix c.  For every m the stored matrix is
//   F^m_pq = C_pqm + C_pmq  (q < m),  F^m_pm = C_pmm,     p < m, q <= m,
// and with D_p = sum_q F^m_pq u_q the term is
//   c_p += D_p u_m  (p < m),     c_m -= sum_p D_p u_p.
// (Adding a totally antisymmetric tensor to a skew one leaves c unchanged;
// the layout takes the one that clears the entries whose middle index is the
// largest.  Each stored value is one FP64 sum of two entries, rounded once
// into the storage.)  u . c = 0 holds term by term, as for the entries
// themselves.  Against one entry of each pair (n^3 / 2) the bytes and the
// multiply-adds are two thirds: a step of n = 1024 F32X2, bound by HBM (2.89
// GB at 6.6 TB/s), takes 433 us instead of 650; an evaluation of n = 769 F64,
// three trajectories, bound by the FP64 pipe (0.7 ms of it at two
// multiply-adds a clock and SM), 975 us instead of 1759.
//
// Group m holds m + 1 rows q of the m values p (p contiguous; F32X2: the hi
// values, then the lo ones), each zero-padded to 128 bytes, so that every row
// starts on such a boundary.  A CTA streams a contiguous range of rows through a ring
// of bulk copies; a consumer thread owns positions p and accumulates D_p over
// the rows, so nothing is reduced per row.  At the end of a group it adds
// D_p u_m to its own c_p, kept for the whole range, and the warp sums D_p u_p;
// the CTA ends with one window of c.  Row ranges are cut so that bytes plus a
// charge per group (its end is some dozen FP64 instructions a warp on a pipe
// of two lanes a clock) are equal.  Sixteen consumer warps: with eight, the
// waits and loads of a chunk were not covered (F32X2: 640 us).
#pragma once

#include <type_traits>

#include "k1_stream.cuh"
#include "k1t_types.h"
#include "step_elem.cuh"

namespace grom {

// Sums d over the 2^lgR row groups of a warp (lanes 8 apart, group `ro`):
// lane ro ends with the complete elements k1t_first .. + EPV / 2^lgR in
// d[0 ..]; with more row groups than elements, both groups of a pair hold one.
template <int EPV>
__device__ __forceinline__ void k1t_gather(double (&d)[EPV], int lgR, int ro) {
  if (lgR >= 1) {
    const bool up = ro & 1;
#pragma unroll
    for (int e = 0; e < EPV / 2; ++e) {
      const double send = up ? d[e] : d[e + EPV / 2], keep = up ? d[e + EPV / 2] : d[e];
      d[e] = keep + __shfl_xor_sync(0xffffffffu, send, 8);
    }
  }
  if (lgR >= 2) {
    if constexpr (EPV == 4) {
      const bool up = ro & 2;
      const double send = up ? d[0] : d[1], keep = up ? d[1] : d[0];
      d[0] = keep + __shfl_xor_sync(0xffffffffu, send, 16);
    } else {
      d[0] += __shfl_xor_sync(0xffffffffu, d[0], 16);
    }
  }
}
template <int EPV>
__device__ __forceinline__ int k1t_first(int lgR, int ro) {
  int e = lgR >= 1 && (ro & 1) ? EPV / 2 : 0;
  if (EPV == 4 && lgR >= 2 && (ro & 2)) e += 1;
  return e;
}

// Grid barrier of the consumer warps of every CTA (cooperative launch): CTA 0
// adds 2^31 - (G - 1), the others 1, so the top bit flips once per barrier and
// the low bits return to their value.  Gives up after the time limit.
__device__ __forceinline__ bool k1t_barrier(unsigned int* bar, int* err, volatile int* abort_flag, int* ok_sh) {
  ptx::named_sync(1, K1T_CONSUMERS);
  if (threadIdx.x == 0) {
    const unsigned int inc = blockIdx.x == 0 ? 0x80000000u - (gridDim.x - 1) : 1u;
    __threadfence();
    const unsigned int old = atomicAdd(bar, inc);
    int ok = 1;
    const uint64_t t0 = ptx::globaltimer();
    for (uint32_t spin = 0;; ++spin) {
      const unsigned int now = *reinterpret_cast<volatile unsigned int*>(bar);
      if ((now ^ old) & 0x80000000u) break;
      if ((spin & 255u) == 255u && ptx::globaltimer() - t0 > ptx::WAIT_LIMIT_NS) {
        atomicOr(err, DEV_ERR_TIMEOUT);
        *abort_flag = 1;
        ok = 0;
        break;
      }
    }
    __threadfence();
    *ok_sh = ok;
  }
  ptx::named_sync(1, K1T_CONSUMERS);
  return *ok_sh != 0;
}

// A consumer thread's accumulators D_p over its QM vectors of a row, NB
// trajectories, and the arithmetic on them.  rows<NR, QO> takes NR rows of the
// first QO vectors (one straight-line block, so that the rows' chains
// interleave; a predicate on the vectors would leave the skipped FP64
// instructions on their pipe), u of row t at index j + t jstep, rows from
// `have` on zeros, after `loaded` has given the stage back.
template <int ST, int QM, int NB>
struct K1TAcc;

template <int QM, int NB>
struct K1TAcc<GROM_F64, QM, NB> {
  double v[QM][2][NB];
  __device__ __forceinline__ void zero() {
#pragma unroll
    for (int q = 0; q < QM; ++q)
#pragma unroll
      for (int b = 0; b < NB; ++b) v[q][0][b] = v[q][1][b] = 0.0;
  }
  __device__ __forceinline__ void take(int q, int b, double (&d)[2]) {
    d[0] = v[q][0][b];
    d[1] = v[q][1][b];
    v[q][0][b] = v[q][1][b] = 0.0;
  }
  template <int NR, int QO, typename F>
  __device__ __forceinline__ void rows(const uint8_t* stg, int t_step, const int (&poff)[QM], int, int have,
                                       const double* ud, const float*, int np, int j, int jstep, int jmax, F loaded) {
    double2 x[NR][QO];
#pragma unroll
    for (int t = 0; t < NR; ++t)
#pragma unroll
      for (int q = 0; q < QO; ++q)
        x[t][q] = t < NR - 1 || t < have ? *reinterpret_cast<const double2*>(stg + t * t_step + poff[q])
                                         : make_double2(0.0, 0.0);
    loaded();
#pragma unroll
    for (int t = 0; t < NR; ++t) {
      const double* u = ud + min(j + t * jstep, jmax);
      double uj[NB];
#pragma unroll
      for (int b = 0; b < NB; ++b) uj[b] = u[b * np];
#pragma unroll
      for (int q = 0; q < QO; ++q) {
#pragma unroll
        for (int b = 0; b < NB; ++b) {
          v[q][0][b] = fma(x[t][q].x, uj[b], v[q][0][b]);
          v[q][1][b] = fma(x[t][q].y, uj[b], v[q][1][b]);
        }
      }
    }
  }
};

template <int QM, int NB>
struct K1TAcc<GROM_F32X2, QM, NB> {
  f32pair S[QM][2][NB], s[QM][2][NB];
  __device__ __forceinline__ void zero() {
#pragma unroll
    for (int q = 0; q < QM; ++q)
#pragma unroll
      for (int e = 0; e < 2; ++e)
#pragma unroll
        for (int b = 0; b < NB; ++b) S[q][e][b].v = s[q][e][b].v = 0ull;
  }
  __device__ __forceinline__ void take(int q, int b, double (&d)[4]) {
#pragma unroll
    for (int e = 0; e < 2; ++e) {
      float h0, h1, l0, l1;
      pair_get(S[q][e][b], h0, h1);
      pair_get(s[q][e][b], l0, l1);
      d[2 * e] = f2d_int(h0) + f2d_int(l0);
      d[2 * e + 1] = f2d_int(h1) + f2d_int(l1);
      S[q][e][b].v = s[q][e][b].v = 0ull;
    }
  }
  template <int NR, int QO, typename F>
  __device__ __forceinline__ void rows(const uint8_t* stg, int t_step, const int (&poff)[QM], int plane, int have,
                                       const double*, const float* uf, int np, int j, int jstep, int jmax, F loaded) {
    ulonglong2 h[NR][QO], l[NR][QO];
#pragma unroll
    for (int t = 0; t < NR; ++t)
#pragma unroll
      for (int q = 0; q < QO; ++q) {
        const uint8_t* p = stg + t * t_step + poff[q];
        const bool on = t < NR - 1 || t < have;
        h[t][q] = on ? *reinterpret_cast<const ulonglong2*>(p) : make_ulonglong2(0ull, 0ull);
        l[t][q] = on ? *reinterpret_cast<const ulonglong2*>(p + plane) : make_ulonglong2(0ull, 0ull);
      }
    loaded();
    // renormalised once a chunk (every few terms; see ds_arith.cuh)
#pragma unroll
    for (int q = 0; q < QO; ++q)
#pragma unroll
      for (int e = 0; e < 2; ++e)
#pragma unroll
        for (int b = 0; b < NB; ++b) ds_renorm2(S[q][e][b], s[q][e][b]);
#pragma unroll
    for (int t = 0; t < NR; ++t) {
      const float* u = uf + min(j + t * jstep, jmax);
      f32pair uh[NB], ul[NB];
#pragma unroll
      for (int b = 0; b < NB; ++b) {
        uh[b] = pair_make(u[b * np], u[b * np]);
        ul[b] = pair_make(u[(NB + b) * np], u[(NB + b) * np]);
      }
#pragma unroll
      for (int q = 0; q < QO; ++q) {
#pragma unroll
        for (int b = 0; b < NB; ++b) {
          ds_mac2(f32pair{h[t][q].x}, f32pair{l[t][q].x}, uh[b], ul[b], S[q][0][b], s[q][0][b]);
          ds_mac2(f32pair{h[t][q].y}, f32pair{l[t][q].y}, uh[b], ul[b], S[q][1][b], s[q][1][b]);
        }
      }
    }
  }
};

// STEP false: one evaluation for the NB trajectories from a.b0 (windows only;
// k1t_finish sums them).  STEP true: st-steps of up to NB trajectories in one
// cooperative launch; per step the windows, a grid barrier, every CTA
// finalises and steps its own test indices, a grid barrier.  The producer
// warp takes no part in the barriers: the tensor does not depend on u, so the
// next step's rows stream in meanwhile.
template <int ST, int QM, int NB, bool STEP>
__global__ void __launch_bounds__(K1T_THREADS, 1) k1t_kernel(const K1TArgs a, const StepArgs st) {
  constexpr int EPV = K1Traits<ST>::EPV;
  constexpr int PLANES = ST == GROM_F32X2 ? 2 : 1;  // 16-byte vectors of a position
  constexpr int RMAX = k1t_rmax(ST, QM, NB);
  constexpr bool CS = k1t_c_shared(ST, QM, NB);
  extern __shared__ uint8_t smem_raw[];
  uint8_t* smem = reinterpret_cast<uint8_t*>((reinterpret_cast<uintptr_t>(smem_raw) + 1023) & ~uintptr_t(1023));
  uint8_t* stages = smem;
  const int NS = a.stages;
  uint64_t* full = reinterpret_cast<uint64_t*>(smem + (size_t)NS * K1_STAGE_BYTES);
  uint64_t* empty = full + NS;
  // u of the NB trajectories in FP64 and, for F32X2, as hi and lo floats
  double* ud = reinterpret_cast<double*>(empty + NS);
  float* uf = reinterpret_cast<float*>(ud + (size_t)NB * a.np);
  // c of the range, where CS (F64 has no float planes)
  double* cs = ud + (ST == GROM_F64 ? 1 : 2) * (size_t)NB * a.np;
  __shared__ volatile int abort_sh;
  __shared__ int mlast_tab[STEP ? K1T_MAX_GRID : 1];
  __shared__ double wpart[K1T_WARPS][NB][2];
  __shared__ int ok_sh;
  __shared__ int64_t l0s[NB];
  volatile int* abort_flag = &abort_sh;

  const int tid = threadIdx.x, warp = tid >> 5, lane = tid & 31;
  const int n = a.n, np = a.np, G = gridDim.x, g = blockIdx.x;
  const int4 rg = a.ranges[g];  // rows (m0, q0) up to, not including, (m1, q1)
  const int m0 = rg.x, q0 = rg.y, m1 = rg.z, q1 = rg.w;
  const int mlast = k1t_last_group(rg);  // -1: no rows
  // row groups of a warp that share its positions: as many as the widest row leaves room for
  const int ptop = mlast > 0 ? (mlast + EPV - 1) / EPV : 1;
  const int lgR = 4 * ptop <= K1T_CONSUMERS ? 2 : 2 * ptop <= K1T_CONSUMERS ? 1 : 0;
  const int R = 1 << lgR;

  if (tid == 0) {
    for (int s = 0; s < NS; ++s) {
      ptx::mbar_init(&full[s], 1);
      ptx::mbar_init(&empty[s], K1T_WARPS);
    }
    abort_sh = 0;
    ptx::fence_mbar_init();
  }
  if constexpr (STEP) {
    for (int q = tid; q < G; q += K1T_THREADS) mlast_tab[q] = k1t_last_group(a.ranges[q]);
    if (tid < NB) l0s[tid] = tid < a.nb ? st.taken[tid] : 0;
  }
  __syncthreads();
  const int nsteps = STEP ? a.nsteps : 1;

  if (warp == K1T_WARPS) {
    // ------------------------------------------------ producer, all steps
    if (lane == 0) {
      int64_t it = 0;
      int s = 0;
      uint32_t ph = 0;
      bool stop = false;
      for (int step = 0; step < nsteps && !stop; ++step) {
        for (int m = m0; m <= mlast && !stop; ++m) {
          const int rb = k1t_row_bytes(m);
          const int rpc = k1t_rows_per_chunk(rb, RMAX * R);
          const int qe = m == m1 ? q1 : m + 1;
          const uint8_t* src = a.tensor + a.off[m];
          for (int q = m == m0 ? q0 : 0; q < qe; q += rpc, ++it) {
            if (it >= NS && !ptx::mbar_wait(&empty[s], ph ^ 1u, abort_flag)) {
              *abort_flag = 1;
              atomicOr(a.err, DEV_ERR_TIMEOUT);
              stop = true;
              break;
            }
            const uint32_t bytes = (uint32_t)((qe - q < rpc ? qe - q : rpc) * rb);
            ptx::mbar_arrive_expect_tx(&full[s], bytes);
            ptx::bulk_g2s(stages + (size_t)s * K1_STAGE_BYTES, src + (int64_t)q * rb, bytes, &full[s]);
            if (++s == NS) { s = 0; ph ^= 1u; }
          }
        }
      }
      const int64_t issued = it;
      for (int64_t q = issued > NS ? issued - NS : 0; q < issued; ++q) {
        if (!ptx::mbar_wait(&full[q % NS], (uint32_t)((q / NS) & 1), nullptr)) atomicOr(a.err, DEV_ERR_TIMEOUT);
      }
    }
  } else {
    // ------------------------------------------------------------ consumers
    const int W = K1T_CONSUMERS >> lgR;  // positions per q-slab
    const int ro = (tid >> 3) & (R - 1);
    const int pos0 = ((tid >> (3 + lgR)) << 3) + (tid & 7);
    const int wpos = (warp * 32 >> (3 + lgR)) << 3;  // smallest position of the warp
    const int uplane = NB * np;
    // after k1t_gather: the elements [e0, e0 + ne) of the lane's vector are its own
    const int ne = EPV >> lgR > 0 ? EPV >> lgR : 1;
    const int e0 = k1t_first<EPV>(lgR, ro);
    const bool mine = R <= EPV || (ro >> 1) == 0;
    double* part = a.part + (int64_t)g * a.maxseg * (K1T_WARPS) * NB;
    double* win = a.win + (int64_t)g * NB * np;
    int s = 0;
    uint32_t ph = 0;

    for (int step = 0; step < nsteps; ++step) {
      // ---- u^l into shared memory (in a stepping launch written by every CTA
      // in the previous step: read through L2)
      for (int idx = tid; idx < NB * np; idx += K1T_CONSUMERS) {
        const int b = idx / np, k = idx - b * np;
        double v = 0.0;
        if (b < a.nb && k < n) {
          if constexpr (STEP) {
            v = __ldcg(a.hist + b * a.hist_stride + ((l0s[b] + step) % 3) * n + k);
          } else {
            const int bg = a.b0 + b;
            if (!a.active || a.active[bg])
              v = a.taken ? a.hist[bg * a.hist_stride + (a.taken[bg] % 3) * n + k] : a.u[bg * a.u_stride + k];
          }
        }
        ud[idx] = v;
        if constexpr (ST == GROM_F32X2) ds_split(v, uf[idx], uf[uplane + idx]);
        if constexpr (CS) cs[idx] = 0.0;
      }
      ptx::named_sync(1, K1T_CONSUMERS);

      K1TAcc<ST, QM, NB> acc;
      acc.zero();
      // c at the owned positions, in registers or in shared memory
      double cacc[CS ? 1 : QM][CS ? 1 : EPV][CS ? 1 : NB];
      if constexpr (!CS) {
#pragma unroll
        for (int q = 0; q < QM; ++q)
#pragma unroll
          for (int e = 0; e < EPV; ++e)
#pragma unroll
            for (int b = 0; b < NB; ++b) cacc[q][e][b] = 0.0;
      }

      bool stop = false;
      for (int m = m0; m <= mlast && !stop; ++m) {
        const int rb = k1t_row_bytes(m);
        const int rpc = k1t_rows_per_chunk(rb, RMAX * R);
        const int qe = m == m1 ? q1 : m + 1;
        const int P = rb / (16 * PLANES);  // 16-byte vectors of a row and plane
        const int t_step = R * rb, plane_off = rb >> 1;
        // a lane past the row's end reads its last vector; its sums are not used
        int poff[QM];
#pragma unroll
        for (int q = 0; q < QM; ++q) poff[q] = (pos0 + q * W < P ? pos0 + q * W : P - 1) * 16;
        const int qon = P > wpos ? (P - wpos + W - 1) / W : 0;  // slabs in which the warp has a position
        for (int qr = m == m0 ? q0 : 0; qr < qe; qr += rpc) {
          const int rows = qe - qr < rpc ? qe - qr : rpc;
          // warp-uniform: a lane whose wait timed out takes its whole warp
          // along (the shuffles and the named barriers need every lane)
          if (!__all_sync(0xffffffffu, ptx::mbar_wait(&full[s], ph, abort_flag))) {
            if (lane == 0) {
              *abort_flag = 1;
              atomicOr(a.err, DEV_ERR_TIMEOUT);
            }
            stop = true;
            break;
          }
          const uint8_t* stg = stages + (size_t)s * K1_STAGE_BYTES + ro * rb;
          const int have = (rows - ro + R - 1) >> lgR, most = (rows + R - 1) >> lgR;  // of this thread, of the warp
          const int j = qr + ro;
          auto loaded = [&] {
            __syncwarp();
            if (lane == 0) ptx::mbar_arrive(&empty[s]);
            if (++s == NS) { s = 0; ph ^= 1u; }
          };
          auto take = [&](auto vectors) {
            constexpr int QO = decltype(vectors)::value;
            switch (most) {  // <= RMAX: the plan caps a chunk at RMAX * R rows
#define K1T_ROWS(N)                                                                                      \
  case N:                                                                                                \
    if constexpr (N <= RMAX) acc.template rows<N, QO>(stg, t_step, poff, plane_off, have, ud, uf, np, j, R, m, loaded); \
    break;
              K1T_ROWS(1)
              K1T_ROWS(2)
              K1T_ROWS(3)
              K1T_ROWS(4)
              K1T_ROWS(5)
              K1T_ROWS(6)
              K1T_ROWS(7)
              K1T_ROWS(8)
#undef K1T_ROWS
            }
          };
          switch (qon) {  // <= QM
            case 0: loaded(); break;
            case 1: take(std::integral_constant<int, 1>()); break;
            case 2: if constexpr (QM >= 2) take(std::integral_constant<int, 2>()); break;
            case 3: if constexpr (QM >= 4) take(std::integral_constant<int, 3>()); break;
            case 4: if constexpr (QM >= 4) take(std::integral_constant<int, 4>()); break;
          }
        }
        if (stop) break;
        // ---- end of the group: D_p of the owned positions into c_p and the
        // warp's sum of D_p u_p.  With several row groups a lane hands half of
        // its vector to its partner and adds what it gets, so that each D_p
        // ends up complete in one lane.
        double contrib[NB], um[NB];
#pragma unroll
        for (int b = 0; b < NB; ++b) {
          contrib[b] = 0.0;
          um[b] = ud[b * np + m];
        }
#pragma unroll
        for (int q = 0; q < QM; ++q) {
          if (wpos + q * W >= P) break;  // warp-uniform
          const bool own = pos0 + q * W < P;
          const int p0 = (pos0 + q * W) * EPV + e0;
#pragma unroll
          for (int b = 0; b < NB; ++b) {
            double d[EPV];
            acc.take(q, b, d);
            k1t_gather<EPV>(d, lgR, ro);
#pragma unroll
            for (int e = 0; e < EPV; ++e) {
              if (e >= ne) break;  // uniform: EPV / R elements are this lane's (R > EPV: one, on half the lanes)
              if (own && mine) {
                contrib[b] = fma(ud[b * np + p0 + e], d[e], contrib[b]);
                if constexpr (CS)
                  cs[b * np + p0 + e] = fma(d[e], um[b], cs[b * np + p0 + e]);
                else
                  cacc[q][e][b] = fma(d[e], um[b], cacc[q][e][b]);
              }
            }
          }
        }
#pragma unroll
        for (int b = 0; b < NB; ++b) {
          double v = contrib[b];
#pragma unroll
          for (int off = 16; off > 0; off >>= 1) v += __shfl_xor_sync(0xffffffffu, v, off);
          if (lane == 0) part[((m - m0) * (K1T_WARPS) + warp) * NB + b] = v;
        }
      }
      // every consumer warp arrives here; thread 0 reads the abort flag (the
      // producer may set it at any time) and every consumer acts on that value
      ptx::named_sync(1, K1T_CONSUMERS);
      if (tid == 0) ok_sh = *abort_flag ? 0 : 1;
      ptx::named_sync(1, K1T_CONSUMERS);
      if (!ok_sh) break;

      // ---- this CTA's window of c: positions 0 .. mlast
#pragma unroll
      for (int q = 0; q < QM; ++q)
#pragma unroll
        for (int e = 0; e < EPV; ++e) {
          const int p = (pos0 + q * W) * EPV + e0 + e;
          if (e < ne && mine && p < mlast)
#pragma unroll
            for (int b = 0; b < NB; ++b) {
              if constexpr (CS)
                win[b * np + p] = cs[b * np + p];
              else
                win[b * np + p] = cacc[q][e][b];
            }
        }
      ptx::named_sync(1, K1T_CONSUMERS);
      for (int idx = tid; idx < (mlast + 1 - m0) * NB && mlast >= 0; idx += K1T_CONSUMERS) {
        const int b = idx % NB, m = m0 + idx / NB;
        double v = m < mlast ? __ldcg(win + b * np + m) : 0.0;
#pragma unroll
        for (int w = 0; w < K1T_WARPS; ++w)
          v -= __ldcg(part + ((m - m0) * (K1T_WARPS) + w) * NB + b);
        win[b * np + m] = v;
      }
      if constexpr (STEP) {
        if (!k1t_barrier(a.bar, a.err, abort_flag, &ok_sh)) break;

        // ---- finalise and step the owned test indices (a warp per index)
        const int i_lo = (int)((int64_t)g * n / G), i_hi = (int)((int64_t)(g + 1) * n / G);
        double ew[NB], iw[NB];
#pragma unroll
        for (int b = 0; b < NB; ++b) ew[b] = iw[b] = 0.0;
        int bad = 0;
        for (int i = i_lo + warp; i < i_hi; i += K1T_WARPS) {
#pragma unroll
          for (int b = 0; b < NB; ++b) {
            if (b >= a.nb) break;
            double v = 0.0;
            for (int q = lane; q < G; q += 32)
              if (mlast_tab[q] >= i) v += __ldcg(a.win + ((int64_t)q * NB + b) * np + i);
#pragma unroll
            for (int off = 16; off > 0; off >>= 1) v += __shfl_xor_sync(0xffffffffu, v, off);
            if (lane == 0) {
              const int64_t l = l0s[b] + step;
              const int k = (int)(l + 1 < st.order ? l + 1 : st.order);
              double* h = st.hist + b * st.hist_stride;
              h[(3 + l % 3) * n + i] = v;
              double ep, ip;
              int bb;
              // (loaded before the windows, these operands cost the F32X2
              // stream 2 %: 435 us a step of n = 1024 against 444; loaded
              // whatever the order, 2 % at n = 1000)
              step_elem(st, h, n, l, k, i, step_load<false, false>(st, h, n, l, k, i), v, ep, ip, bb);
              ew[b] += ep;
              iw[b] += ip;
              if (bb) {
                bad = 1;
                atomicMin(st.first_bad, b);
              }
            }
          }
        }
        if (lane == 0) {
#pragma unroll
          for (int b = 0; b < NB; ++b) {
            wpart[warp][b][0] = ew[b];
            wpart[warp][b][1] = iw[b];
          }
          if (bad) atomicOr(st.err, DEV_ERR_NONFINITE);
        }
        ptx::named_sync(1, K1T_CONSUMERS);
        if (tid < NB) {
          double e = 0.0, v = 0.0;
          for (int w = 0; w < K1T_WARPS; ++w) {
            e += wpart[w][tid][0];
            v += wpart[w][tid][1];
          }
          a.red[((int64_t)g * NB + tid) * 2] = e;
          a.red[((int64_t)g * NB + tid) * 2 + 1] = v;
        }
        if (!k1t_barrier(a.bar, a.err, abort_flag, &ok_sh)) break;

        // ---- energy / invariant of the step: warp b of CTA 0 sums the CTA
        // partials of trajectory b (lane q adds CTAs q, q + 32, ... in order)
        if (g == 0 && warp < a.nb && warp < NB && (st.energy || st.invariant)) {
          double e = 0.0, v = 0.0;
          for (int q = lane; q < G; q += 32) {
            e += __ldcg(a.red + ((int64_t)q * NB + warp) * 2);
            v += __ldcg(a.red + ((int64_t)q * NB + warp) * 2 + 1);
          }
#pragma unroll
          for (int off = 16; off > 0; off >>= 1) {
            e += __shfl_xor_sync(0xffffffffu, e, off);
            v += __shfl_xor_sync(0xffffffffu, v, off);
          }
          if (lane == 0) {
            if (st.energy) st.energy[(int64_t)step * st.batch + warp] = 0.5 * e;
            if (st.invariant) st.invariant[(int64_t)step * st.batch + warp] = v;
          }
        }
      }
    }
    if constexpr (STEP) {
      // the step count of every trajectory, once all CTAs are done with it
      if (g == 0 && tid < a.nb && !*abort_flag) st.taken[tid] = l0s[tid] + nsteps;
    }
  }
  __syncthreads();
}

// Launches of one storage type (k1t_f64.cu, k1t_f32x2.cu): nb trajectories,
// one evaluation (nsteps 0) or nsteps steps.
template <int ST, int QM, int NB, bool STEP>
cudaError_t k1t_launch_one(const K1TArgs& a, const StepArgs& st, int grid, size_t smem, cudaStream_t s) {
  auto kern = k1t_kernel<ST, QM, NB, STEP>;
  cudaError_t e = cudaFuncSetAttribute(kern, cudaFuncAttributeMaxDynamicSharedMemorySize, (int)smem);
  if (e != cudaSuccess) return e;
  if constexpr (STEP) {
    int per_sm = 0;
    e = cudaOccupancyMaxActiveBlocksPerMultiprocessor(&per_sm, kern, K1T_THREADS, smem);
    if (e != cudaSuccess) return e;
    if (per_sm < 1) return cudaErrorCooperativeLaunchTooLarge;
    K1TArgs ac = a;
    StepArgs stc = st;
    void* args[] = {&ac, &stc};
    return cudaLaunchCooperativeKernel(reinterpret_cast<const void*>(kern), dim3(grid), dim3(K1T_THREADS), args, smem, s);
  } else {
    kern<<<grid, K1T_THREADS, smem, s>>>(a, st);
    return cudaGetLastError();
  }
}

template <int ST, int QM, int NB>
cudaError_t k1t_pick(const K1TArgs& a, const StepArgs& st, int grid, size_t smem, cudaStream_t s) {
  if constexpr (NB <= k1t_nb_cap(ST, QM)) {
    if (a.nsteps > 0) return k1t_launch_one<ST, QM, NB, true>(a, st, grid, smem, s);
    return k1t_launch_one<ST, QM, NB, false>(a, st, grid, smem, s);
  }
  return cudaErrorInvalidValue;
}

template <int ST, int QM>
cudaError_t k1t_pick_nb(int nb, const K1TArgs& a, const StepArgs& st, int grid, size_t smem, cudaStream_t s) {
  switch (nb) {
    case 1: return k1t_pick<ST, QM, 1>(a, st, grid, smem, s);
    case 2: return k1t_pick<ST, QM, 2>(a, st, grid, smem, s);
    case 3: return k1t_pick<ST, QM, 3>(a, st, grid, smem, s);
    case 4: return k1t_pick<ST, QM, 4>(a, st, grid, smem, s);
  }
  return cudaErrorInvalidValue;
}

}  // namespace grom
