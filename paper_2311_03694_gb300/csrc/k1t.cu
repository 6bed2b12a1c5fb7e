// Folded skew-packed layout: plan, conversion, finalize and launches (k1t.cuh).
#include <algorithm>

#include "ds_arith.cuh"
#include "grom_internal.h"

namespace grom {

cudaError_t k1t_dispatch_f64(int, int, const K1TArgs&, const StepArgs&, int, size_t, cudaStream_t);
cudaError_t k1t_dispatch_f32x2(int, int, const K1TArgs&, const StepArgs&, int, size_t, cudaStream_t);

// Bytes of a pass's states (and sums, where they lie in shared memory), and
// the stages of the ring beside them.
static int64_t k1t_state_bytes(const K1TPlan& p, int nb) {
  return (int64_t)nb * p.np * ((p.storage == GROM_F64 ? 8 : 16) + (k1t_c_shared(p.storage, p.qm, nb) ? 8 : 0));
}
static int k1t_stages(const K1TPlan& p, int nb) {
  const int64_t left = 232448 - 1024 - 4096 - k1t_state_bytes(p, nb);  // static tables and barriers: below 4 KB
  return (int)std::min<int64_t>(K1_STAGES, left / K1_STAGE_BYTES);
}
static size_t k1t_smem(const K1TPlan& p, int nb) {
  const int ns = k1t_stages(p, nb);
  return 1024 + (size_t)ns * K1_STAGE_BYTES + 2 * (size_t)ns * 8 + (size_t)k1t_state_bytes(p, nb);
}

// Cost of a group's end in bytes streamed, which the row ranges balance
// (n = 1024 F32X2, a step: 444 us with 192 KB, 476 with 96, 439 with 300; n =
// 769 F64, three trajectories: 973 us with 96 KB, 1000 with 36, 993 with 192).
static int64_t k1t_group_cost(int storage) { return storage == GROM_F64 ? 96 << 10 : 256 << 10; }

K1TPlan k1t_plan(int64_t n, int storage, int sm_count) {
  K1TPlan p;
  p.n = (int)n;
  p.np = (int)padded_n(n);
  p.storage = storage;
  p.epv = storage == GROM_F64 ? 2 : 4;
  const int64_t pmax = (n + p.epv - 1) / p.epv;
  while ((int64_t)p.qm * K1T_CONSUMERS < pmax) p.qm *= 2;
  p.nb_max = k1t_nb_cap(storage, p.qm);
  while (p.nb_max > 1 && k1t_stages(p, p.nb_max) < 3) --p.nb_max;
  p.off.resize((size_t)n + 1);
  const int64_t group = k1t_group_cost(storage);
  int64_t off = 0, total = 0;
  for (int m = 0; m <= n; ++m) {
    p.off[m] = off;
    if (m == 0 || m == n) continue;
    const int64_t rows = (int64_t)(m + 1) * k1t_row_bytes(m);
    off += (rows + 127) / 128 * 128;
    total += rows + group;
  }
  p.bytes = (size_t)std::max<int64_t>(off, 128);
  p.grid = (int)std::max<int64_t>(1, std::min<int64_t>(std::min(sm_count, K1T_MAX_GRID), n * (n - 1) / 2));
  // cut the rows where the running cost passes g / grid of the total
  auto cut = [&](int g, int m, int64_t before, int* q) {  // rows of group m below the cut
    const int64_t rb = k1t_row_bytes(m);
    const double want = (double)total * g / p.grid - (double)before;
    const int64_t x = (int64_t)(want / (double)rb + 0.5);
    *q = (int)std::max<int64_t>(0, std::min<int64_t>(x, m + 1));
  };
  std::vector<int2> start((size_t)p.grid + 1);
  start[0] = make_int2(1, 0);
  start[p.grid] = make_int2((int)n, 0);
  int m = 1;
  int64_t before = 0;  // cost of the groups below m
  for (int g = 1; g < p.grid; ++g) {
    const double want = (double)total * g / p.grid;
    while (m + 1 < n) {
      const int64_t cost = (int64_t)(m + 1) * k1t_row_bytes(m) + group;
      if ((double)(before + cost) > want) break;
      before += cost;
      ++m;
    }
    int q = 0;
    if (m < n) cut(g, m, before, &q);
    int2 x = q > m ? make_int2(m + 1, 0) : make_int2(m, q);
    if (x.x < start[g - 1].x || (x.x == start[g - 1].x && x.y < start[g - 1].y)) x = start[g - 1];
    start[g] = x;
  }
  p.ranges.resize((size_t)p.grid);
  p.maxseg = 1;
  for (int g = 0; g < p.grid; ++g) {
    p.ranges[g] = make_int4(start[g].x, start[g].y, start[g + 1].x, start[g + 1].y);
    const int last = k1t_last_group(p.ranges[g]);
    if (last >= 0) p.maxseg = std::max(p.maxseg, last - p.ranges[g].x + 1);
  }
  return p;
}

static size_t round256(size_t b) { return (b + 255) / 256 * 256; }

// [barrier word][energy / invariant partials][row sums][windows]
size_t k1t_scratch_bytes(const K1TPlan& p) {
  return 256 + round256((size_t)p.grid * p.nb_max * 2 * 8) +
         round256((size_t)p.grid * p.maxseg * (K1T_WARPS) * p.nb_max * 8) + (size_t)p.grid * p.nb_max * p.np * 8;
}

static void k1t_fill(const K1TPlan& p, K1TArgs& a, void* scratch) {
  uint8_t* base = static_cast<uint8_t*>(scratch);
  a.off = p.d_off;
  a.ranges = p.d_ranges;
  a.n = p.n;
  a.np = p.np;
  a.maxseg = p.maxseg;
  a.bar = reinterpret_cast<unsigned int*>(base);
  base += 256;
  a.red = reinterpret_cast<double*>(base);
  base += round256((size_t)p.grid * p.nb_max * 2 * 8);
  a.part = reinterpret_cast<double*>(base);
  base += round256((size_t)p.grid * p.maxseg * (K1T_WARPS) * p.nb_max * 8);
  a.win = reinterpret_cast<double*>(base);
}

static cudaError_t k1t_dispatch(const K1TPlan& p, int nb, K1TArgs& a, const StepArgs& st, cudaStream_t s) {
  a.stages = k1t_stages(p, nb);
  if (a.stages < 2) return cudaErrorInvalidValue;
  const size_t smem = k1t_smem(p, nb);
  return p.storage == GROM_F64 ? k1t_dispatch_f64(p.qm, nb, a, st, p.grid, smem, s)
                               : k1t_dispatch_f32x2(p.qm, nb, a, st, p.grid, smem, s);
}

// c_i = sum over the CTAs whose windows reach i, in CTA order.  A block
// covers 32 test indices of one trajectory; warp w sums CTAs [w G/32, (w+1) G/32).
__global__ void __launch_bounds__(1024) k1t_finish(const K1TArgs a, const int G, const int NB) {
  __shared__ double sh[32][33];
  const int lane = threadIdx.x & 31, warp = threadIdx.x >> 5;
  const int i = blockIdx.x * 32 + lane, bl = blockIdx.y, bg = a.b0 + bl;
  if (a.active && !a.active[bg]) return;  // uniform over the block
  double s = 0.0;
  if (i < a.n)
    for (int g = warp * G / 32; g < (warp + 1) * G / 32; ++g)
      if (k1t_last_group(a.ranges[g]) >= i) s += a.win[((int64_t)g * NB + bl) * a.np + i];
  sh[warp][lane] = s;
  __syncthreads();
  if (warp == 0 && i < a.n) {
    double t = 0.0;
#pragma unroll
    for (int w = 0; w < 32; ++w) t += sh[w][lane];
    double* dst = a.taken ? a.hist + bg * a.hist_stride + (3 + a.taken[bg] % 3) * a.n : a.c + bg * a.c_stride;
    dst[i] = t;
  }
}

cudaError_t k1t_launch(const K1TPlan& p, K1TArgs a, int batch, void* scratch, cudaEvent_t ev0, cudaEvent_t ev1,
                       cudaStream_t s) {
  k1t_fill(p, a, scratch);
  a.nsteps = 0;
  for (int b0 = 0; b0 < batch; b0 += p.nb_max) {
    a.b0 = b0;
    a.nb = std::min(batch - b0, p.nb_max);
    if (ev0 && b0 == 0) prof_record(ev0, s);
    cudaError_t e = k1t_dispatch(p, a.nb, a, StepArgs{}, s);
    if (e != cudaSuccess) return e;
    if (ev1 && b0 + p.nb_max >= batch) prof_record(ev1, s);
    k1t_finish<<<dim3((unsigned)((p.n + 31) / 32), (unsigned)a.nb), 1024, 0, s>>>(a, p.grid, a.nb);
    if ((e = cudaGetLastError()) != cudaSuccess) return e;
  }
  return cudaSuccess;
}

cudaError_t k1tp_launch(const K1TPlan& p, K1TArgs a, const StepArgs& st, int batch, int nsteps, void* scratch,
                        cudaEvent_t ev0, cudaEvent_t ev1, cudaStream_t s) {
  if (batch < 1 || batch > p.nb_max || nsteps < 1) return cudaErrorInvalidValue;
  k1t_fill(p, a, scratch);
  a.b0 = 0;
  a.nb = batch;
  a.nsteps = nsteps;
  if (ev0) prof_record(ev0, s);
  cudaError_t e = k1t_dispatch(p, batch, a, st, s);
  if (e == cudaSuccess && ev1) e = prof_record(ev1, s);
  return e;
}

// ------------------------------------------------------------ conversion
// Group m, row q, position p holds C_pqm + C_pmq (q < m; C_pmp is zero in a
// skew tensor and not read) or C_pmm (q = m).  A block turns a tile of
// T_P test indices p x T_Q rows q x T_M groups m through shared memory: both
// reads run along the tensor's last index, the writes along p.
constexpr int T_P = 16, T_Q = 16, T_M = 8;
__global__ void __launch_bounds__(256) k1t_convert_kernel(const double* __restrict__ src, const int n,
                                                          const int64_t* __restrict__ off, const int i0,
                                                          const int cnt, const int x2, uint8_t* __restrict__ dst) {
  __shared__ double A[T_P][T_Q * T_M + 1], B[T_P][T_M * T_Q + 1];
  const int m0 = blockIdx.x * T_M, q0 = blockIdx.y * T_Q, pl0 = blockIdx.z * T_P;
  if (m0 + T_M - 1 <= i0 + pl0 || q0 > m0 + T_M - 1) return;  // no m > p, or no q <= m (whole block)
  for (int t = threadIdx.x; t < T_P * T_Q * T_M; t += 256) {
    const int mm = t % T_M, qq = t / T_M % T_Q, pp = t / (T_M * T_Q);
    const bool ok = pl0 + pp < cnt && q0 + qq < n && m0 + mm < n;
    A[pp][qq * T_M + mm] = ok ? src[((int64_t)(pl0 + pp) * n + q0 + qq) * n + m0 + mm] : 0.0;
  }
  for (int t = threadIdx.x; t < T_P * T_Q * T_M; t += 256) {
    const int qq = t % T_Q, mm = t / T_Q % T_M, pp = t / (T_M * T_Q);
    const bool ok = pl0 + pp < cnt && q0 + qq < n && m0 + mm < n;
    B[pp][mm * T_Q + qq] = ok ? src[((int64_t)(pl0 + pp) * n + m0 + mm) * n + q0 + qq] : 0.0;
  }
  __syncthreads();
  for (int t = threadIdx.x; t < T_P * T_Q * T_M; t += 256) {
    const int pp = t % T_P, qq = t / T_P % T_Q, mm = t / (T_P * T_Q);
    const int p = i0 + pl0 + pp, q = q0 + qq, m = m0 + mm;
    if (pl0 + pp >= cnt || m >= n || p >= m || q > m) continue;
    double v = A[pp][qq * T_M + mm];
    if (q != m && q != p) v += B[pp][mm * T_Q + qq];
    const int rb = k1t_row_bytes(m);
    uint8_t* row = dst + off[m] + (int64_t)q * rb;
    if (x2) {
      float h, l;
      ds_split(v, h, l);
      reinterpret_cast<float*>(row)[p] = h;
      reinterpret_cast<float*>(row + (rb >> 1))[p] = l;
    } else {
      reinterpret_cast<double*>(row)[p] = v;
    }
  }
}

cudaError_t k1t_convert(const K1TPlan& p, const double* src, int64_t i0, int64_t cnt, uint8_t* dst, cudaStream_t s) {
  const dim3 grid((unsigned)((p.n + T_M - 1) / T_M), (unsigned)((p.n + T_Q - 1) / T_Q), (unsigned)((cnt + T_P - 1) / T_P));
  k1t_convert_kernel<<<grid, 256, 0, s>>>(src, p.n, p.d_off, (int)i0, (int)cnt, p.storage == GROM_F32X2, dst);
  return cudaGetLastError();
}

}  // namespace grom
