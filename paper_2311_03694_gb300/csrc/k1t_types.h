// Plan and arguments of the folded skew-packed layout (k1t.cuh).
#pragma once

#include <cuda_runtime.h>
#include <stdint.h>

#include <vector>

#include "k1_types.h"

namespace grom {

constexpr int K1T_CONSUMERS = 512;              // consumer threads (16 warps)
constexpr int K1T_WARPS = K1T_CONSUMERS / 32;
constexpr int K1T_THREADS = K1T_CONSUMERS + 32;  // + one producer warp
constexpr int K1T_MAX_GRID = 256;  // CTAs whose last groups a stepping CTA tabulates

// Bytes of a row of group m (m >= 1): m values of eight bytes (both storage
// types) padded to a multiple of 128 bytes, so that every copy starts on one.
__host__ __device__ inline int k1t_row_bytes(int m) { return (m + 15) / 16 * 128; }
__host__ __device__ inline int k1t_rows_per_chunk(int row_bytes, int cap) {
  const int r = K1_STAGE_BYTES / row_bytes;
  return r < cap ? r : cap;
}
// The last group of a row range (m0, q0) .. (m1, q1), -1 for an empty one.
__host__ __device__ inline int k1t_last_group(const int4& r) {
  if (r.x > r.z || (r.x == r.z && r.y >= r.w)) return -1;
  return r.w > 0 ? r.z : r.z - 1;
}
// Trajectories a pass can take: accumulators D_p of at most 32 registers.
__host__ __device__ constexpr int k1t_nb_cap(int storage, int qm) {
  return (storage == GROM_F64 ? 8 : 4) / qm > 4 ? 4 : (storage == GROM_F64 ? 8 : 4) / qm;
}
// Whether the sums c_p lie in shared memory: beside many accumulators there
// are no registers for them (F32X2, n = 1024, four trajectories: 1276 us an
// evaluation with them in registers, 1189 in shared memory).
__host__ __device__ constexpr bool k1t_c_shared(int storage, int qm, int nb) {
  return qm * nb >= (storage == GROM_F64 ? 6 : 3);
}
// Rows of a chunk one thread holds: eight 16-byte vectors over its positions and planes.
__host__ __device__ constexpr int k1t_rmax(int storage, int qm, int) {
  const int vectors = (storage == GROM_F64 ? 1 : 2) * qm;
  return 8 / vectors > 0 ? 8 / vectors : 1;
}

struct K1TPlan {
  int n = 0, np = 0, storage = 0;
  int epv = 2;       // elements of a 16-byte vector
  int qm = 1;        // vectors per consumer thread and row
  int nb_max = 1;    // trajectories per pass
  int grid = 1;
  int maxseg = 1;    // groups a CTA touches at most
  size_t bytes = 0;  // stored tensor
  std::vector<int64_t> off;   // n + 1: first byte of group m
  std::vector<int4> ranges;   // grid row ranges (m0, q0, m1, q1)
  int64_t* d_off = nullptr;   // the tables on the device (owned by the ROM)
  int4* d_ranges = nullptr;
};

struct K1TArgs {
  const uint8_t* tensor;
  const int64_t* off;
  const int4* ranges;
  int n, np, stages, maxseg;
  double* part;  // grid x maxseg x K1T_WARPS x NB row sums
  double* win;   // grid x NB x np windows of c
  int nb, b0;    // trajectories of this pass, the first one
  int nsteps;    // 0: one evaluation
  unsigned int* bar;  // grid barrier word (zero at creation)
  double* red;        // grid x NB x 2 energy / invariant partials
  int* err;
  // state: as K1Args
  const double* u;
  int64_t u_stride;
  double* hist;
  const int64_t* taken;
  int64_t hist_stride;
  const int32_t* active;
  double* c;
  int64_t c_stride;
};

K1TPlan k1t_plan(int64_t n, int storage, int sm_count);
size_t k1t_scratch_bytes(const K1TPlan& p);  // barrier word, partials, windows
// Rows [i0, i0 + cnt) of the FP64 tensor into the folded layout (zeroed before).
cudaError_t k1t_convert(const K1TPlan& p, const double* src, int64_t i0, int64_t cnt, uint8_t* dst, cudaStream_t s);
// One evaluation of `batch` trajectories (passes of up to nb_max; ev0 / ev1
// around the streaming kernels when set).
cudaError_t k1t_launch(const K1TPlan& p, K1TArgs a, int batch, void* scratch, cudaEvent_t ev0, cudaEvent_t ev1,
                       cudaStream_t s);

}  // namespace grom
