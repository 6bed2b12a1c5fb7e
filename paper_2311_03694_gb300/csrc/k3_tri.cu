// The slice products of K3O (k3_oz.cu) with 7-bit digits (projections over at
// most 1024 modes): all levels of the triangle in one tile.
//
// With eight 7-bit digit slices A_p (128 rows) and B_q (64 columns), level L
// of the result is sum_{p+q=L} A_p B_q^T.  The eight B slices lie one under
// the other in shared memory, so one product A_p [B_0 .. B_{7-p}]^T has its
// blocks side by side in the order of the levels p .. 7: eight level
// accumulators of 64 columns fill the tensor memory and A_p adds to the last
// 64 (8 - p) columns of it, N up to 256 an instruction.  A CTA takes one
// tile and at most 384 of the contracted index: the digits of a level's pairs
// then sum to at most 384 (2 2^13 + 6 2^12) < 2^24, so every FP32 accumulator
// is exact.  The epilogue adds the eight levels with their weights in
// double-single arithmetic, from the smallest up, and writes one (hi, lo)
// pair per output and split, where one product per pair of slices (36 or 45
// values an output, then their sums) took the time of a step.  Steps of n = R
// = 1024, FP64 tolerance: 64 trajectories 63.4 -> 49.6 us, 256 177 -> 145,
// 1024 541 -> 457; n = R = 512, 256 trajectories 80 -> 54.  What bounds it is
// the L2: a K step of 64 is 192 KB of digits for 2304 columns of products
// (projections of 1024 trajectories: 6.4 TB/s there, the tensor pipe 53 % active,
// cold under ncu), and for small batches the round trip of a tile.
#include <algorithm>

#include "ds_arith.cuh"
#include "grom_internal.h"
#include "tc.cuh"

namespace grom {

constexpr int TRI_S = 8;                     // slices
constexpr int TRI_BITS = 7;
constexpr int TRI_COLS = 64;                 // columns of a tile and slice
constexpr int TRI_KMAX = 6;                  // most K steps of 64 a CTA takes
constexpr int TRI_SPLITS = 32;               // most CTAs of a tile for the SMs' sake: 64 planes fit the scratch of 64 products
constexpr int TRI_A_BYTES = 128 * 128;       // one slice of a tile: 128 rows x 64
constexpr int TRI_B_SLICE = TRI_COLS * 128;  // 64 rows x 64
constexpr int TRI_B_BYTES = TRI_S * TRI_B_SLICE;
constexpr int TRI_SA = 6;                    // A ring
constexpr int TRI_SB = 2;                    // B ring
constexpr int TRI_EPI_WARPS = 8;
constexpr int TRI_THREADS = 64 + 32 * TRI_EPI_WARPS;
constexpr size_t TRI_SMEM = 1024 + TRI_SB * TRI_B_BYTES + TRI_SA * TRI_A_BYTES + (2 * TRI_SA + 2 * TRI_SB + 1) * 8 + 16;

struct K3OTri {
  int64_t mslice, nslice;  // rows of an A slice (the output's rows), of a B slice
  int steps, per, splits;  // K steps of 64, of a CTA, CTAs of a tile
  int mtiles, ctiles;
  float* out;  // [split][hi, lo][nslice][mslice]
  int* err;
};

__device__ __forceinline__ void tri_abort(volatile int* abort_flag, int* err) {
  *abort_flag = 1;
  atomicOr(err, DEV_ERR_TIMEOUT);
}

__global__ void __launch_bounds__(TRI_THREADS, 1)
    k3o_tri(const __grid_constant__ CUtensorMap tmap_a, const __grid_constant__ CUtensorMap tmap_b, const K3OTri g) {
  extern __shared__ uint8_t smem_raw[];
  uint8_t* smem = smem_raw + ((1024u - (ptx::smem_addr(smem_raw) & 1023u)) & 1023u);
  uint8_t* sb = smem;
  uint8_t* sa = smem + TRI_SB * TRI_B_BYTES;
  uint64_t* full_a = reinterpret_cast<uint64_t*>(sa + TRI_SA * TRI_A_BYTES);
  uint64_t* empty_a = full_a + TRI_SA;
  uint64_t* full_b = empty_a + TRI_SA;
  uint64_t* empty_b = full_b + TRI_SB;
  uint64_t* done = empty_b + TRI_SB;
  uint32_t* tmem_slot = reinterpret_cast<uint32_t*>(done + 1);
  volatile int* abort_flag = reinterpret_cast<volatile int*>(tmem_slot + 1);
  const int warp = threadIdx.x >> 5, lane = threadIdx.x & 31;
  const int split = blockIdx.x % g.splits, rest = blockIdx.x / g.splits;
  const int ct = rest % g.ctiles, mt = rest / g.ctiles;
  const int k0 = split * g.per, k1 = k0 + g.per < g.steps ? k0 + g.per : g.steps;  // not empty: the host's split

  if (threadIdx.x == 0) {
    for (int s = 0; s < TRI_SA; ++s) {
      ptx::mbar_init(&full_a[s], 1);
      ptx::mbar_init(&empty_a[s], 1);
    }
    for (int s = 0; s < TRI_SB; ++s) {
      ptx::mbar_init(&full_b[s], 1);
      ptx::mbar_init(&empty_b[s], 1);
    }
    ptx::mbar_init(done, 1);
    *abort_flag = 0;
    ptx::fence_mbar_init();
  }
  if (warp == 0 && lane == 0) {
    tc::prefetch_tmap(&tmap_a);
    tc::prefetch_tmap(&tmap_b);
  }
  if (warp == 1) {
    tc::tmem_alloc(tmem_slot, TRI_S * TRI_COLS);
    tc::tmem_relinquish();
  }
  tc::fence_before_sync();
  __syncthreads();
  tc::fence_after_sync();
  const uint32_t tmem = *tmem_slot;
  grid_trigger();

  if (warp == 0) {
    // ---------------------------------------------------------- TMA producer
    if (lane == 0) {
      int ia = 0, ib = 0;  // boxes issued
      bool stop = false;
      auto load_a = [&](int k, int p, int t) {
        ptx::mbar_arrive_expect_tx(&full_a[t], TRI_A_BYTES);
        tc::tma_load_2d(sa + t * TRI_A_BYTES, &tmap_a, k * 64, (int32_t)(p * g.mslice + mt * 128), &full_a[t]);
      };
      // the factors' digits do not depend on the kernels before this one
      for (; ia < TRI_SA; ++ia) load_a(k0, ia, ia);
      grid_wait();
      for (int k = k0; k < k1 && !stop; ++k, ++ib) {
        const int s = ib % TRI_SB;
        if (ib >= TRI_SB && !ptx::mbar_wait(&empty_b[s], (uint32_t)(ib / TRI_SB - 1) & 1u, abort_flag)) {
          tri_abort(abort_flag, g.err);
          break;
        }
        ptx::mbar_arrive_expect_tx(&full_b[s], TRI_B_BYTES);
        for (int q = 0; q < TRI_S; ++q)
          tc::tma_load_2d(sb + s * TRI_B_BYTES + q * TRI_B_SLICE, &tmap_b, k * 64,
                          (int32_t)(q * g.nslice + ct * TRI_COLS), &full_b[s]);
        for (int p = k == k0 ? TRI_SA : 0; p < TRI_S; ++p, ++ia) {
          const int t = ia % TRI_SA;
          if (ia >= TRI_SA && !ptx::mbar_wait(&empty_a[t], (uint32_t)(ia / TRI_SA - 1) & 1u, abort_flag)) {
            tri_abort(abort_flag, g.err);
            stop = true;
            break;
          }
          load_a(k, p, t);
        }
      }
      // every copy lands before the CTA can exit
      for (int q = ia > TRI_SA ? ia - TRI_SA : 0; q < ia; ++q)
        if (!ptx::mbar_wait(&full_a[q % TRI_SA], (uint32_t)(q / TRI_SA) & 1u, nullptr)) atomicOr(g.err, DEV_ERR_TIMEOUT);
      for (int q = ib > TRI_SB ? ib - TRI_SB : 0; q < ib; ++q)
        if (!ptx::mbar_wait(&full_b[q % TRI_SB], (uint32_t)(q / TRI_SB) & 1u, nullptr)) atomicOr(g.err, DEV_ERR_TIMEOUT);
    }
  } else if (warp == 1) {
    // ------------------------------------------------------------ MMA issuer
    if (lane == 0) {
      int ia = 0, ib = 0;
      bool stop = false;
      for (int k = k0; k < k1 && !stop; ++k, ++ib) {
        const int s = ib % TRI_SB;
        if (!ptx::mbar_wait(&full_b[s], (uint32_t)(ib / TRI_SB) & 1u, abort_flag)) {
          tri_abort(abort_flag, g.err);
          break;
        }
        const uint64_t b0 = tc::sw128_kmajor_desc(sb + s * TRI_B_BYTES);
        const uint64_t b1 = tc::sw128_kmajor_desc(sb + s * TRI_B_BYTES + 4 * TRI_B_SLICE);
        for (int p = 0; p < TRI_S; ++p, ++ia) {
          const int t = ia % TRI_SA;
          if (!ptx::mbar_wait(&full_a[t], (uint32_t)(ia / TRI_SA) & 1u, abort_flag)) {
            tri_abort(abort_flag, g.err);
            stop = true;
            break;
          }
          tc::fence_after_sync();
          const uint64_t a = tc::sw128_kmajor_desc(sa + t * TRI_A_BYTES);
          const int n0 = (TRI_S - p < 4 ? TRI_S - p : 4) * TRI_COLS, n1 = (TRI_S - p) * TRI_COLS - n0;
          const uint32_t d0 = tmem + (uint32_t)(p * TRI_COLS);
#pragma unroll
          for (int kk = 0; kk < 4; ++kk) {  // 4 x K = 16 inside the 128-byte swizzle span
            // slice 0 covers every level's columns: it starts the accumulators
            const uint32_t add = ib > 0 || p > 0 || kk > 0 ? 1u : 0u;
            tc::mma_bf16(d0, a + 2 * kk, b0 + 2 * kk, tc::idesc_bf16_f32(128, n0), add);
            if (n1 > 0) tc::mma_bf16(d0 + 256, a + 2 * kk, b1 + 2 * kk, tc::idesc_bf16_f32(128, n1), add);
          }
          tc::commit(&empty_a[t]);
        }
        tc::commit(&empty_b[s]);
      }
      tc::commit(done);  // arrives once every issued MMA has completed
    }
  } else {
    // -------------------------------------------------------------- epilogue
    const int e = warp - 2, lanes = (warp & 3) * 32, half = e / 4;  // 32 rows, 32 of the 64 columns
    if (ptx::mbar_wait(done, 0u, nullptr)) {
      tc::fence_after_sync();
      if (!__any_sync(0xffffffffu, *abort_flag != 0)) {
        const int64_t m = (int64_t)mt * 128 + lanes + lane;
        float* hi = g.out + ((int64_t)split * 2 * g.nslice + ct * TRI_COLS) * g.mslice + m;
        float* lo = hi + g.nslice * g.mslice;
#pragma unroll
        for (int c0 = 0; c0 < 32; c0 += 16) {
          uint32_t v[TRI_S][16];
#pragma unroll
          for (int L = 0; L < TRI_S; ++L)
            tc::tmem_ld_32x32b_x16(tmem + ((uint32_t)lanes << 16) + (uint32_t)(L * TRI_COLS + half * 32 + c0), v[L]);
          tc::tmem_ld_wait();
#pragma unroll
          for (int c = 0; c < 16; c += 2) {  // two columns in packed arithmetic
            f32pair S{0ull}, s{0ull};
#pragma unroll
            for (int L = TRI_S - 1; L >= 0; --L) {
              // x = the level's sum times its weight is exact, so S + x and
              // x - bb in one rounding each are TwoSum's operations
              const float w = __int_as_float((127 - TRI_BITS * (L + 2)) << 23);
              const f32pair x = pair_make(__uint_as_float(v[L][c]), __uint_as_float(v[L][c + 1])), ww = pair_make(w, w);
              const f32pair S1 = pair_fma(x, ww, S), nb = pair_sub(S, S1);
              s = pair_add(s, pair_add(pair_sub(S, pair_add(S1, nb)), pair_fma(x, ww, nb)));
              S = S1;
            }
            const int64_t row = half * 32 + c0 + c;
            float h0, h1, l0, l1;
            pair_get(S, h0, h1);
            pair_get(s, l0, l1);
            hi[row * g.mslice] = h0;
            hi[(row + 1) * g.mslice] = h1;
            lo[row * g.mslice] = l0;
            lo[(row + 1) * g.mslice] = l1;
          }
        }
      }
    } else if (lane == 0) {
      tri_abort(abort_flag, g.err);
    }
  }
  tc::fence_before_sync();
  __syncthreads();
  if (warp == 1) {
    tc::fence_after_sync();
    tc::tmem_dealloc(tmem, TRI_S * TRI_COLS);
  }
}

// ------------------------------------------------------------------- host
// CTAs of a tile: enough for the SMs, at most TRI_KMAX K steps each (the exact
// range of the accumulators), every one with work.
int k3o_tri_splits(int64_t mslice, int64_t nslice, int64_t K, int sm_count) {
  const int64_t steps = K / 64, tiles = mslice / 128 * (nslice / TRI_COLS);
  const int64_t fill = std::min<int64_t>(std::min(steps, sm_count / tiles), TRI_SPLITS);
  const int64_t s = std::max((steps + TRI_KMAX - 1) / TRI_KMAX, fill);
  const int64_t per = (steps + s - 1) / s;
  return (int)((steps + per - 1) / per);
}

static bool tri_tmap(CUtensorMap* m, const void* base, int64_t cols, int64_t rows, int box_rows) {
  auto fn = tmap_encode_fn();
  if (!fn) return false;
  cuuint64_t dims[2] = {(cuuint64_t)cols, (cuuint64_t)rows};
  cuuint64_t strides[1] = {(cuuint64_t)(cols * 2)};
  cuuint32_t box[2] = {64, (cuuint32_t)box_rows};
  cuuint32_t estr[2] = {1, 1};
  return fn(m, CU_TENSOR_MAP_DATA_TYPE_BFLOAT16, 2, const_cast<void*>(base), dims, strides, box, estr,
            CU_TENSOR_MAP_INTERLEAVE_NONE, CU_TENSOR_MAP_SWIZZLE_128B, CU_TENSOR_MAP_L2_PROMOTION_L2_256B,
            CU_TENSOR_MAP_FLOAT_OOB_FILL_NONE) == CUDA_SUCCESS;
}

// A: 8 slices of mslice rows (a multiple of 128), B: 8 slices of nslice rows
// (a multiple of 64), K a multiple of 64, all BF16 digits of 7 bits.
cudaError_t k3o_tri_launch(const void* A, int64_t mslice, const void* B, int64_t nslice, int64_t K, float* out, int* err,
                           int sm_count, cudaStream_t s) {
  if (mslice % 128 || nslice % TRI_COLS || K % 64 || K <= 0) return cudaErrorInvalidValue;
  CUtensorMap ma, mb;
  if (!tri_tmap(&ma, A, K, TRI_S * mslice, 128) || !tri_tmap(&mb, B, K, TRI_S * nslice, TRI_COLS))
    return cudaErrorInvalidValue;
  K3OTri g{};
  g.mslice = mslice;
  g.nslice = nslice;
  g.steps = (int)(K / 64);
  g.splits = k3o_tri_splits(mslice, nslice, K, sm_count);
  g.per = (g.steps + g.splits - 1) / g.splits;
  g.mtiles = (int)(mslice / 128);
  g.ctiles = (int)(nslice / TRI_COLS);
  g.out = out;
  g.err = err;
  cudaError_t e = cudaFuncSetAttribute(k3o_tri, cudaFuncAttributeMaxDynamicSharedMemorySize, (int)TRI_SMEM);
  if (e != cudaSuccess) return e;
  return launch_dependent(k3o_tri, dim3((unsigned)(g.mtiles * g.ctiles * g.splits)), TRI_THREADS, TRI_SMEM, s, ma, mb, g);
}

}  // namespace grom
