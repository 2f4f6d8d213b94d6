// cg.cuh — device helpers shared by the two forms of the charge CG: the
// per-iteration kernels (cg.cu) and the whole-solve kernel (cgsolve.cu).
#pragma once
#include <cuda_fp16.h>
#include "internal.cuh"

namespace ct {

// Storage of the block inverses: FP16 on the FP32 path (a fixed symmetric
// preconditioner steers only the iteration count; FP16 halves the largest
// stream of the update pass, 128 of its 176 bytes per atom), FP64 on the
// FP64 path. The stored values are exactly symmetric (see k_block_setup), so
// their FP16 roundings are too, and d = M^-1 1 is summed from the stored
// values.
template <class R> struct BlockStore { using T = R; };
// largest block-inverse entry kept (FP16's largest finite value is 65504)
constexpr double kBlockMax = 6.0e4;
template <> struct BlockStore<float> { using T = __half; };
__device__ inline __half blk_pack(float v) { return __float2half_rn(v); }
__device__ inline double blk_pack(double v) { return v; }
__device__ inline float blk_unpack(__half h) { return __half2float(h); }
__device__ inline double blk_unpack(double v) { return v; }

// y = M_b^-1 r for the warp's block: every lane of a full warp, i = 32b +
// lane, r_i of this lane (zero where no atom). A warp wholly past the last
// atom (the tail of a 256-atom tile) has no block: binv ends at the last
// started one, so such a warp reads nothing.
// The block is stored row by row (row a = element (a, j) for j = 0..31,
// contiguous), so a lane reads its row with 16-byte loads (4 in FP16, 16 in
// FP64; the inverse is symmetric, so the row is also the column).
template <class R>
__device__ inline R block_apply(const typename BlockStore<R>::T* __restrict__ binv, int N, int i, R ri) {
  if ((i & ~31) >= N) return R(0);   // (uniform over the warp)
  using BT = typename BlockStore<R>::T;
  constexpr int NV = 32 * (int)sizeof(BT) / 16;
  const uint4* rp = reinterpret_cast<const uint4*>(binv + (size_t)(i >> 5) * 1024 + (size_t)(i & 31) * 32);
  union {
    uint4 v[NV];
    BT b[32];
  } row;
#pragma unroll
  for (int k = 0; k < NV; ++k) row.v[k] = __ldg(rp + k);   // all in flight
  R y = R(0);
#pragma unroll
  for (int j = 0; j < 32; ++j) y += (R)blk_unpack(row.b[j]) * __shfl_sync(CT_FULL, ri, j);
  return y;
}

// Row sums sum_e M_e v_j(e) of atom i over its column of the list, for one
// or two gathered vectors (NV = 1, 2), plus sum_e M_e (NV = 3). In FP32 the
// products are summed with compensation: a plain FP32 sum of ~230 terms
// whose partial sums are much larger than the result limits the reachable
// residual of the charge solve (about 1e-4 eV/e); compensated, the limit is
// the rounding of the stored entries.
template <class R>
struct RowAcc {
  R s = R(0), c = R(0);
  __device__ inline void add(R x) {
    if (sizeof(R) == 4) {
      R t = s + x;
      c += (fabs(s) >= fabs(x)) ? ((s - t) + x) : ((x - t) + s);
      s = t;
    } else {
      s += x;
    }
  }
  __device__ inline R value() const { return s + c; }
};

}  // namespace ct
