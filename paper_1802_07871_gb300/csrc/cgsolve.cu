// cgsolve.cu — the charge minimisation as one kernel per solve, for systems
// whose iteration is bound by latency instead of by streaming the matrix.
//
// The arithmetic is that of the per-iteration kernels (see cg.cu: the
// projected one-reduction CG, its preconditioner, re-centring, starting
// guess and convergence test); what changes is who waits for whom. There an
// iteration is two launches of a graph's WHILE node, each with its tail of
// per-replica atomics, a last-block decision and a cold start: about 40 us
// per iteration at 512 to 20,000 atoms, whatever the work. Here a team of
// blocks stays on the device for the whole solve and meets at two barriers
// per iteration, one for the dots (r.z, w.z), one for the new y and the sums
// that give c and the convergence test.
//
// Two teams:
//   * a thread-block cluster per replica (CL): the cluster's hardware
//     barrier, partial sums exchanged through distributed shared memory, and
//     every block holding the replica's whole y, which the others write into
//     its shared memory. Replicas converge and leave on their own.
//   * all blocks of a cooperative launch on a lone replica: y and the partial
//     sums in global memory, a counter as the barrier (cooperative, so every
//     block is resident; the wait is bounded all the same).
//
// Layout: a block owns up to CS_W groups of 32 consecutive atoms (the
// preconditioner's blocks). Warp g of it holds group g's vectors (r, p, s,
// dq, y, d, v) in registers for the whole solve; in a matrix pass all warps
// work: the rows of a group are cut into S slices of CS_B-entry batches,
// taken by S warps, and the slices' compensated sums meet in shared memory.
//
// Sums are taken in a fixed order (lanes, warps, blocks), so a solve is
// reproducible, and every block forms the same alpha, beta and decision.
#include <algorithm>
#include <cmath>
#include <type_traits>
#include <cooperative_groups.h>

#include "cg.cuh"
#include "kernels.h"

namespace ct {

namespace cgr = cooperative_groups;

#define CS_T 512                 // threads per block
#define CS_W (CS_T / 32)         // warps per block = groups of 32 atoms it can own
#define CS_B 8                   // matrix entries in flight per thread
#define CS_NV 6                  // values of one exchange, at most: pairs of sums, then a pair of maxima
#define CS_GMAX 256              // groups of a cluster (CS_CLMAX * CS_W)
#define CS_CLMAX 16              // blocks of the largest cluster
#define CS_CL_ONE 4096           // atoms of the largest lone replica a cluster solves
#define CS_CUT 2e-6              // how far one FP32 cycle of the FP64 policy takes the residual
#define CS_SPIN (1 << 22)        // polls of a team barrier before it gives up (seconds)

template <class R>
struct SolveArgs {
  int N, ld, Rn;
  const int2* nl;
  const int* nmat;
  const void* M;
  const R *Dg, *dinv, *dvec;
  const typename BlockStore<R>::T* binv;
  const int* type;
  const RepInfo* reps;
  TypeParams T;
  double *q, *h1, *h2;
  R *qr, *y;
  double* cg;
  int *conv, *iters, *it, *hist;
  long long* total;
  unsigned* err;
  double tol;
  int max_iter;
  const double* rhs;
  int* ctl;          // [4], zero between solves: maximum of the iterations, replicas done, blocks gone, arrivals
  double* part;      // [2][CS_NV][gridDim.x]: partial sums of the grid-wide team
  int2* Mf;          // FP64 policy: the matrix once more as FP32 (j, coefficient) pairs, written by each solve
  int maxn;          // atoms of the largest replica (the cluster team's y buffers)
  int per;           // groups a block owns, at most
};

// The block inverses of a thread block's groups stay in shared memory for the
// solve, 16 bytes of a row at a time ([group][chunk][row]: a warp reads a
// chunk of all rows without bank conflicts), as FP16 (mixed policy, as they
// are stored) or FP32 (FP64 policy: rounded alike on both sides of the
// diagonal, so still one symmetric positive definite preconditioner).
template <class R> struct StageType { using T = float; };
template <> struct StageType<float> { using T = __half; };
template <class R> struct BlockChunk {
  using BT = typename StageType<R>::T;
  static constexpr int PER = 16 / (int)sizeof(BT);   // elements of a chunk
  static constexpr int NCH = 32 / PER;               // chunks of a row
};
__device__ inline float blk_unpack(float v) { return v; }
__device__ inline void stage_block(uint4* dst, const __half* __restrict__ binv, int i) {
  const uint4* src = reinterpret_cast<const uint4*>(binv + (size_t)(i >> 5) * 1024 + (size_t)(i & 31) * 32);
#pragma unroll
  for (int c = 0; c < 4; ++c) dst[c * 32 + (i & 31)] = __ldg(src + c);
}
__device__ inline void stage_block(uint4* dst, const double* __restrict__ binv, int i) {
  const double2* src = reinterpret_cast<const double2*>(binv + (size_t)(i >> 5) * 1024 + (size_t)(i & 31) * 32);
#pragma unroll
  for (int c = 0; c < 8; ++c) {
    const double2 a = __ldg(src + 2 * c), b = __ldg(src + 2 * c + 1);
    dst[c * 32 + (i & 31)] = make_uint4(__float_as_uint((float)a.x), __float_as_uint((float)a.y),
                                        __float_as_uint((float)b.x), __float_as_uint((float)b.y));
  }
}
// sum over chunks [c0, c1) of the lane's row times r (of the 32 atoms, in
// shared memory), in F
template <class R, class F>
__device__ inline F chunk_dot(const uint4* blk, const F* r, int c0, int c1) {
  constexpr int PER = BlockChunk<R>::PER;
  F y = F(0);
#pragma unroll 4
  for (int c = c0; c < c1; ++c) {
    union {
      uint4 v;
      typename BlockChunk<R>::BT b[PER];
    } u;
    u.v = blk[c * 32 + (threadIdx.x & 31)];
    union {
      uint4 v[sizeof(F) * PER / 16];
      F x[PER];
    } w;
#pragma unroll
    for (int k = 0; k < (int)sizeof(F) * PER / 16; ++k)
      w.v[k] = reinterpret_cast<const uint4*>(r + c * PER)[k];   // (the same for all lanes)
#pragma unroll
    for (int k = 0; k < PER; ++k) y += (F)blk_unpack(u.b[k]) * w.x[k];
  }
  return y;
}

// Sums of CS_B products at a time: FP32 batches are added as a small tree
// into a compensated sum (as in the streamed matrix pass), FP64 ones by
// fused multiply-adds into four running sums (the FP64 pipe bounds that
// pass: one instruction per entry instead of two).
template <class R> struct PartSum;
template <> struct PartSum<float> {
  RowAcc<float> a;
  __device__ inline void batch(const float (&m)[CS_B], const float (&x)[CS_B]) {
    float t[CS_B];
#pragma unroll
    for (int k = 0; k < CS_B; ++k) t[k] = m[k] * x[k];
#pragma unroll
    for (int w = 1; w < CS_B; w <<= 1)
#pragma unroll
      for (int k = 0; k + w < CS_B; k += 2 * w) t[k] += t[k + w];
    a.add(t[0]);
  }
  __device__ inline float hi() const { return a.s; }
  __device__ inline float lo() const { return a.c; }
};
template <> struct PartSum<double> {
  double s[4] = {0.0, 0.0, 0.0, 0.0};
  __device__ inline void batch(const double (&m)[CS_B], const double (&x)[CS_B]) {
#pragma unroll
    for (int k = 0; k < CS_B; ++k) s[k & 3] = fma(m[k], x[k], s[k & 3]);
  }
  __device__ inline double hi() const { return (s[0] + s[1]) + (s[2] + s[3]); }
  __device__ inline double lo() const { return 0.0; }
};

// Order-preserving map of doubles to unsigned integers: maxima are taken on
// integers (an FP64 maximum costs 97 cycles here).
__device__ inline unsigned long long key_of(double x) {
  const unsigned long long b = (unsigned long long)__double_as_longlong(x);
  return (b >> 63) ? ~b : (b | 0x8000000000000000ull);
}
__device__ inline double of_key(unsigned long long u) {
  const unsigned long long b = (u >> 63) ? (u & 0x7fffffffffffffffull) : ~u;
  return __longlong_as_double((long long)b);
}
__device__ inline unsigned long long shfl_xor_u64(unsigned long long v, int o) {
  return __shfl_xor_sync(CT_FULL, v, o);
}

// Two maxima likewise.
__device__ inline float pair_max(float a, float b) {
  const bool up = (threadIdx.x & 16) != 0;
  float v = fmaxf(up ? b : a, __shfl_xor_sync(CT_FULL, up ? a : b, 16));
#pragma unroll
  for (int o = 8; o > 0; o >>= 1) v = fmaxf(v, __shfl_xor_sync(CT_FULL, v, o));
  return v;
}
__device__ inline double pair_max(double a, double b) {
  const bool up = (threadIdx.x & 16) != 0;
  const unsigned long long ka = key_of(a), kb = key_of(b);
  unsigned long long v = max(up ? kb : ka, shfl_xor_u64(up ? ka : kb, 16));
#pragma unroll
  for (int o = 8; o > 0; o >>= 1) v = max(v, shfl_xor_u64(v, o));
  return of_key(v);
}

// A team and its exchange: NP pairs of sums, then (MX) one pair of maxima,
// over all owner warps of the team into s_tot[0..], the same bits on every
// block. Owner warps bring each pair as pair_sum / pair_max leave it (a value
// per half warp). It is also the team's barrier: what a block wrote before it
// (its y) is visible to the others after it. Every thread calls it.
template <bool CL> struct Team;

// Cluster: an owner warp writes its values straight into every block's
// shared memory, in the slot of its group; the hardware barrier; each block
// sums the slots.
template <> struct Team<true> {
  int rank, size, par = 0;
  double* slots;     // [2][CS_NV][CS_GMAX]
  template <int NP, bool MX>
  __device__ bool exchange(bool own, int slot, int ng, int, const double (&val)[NP + (MX ? 1 : 0)], double* s_tot) {
    constexpr int NE = NP + (MX ? 1 : 0);
    const int lane = threadIdx.x & 31, warp = threadIdx.x >> 5, peer = lane & 15, h = lane >> 4;
    double* base = slots + (size_t)par * CS_NV * CS_GMAX;
    if (own && peer < size) {
      double* dst = cgr::this_cluster().map_shared_rank(base, peer) + slot;
#pragma unroll
      for (int k = 0; k < NE; ++k) dst[(2 * k + h) * CS_GMAX] = val[k];
    }
    cgr::this_cluster().sync();
    if (warp < NE) {   // a warp per pair
      const double* src = base + (2 * warp + h) * CS_GMAX;
      double v;
      if (MX && warp == NP) {
        unsigned long long u = 0ull;
        for (int k = peer; k < ng; k += 16) u = max(u, key_of(src[k]));
#pragma unroll
        for (int o = 8; o > 0; o >>= 1) u = max(u, shfl_xor_u64(u, o));
        v = of_key(u);
      } else {
        v = peer < ng ? src[peer] : 0.0;
        for (int k = peer + 16; k < ng; k += 16) v += src[k];
#pragma unroll
        for (int o = 8; o > 0; o >>= 1) v += __shfl_xor_sync(CT_FULL, v, o);
      }
      if (peer == 0) s_tot[2 * warp + h] = v;
    }
    par ^= 1;
    __syncthreads();
    return true;
  }
};

// Grid: the warps of a block first, then one double per value and block in
// global memory; a counter that thread 0 polls until every block has added
// one (bounded), then each block sums the values of all. (Polling the values
// themselves, with no counter, took 15,000 cycles an exchange at 180 blocks
// against 5,000: every block then reads every block's line all the time.)
template <> struct Team<false> {
  int rank, size, par = 0;
  double* slots;     // [2][CS_NV][size]
  int* counter;
  int target = 0;
  unsigned* err;
  template <int NP, bool MX>
  __device__ bool exchange(bool own, int, int, int G, const double (&val)[NP + (MX ? 1 : 0)], double* s_tot) {
    constexpr int NE = NP + (MX ? 1 : 0), NV = 2 * NE;
    __shared__ double s_red[CS_NV][CS_W];
    __shared__ int s_ok;
    const int lane = threadIdx.x & 31, warp = threadIdx.x >> 5, h = lane >> 4;
    double* base = slots + ((size_t)par * CS_NV + warp) * size;
    const bool mx = MX && warp >= 2 * NP;
    if (own && (lane & 15) == 0) {
#pragma unroll
      for (int k = 0; k < NE; ++k) s_red[2 * k + h][warp] = val[k];
    }
    __syncthreads();
    if (warp < NV) {   // a warp per value
      double v = lane < G ? s_red[warp][lane] : (mx ? -INFINITY : 0.0);
      if (mx) {
        unsigned long long u = key_of(v);
#pragma unroll
        for (int o = 8; o > 0; o >>= 1) u = max(u, shfl_xor_u64(u, o));
        v = of_key(u);
      } else {
#pragma unroll
        for (int o = 8; o > 0; o >>= 1) v += __shfl_xor_sync(CT_FULL, v, o);
      }
      if (lane == 0) __stcg(base + rank, v);
    }
    __syncthreads();
    target += size;
    if (threadIdx.x == 0) {
      __threadfence();   // the block's values and y before its count
      atomicAdd(counter, 1);
      int n = 0, ok = 1;
      for (;;) {
        int c;
        asm volatile("ld.acquire.gpu.global.s32 %0, [%1];" : "=r"(c) : "l"(counter) : "memory");
        if (c >= target) break;
        if (++n > CS_SPIN) {   // a block of the team is gone: give up (reported to the host)
          atomicOr(err, CT_ERR_SOLVER);
          ok = 0;
          break;
        }
      }
      s_ok = ok;
    }
    __syncthreads();   // (orders the block's loads after thread 0's acquire)
    if (warp < NV) {
      double v = mx ? -INFINITY : 0.0;
      unsigned long long u = key_of(v);
      for (int b = lane; b < size; b += 32) {
        const double x = __ldcg(base + b);
        if (mx) u = max(u, key_of(x)); else v += x;
      }
      if (mx) {
#pragma unroll
        for (int o = 16; o > 0; o >>= 1) u = max(u, shfl_xor_u64(u, o));
        v = of_key(u);
      } else {
        v = warp_sum(v);
      }
      if (lane == 0) s_tot[warp] = v;
    }
    par ^= 1;
    __syncthreads();
    return s_ok != 0;
  }
};

template <class R, bool CL>
__global__ void __launch_bounds__(CS_T, CL && sizeof(R) == 4 ? 2 : 1) k_cg_solve(const SolveArgs<R> A) {
  extern __shared__ __align__(16) unsigned char smem_raw[];
  __shared__ double s_slots[CL ? 2 * CS_NV * CS_GMAX : 1];
  __shared__ double s_tot[CS_NV];
  __shared__ R s_hi[3][CS_W][32];
  __shared__ float s_lo[sizeof(R) == 4 ? 3 : 1][CS_W][32];   // (compensations: FP32 sums only)
  __shared__ __align__(16) R s_r[CS_W][32];
  // Words of the scalars, all written by the boss thread alone. A word is read
  // only after the first __syncthreads past its store, and stored again only
  // after an exchange that every reader of the old value entered (an exchange
  // is a barrier of the block too):
  __shared__ double s_abc[2];   // alpha, beta: stored after the dots' exchange; c, mean: after that of y's sums
  __shared__ int s_stop;        // max |r - mean| met the goal: stored after the exchange of y's sums
  __shared__ int s_fell;        // (FP64) the residual fell tenfold: stored with a cycle's first s_stop
  __shared__ double s_shift;    // (FP64) the shift with the mean: stored after the CG of a cycle
  // (s_tot: stored by the exchanges between two of their own barriers, read by
  // any thread after an exchange and before it enters the next)
  const int lane = threadIdx.x & 31, warp = threadIdx.x >> 5;
  // the thread that forms the scalars: of the last warp, which owns no group
  // unless the block has all it can, so its divisions run beside the update
  const bool boss = threadIdx.x == CS_T - 32;
  Team<CL> T;
  if constexpr (CL) {
    T.rank = (int)cgr::this_cluster().block_rank();
    T.size = (int)cgr::this_cluster().num_blocks();
    T.slots = s_slots;
    cgr::this_cluster().sync();   // every block is running: its shared memory may be written
  } else {
    T.rank = blockIdx.x;
    T.size = gridDim.x;
    T.slots = A.part;
    T.counter = A.ctl + 3;
    T.err = A.err;
  }
  uint4* s_blk = reinterpret_cast<uint4*>(smem_raw);   // [per][chunks][32]: block inverses
  constexpr int NCH = BlockChunk<R>::NCH;
  R* yb0 = reinterpret_cast<R*>(s_blk + (A.binv ? (size_t)A.per * NCH * 32 : 0));   // cluster team: the replica's q,
  R* yb1 = yb0 + A.maxn;                               // and its y, both written by every block of the cluster
  // (one replica either way: the plan gives the grid lone ones. Compiled without
  // the loop the FP64 grid took 2% more on a slab of 19,548 atoms, 716 -> 733 us, and
  // 3% less on a crystal of 18,928, 643 -> 626)
  const int r_first = CL ? (int)(blockIdx.x / T.size) : 0, r_end = CL ? r_first + 1 : A.Rn;
  const int nh = *A.hist;
  bool alive = true;
  for (int rr = r_first; rr < r_end && alive; ++rr) {
    double* cc = A.cg + (size_t)rr * CG_STRIDE;
    const int a0 = A.reps[rr].atom_off, n = A.reps[rr].natoms;
    int its = 0, total = 0, conv = 0;   // iterations of this CG, of the ones before it
    if (n == 0) {
      if (T.rank == 0 && threadIdx.x == 0) cc[CG_RESMAX] = cc[CG_RES0] = INFINITY;
      conv = 1;
    } else {
      // this block's groups of the replica and this warp's unit of a pass
      const int g0 = a0 >> 5, ng = ((a0 + n - 1) >> 5) - g0 + 1;
      const int per = (ng + T.size - 1) / T.size;
      const int gb = min(T.rank * per, ng), G = min(gb + per, ng) - gb;
      const int S = G > 0 ? CS_W / G : 0;                 // slices of a row
      const int ug = G > 0 ? warp % G : 0, us = G > 0 ? warp / G : 0;
      const bool unit = G > 0 && us < S, own = warp < G;
      const int iu = (g0 + gb + ug) * 32 + lane;          // the atom of the unit's row
      const bool inu = unit && iu >= a0 && iu < a0 + n;
      const int nau = inu ? A.nmat[iu] : 0;
      const int nwu = (int)__reduce_max_sync(CT_FULL, (unsigned)nau);
      const int nfu = (int)__reduce_min_sync(CT_FULL, (unsigned)nau);
      const int i = (g0 + gb + warp) * 32 + lane;         // the atom this lane owns
      const bool in = own && i >= a0 && i < a0 + n;
      const MatView<R> mat(A.nl, A.M);
      const double inv_n = 1.0 / (double)n;
      // a batch of the unit's row; past its end, zero coefficients on the
      // replica's first atom
      auto entry = [&](size_t o, int& j, auto& m) {
        if constexpr (sizeof(m) == sizeof(R)) {
          mat.get(o, j, m);
        } else {   // (written by this thread in the first cycle: a plain load)
          const int2 t = A.Mf[o];
          j = t.x;
          m = __int_as_float(t.y);
        }
      };
      auto fetch = [&](int e0, int (&j)[CS_B], auto (&m)[CS_B]) {
        const size_t o = (size_t)e0 * A.ld + iu;
        if (e0 + CS_B <= nfu) {
#pragma unroll
          for (int k = 0; k < CS_B; ++k) entry(o + (size_t)k * A.ld, j[k], m[k]);
        } else {
#pragma unroll
          for (int k = 0; k < CS_B; ++k) {
            j[k] = a0;
            m[k] = 0;
            if (e0 + k < nau) entry(o + (size_t)k * A.ld, j[k], m[k]);
          }
        }
      };
      // partial row sums of the unit over one vector, into s_hi/s_lo[slot],
      // and the row sum of this warp's own group from them
      auto put = [&](int slot, auto hi, auto lo) {
        using F = decltype(hi);
        reinterpret_cast<F(*)[32]>(&s_hi[slot][0][0])[warp][lane] = hi;
        if (sizeof(F) == 4) s_lo[slot][warp][lane] = (float)lo;
      };
      auto take = [&](int slot, auto zero) {
        using F = decltype(zero);
        auto hi = reinterpret_cast<F(*)[32]>(&s_hi[slot][0][0]);
        RowAcc<F> a[4];   // (four chains: the additions wait for one another)
        F c = F(0);
        for (int k = 0; k < S; k += 4) {
#pragma unroll
          for (int m = 0; m < 4; ++m)
            if (k + m < S) {
              a[m].add(hi[(k + m) * G + warp][lane]);
              if (sizeof(F) == 4) c += (F)s_lo[slot][(k + m) * G + warp][lane];
            }
        }
        a[0].add(a[1].s);
        a[2].add(a[3].s);
        a[0].add(a[2].s);
        if (sizeof(F) == 4) c += (a[1].c + a[3].c) + a[2].c;
        return sizeof(F) == 4 ? a[0].s + (a[0].c + c) : a[0].s;
      };
      // y = M^-1 r of the block's groups. FP32: a warp per group. FP64: a
      // group's 32 additions at 64 cycles each are shared by up to four
      // warps (one per scheduler).
      const int SA = G > 0 ? min(4, CS_W / G) : 0;
      auto precond = [&](auto r) {
        using F = decltype(r);
        F* sr = reinterpret_cast<F*>(&s_r[warp][0]);
        if (!A.binv) return in ? (F)A.dinv[i] * r : F(0);
        if (own) sr[lane] = in ? r : F(0);
        F y = F(0);
        if constexpr (sizeof(F) == 4) {
          __syncwarp();
          if (own) y = chunk_dot<R, F>(s_blk + warp * NCH * 32, sr, 0, NCH);
          __syncwarp();
        } else {
          __syncthreads();
          if (warp < SA * G)
            s_hi[1][warp][lane] = chunk_dot<R, F>(s_blk + ug * NCH * 32, reinterpret_cast<F*>(&s_r[ug][0]),
                                                  NCH * us / SA, NCH * (us + 1) / SA);
          __syncthreads();
          if (own)
            for (int k = 0; k < SA; ++k) y += s_hi[1][k * G + warp][lane];
        }
        return y;
      };
      if (own && A.binv) stage_block(s_blk + warp * NCH * 32, A.binv, i);
      __syncthreads();
      // one vector to the whole team
      auto share = [&](R* buf, R* glob, auto v) {
        using F = decltype(v);
        if constexpr (CL) {
          for (int p = 0; p < T.size; ++p) reinterpret_cast<F*>(cgr::this_cluster().map_shared_rank(buf, p))[i - a0] = v;
        } else {
          reinterpret_cast<F*>(glob)[i] = v;
        }
      };
      auto exchange1 = [&](double v) {   // a single FP64 sum
        const double val[1] = {own ? pair_sum(v, 0.0) : 0.0};   // (idle warps issue no FP64)
        return T.template exchange<1, false>(own, gb + warp, ng, G, val, s_tot);
      };
      // sums of y, r (and d) and the extremes of r over the team
      auto exchange_y = [&](auto first, auto yi, auto ri, auto di) {
        using F = decltype(yi);
        constexpr int NP = decltype(first)::value ? 2 : 1;
        double val[NP + 1] = {};
        if (own) {
          const F none = -F(INFINITY);
          val[0] = (double)pair_sum(in ? yi : F(0), in ? ri : F(0));
          if (NP == 2) val[1] = (double)pair_sum(in ? di : F(0), F(0));
          val[NP] = (double)pair_max(in ? ri : none, in ? -ri : none);
        }
        return T.template exchange<NP, true>(own, gb + warp, ng, G, val, s_tot);
      };
      // ---- starting guess
      double qi = 0.0;
      if (in) {
        const double qo = A.q[i], x1 = A.h1[i], x2 = A.h2[i];
        if (nh >= 3) qi = 3.0 * qo - 3.0 * x1 + x2;
        else if (nh == 2) qi = 2.0 * qo - x1;
        else if (nh == 1) qi = qo;
        A.h2[i] = x1;
        A.h1[i] = qo;
      }
      const double mp = cc[CG_MU];
      double shift = isfinite(mp) ? -mp : 0.0;   // subtracted from every stored r
      double mean = 0.0, bound = 0.0, res0 = 0.0, inv_sd = 0.0;
      R Di = R(0), di = R(0), vi = R(0), hm = R(0);
      double chi = 0.0;
      if (in) {
        Di = A.Dg[i];
        di = A.dvec[i];
        chi = A.rhs ? A.rhs[i] : by_type(A.T.chi, A.type[i]);
      }
      auto test = [&](double sy, double sr, double hi, double lo, double tol) {   // (the boss)
        mean = sr * inv_n;
        const double bh = hi - mean, bl = lo + mean;
        bound = of_key(max(key_of(bh), key_of(bl)));   // max_i |r_i - mean|
        if (!isfinite(bh) || !isfinite(bl)) bound = INFINITY;
        s_abc[0] = sy * inv_sd;
        s_abc[1] = mean;
        s_stop = key_of(bound) <= key_of(tol) ? 1 : 0;
      };
      // The CG in F from the residual ri (y = M^-1 r shared, its sums in
      // s_abc), adding to dq, until max |r - mean| <= goal (the boss's; then
      // `done`) or max_iter iterations are used up. The cap is that of one CG:
      // the cycles of the FP64 policy each have it, because a CG that starts
      // anew for every few digits takes more iterations in all than one that
      // runs through (7 -> 11, 37 -> 44, 45 -> 50, 53 -> 55 from no charges), and
      // what converged under a cap in one run has to converge under it here.
      // Every block takes the same decisions.
      int done = 1;
      auto iterate = [&](auto ri, auto yi, double goal, double& dq) -> bool {
        using F = decltype(ri);
        const F D = (F)Di, d = (F)di, v = (F)vi;
        F pi = F(0), si = F(0), dqi = F(0);
        double gp = 0.0, ap = 0.0, inv_gp = 0.0, inv_ap = 0.0;
        F cR = (F)s_abc[0], mprev = (F)s_abc[1];
        int stop = 0;
        const F* yb = reinterpret_cast<const F*>(yb1);
        const F* yg = reinterpret_cast<const F*>(A.y);
        while (!stop && its < A.max_iter) {
          // ---- w = H z = H y - c v, z = y - c d, and the dots r.z, w.z
          if (unit) {
            PartSum<F> p0;
            // the next batch is in flight while this one's y are gathered,
            // but in the FP32 cluster team: two blocks per SM hide that
            // latency there, and 64 registers leave no room for a second batch
            constexpr bool AHEAD = !(CL && sizeof(R) == 4);
            int j[CS_B];
            F m[CS_B];
            if (AHEAD) fetch(us * CS_B, j, m);
            for (int e0 = us * CS_B; e0 < nwu; e0 += S * CS_B) {
              F x0[CS_B];
              if (!AHEAD) fetch(e0, j, m);
#pragma unroll
              for (int k = 0; k < CS_B; ++k) x0[k] = CL ? yb[j[k] - a0] : yg[j[k]];
              if (AHEAD) {
                F mc[CS_B];
#pragma unroll
                for (int k = 0; k < CS_B; ++k) mc[k] = m[k];
                fetch(e0 + S * CS_B, j, m);
                p0.batch(mc, x0);
              } else {
                p0.batch(m, x0);
              }
            }
            put(0, p0.hi(), p0.lo());
          }
          __syncthreads();
          F wi = F(0), zi = F(0);
          double val[1] = {0.0};
          if (own) {
            F d0 = F(0), d1 = F(0);
            if (in) {
              zi = yi - cR * d;
              wi = D * yi + take(0, F(0)) - cR * v;
              d0 = (ri - mprev) * zi;
              d1 = wi * zi;
            }
            val[0] = (double)pair_sum(d0, d1);
          }
          if (!T.template exchange<1, false>(own, gb + warp, ng, G, val, s_tot)) return false;
          if (boss) {
            // beta = g / g_prev, alpha = g / (w.z - beta g / alpha_prev)
            const double g = s_tot[0], b = g * inv_gp;
            double den = s_tot[1];
            if (ap != 0.0) den -= b * g * inv_ap;
            const double a = den != 0.0 ? g * inv(den) : 0.0;
            s_abc[0] = a;
            s_abc[1] = b;
            shift += (double)mprev;   // the mean this update subtracts
            gp = g;
            ap = a;
            inv_ap = den;             // (times 1 / g below)
          }
          __syncthreads();
          const F a = (F)s_abc[0], b = (F)s_abc[1];
          if (boss) {   // off the critical path: for the next beta and alpha
            inv_gp = gp != 0.0 ? inv(gp) : 0.0;
            inv_ap *= inv_gp;
          }
          if (in) {
            pi = zi + b * pi;
            si = wi + b * si;
            ri = (ri - a * si) - mprev;
            dqi += a * pi;
          }
          yi = precond(ri);
          if (in) share(yb1, A.y, yi);
          if (!exchange_y(std::false_type(), yi, ri, yi)) return false;
          if (boss) test(s_tot[0], s_tot[1], s_tot[2], s_tot[3], goal);
          ++its;
          __syncthreads();
          stop = s_stop;
          cR = (F)s_abc[0];
          mprev = (F)s_abc[1];
        }
        dq += (double)dqi;
        done = stop;
        return true;
      };
      // A cycle: the residual of q shifted onto sum q = Q, in R, then the CG
      // from it. The mixed policy takes one, down to its tolerance. The FP64
      // policy refines: its matrix passes are bound by the FP64 pipe, so the
      // CG runs in FP32 on the FP64 residual, for as many digits as FP32
      // rounding allows (CS_CUT), and the next cycle's FP64 residual decides,
      // the one that must meet the tolerance (19,555 atoms: 756 us in 43
      // iterations against 1,005 in 38 with the CG in FP64; the charges end
      // nearer the minimiser than by the recursion's residual). Should a cycle gain less than a
      // digit, the CG goes on in FP64, to the tolerance by its own recursion (a
      // tolerance at the FP64 residual's rounding can be met that way only).
      double last = 1e308;
      bool final_shift = false;
      for (int cycle = 0;; ++cycle) {
        if (in) share(yb0, A.qr, (R)qi);
        if (!exchange1(qi)) { alive = false; break; }
        const double dq0 = (cc[CG_Q] - s_tot[0]) * inv_n;
        if (unit) {
          if (cycle == 0) {   // with H d and the row sum of H for the shifts
            PartSum<R> p0, p1, p2;
            for (int e0 = us * CS_B; e0 < nwu; e0 += S * CS_B) {
              int j[CS_B];
              R m[CS_B], x0[CS_B], x1[CS_B], one[CS_B];
              fetch(e0, j, m);
#pragma unroll
              for (int k = 0; k < CS_B; ++k) {
                x0[k] = CL ? yb0[j[k] - a0] : A.qr[j[k]];
                x1[k] = A.dvec[j[k]];
                one[k] = R(1);
                if (sizeof(R) == 8 && e0 + k < nau)
                  A.Mf[(size_t)(e0 + k) * A.ld + iu] = make_int2(j[k], __float_as_int((float)m[k]));
              }
              p0.batch(m, x0);
              p1.batch(m, x1);
              p2.batch(m, one);
            }
            put(0, p0.hi(), p0.lo());
            put(1, p1.hi(), p1.lo());
            put(2, p2.hi(), p2.lo());
          } else {
            PartSum<R> p0;
            for (int e0 = us * CS_B; e0 < nwu; e0 += S * CS_B) {
              int j[CS_B];
              R m[CS_B], x0[CS_B];
              fetch(e0, j, m);
#pragma unroll
              for (int k = 0; k < CS_B; ++k) x0[k] = CL ? yb0[j[k] - a0] : A.qr[j[k]];
              p0.batch(m, x0);
            }
            put(0, p0.hi(), p0.lo());
          }
        }
        __syncthreads();
        R ri = R(0);
        if (in) {
          const R hq = take(0, R(0));
          if (cycle == 0) {
            vi = Di * di + take(1, R(0));
            hm = take(2, R(0));
          }
          // q shifted by dq0: H (q + dq0 1) = D (q + dq0) + sum M q_j + dq0 sum M
          qi += dq0;
          ri = (R)(-chi - ((double)Di * qi + (double)hq + dq0 * (double)hm) - shift);
        }
        // (FP32: what the CG starts from; every block's `shift` is the boss's)
        float yf = precond((float)ri);
        if (in) share(yb1, A.y, yf);
        const bool ok = cycle == 0 ? exchange_y(std::true_type(), (R)yf, ri, di) : exchange_y(std::false_type(), (R)yf, ri, di);
        if (!ok) { alive = false; break; }
        if (boss) {
          if (cycle == 0) {
            inv_sd = s_tot[2] != 0.0 ? 1.0 / s_tot[2] : 0.0;
            test(s_tot[0], s_tot[1], s_tot[4], s_tot[5], A.tol);
            res0 = bound;
          } else {
            test(s_tot[0], s_tot[1], s_tot[2], s_tot[3], A.tol);
          }
          if constexpr (sizeof(R) == 8) {
            s_fell = bound <= 0.1 * last ? 1 : 0;   // (0 if it is not finite)
            last = bound;
          }
        }
        __syncthreads();
        conv = s_stop;
        // (uniform: the word stays until the next exchange)
        if (conv || !done) break;
        double dq = 0.0;
        bool go;
        total += its;
        its = 0;
        if constexpr (sizeof(R) == 4) {
          go = iterate(ri, yf, A.tol, dq);
          qi += dq;
          conv = done;
          final_shift = true;
          if (!go) alive = false;
          break;
        } else {
          const bool fell = s_fell != 0;
          if (fell) {
            go = iterate((float)ri, yf, fmax(0.3 * A.tol, bound * CS_CUT), dq);
          } else {
            const double yd = precond((double)ri);
            if (in) share(yb1, A.y, yd);
            go = exchange_y(std::false_type(), yd, ri, yd);
            if (go) {
              if (boss) test(s_tot[0], s_tot[1], s_tot[2], s_tot[3], A.tol);
              __syncthreads();
              go = iterate((double)ri, yd, A.tol, dq);
            }
          }
          qi += dq;
          if (!go) { alive = false; break; }
          if (!fell) {
            conv = done;
            final_shift = true;
            break;
          }
          // the mean is part of the shift from here on (the boss's, to all)
          if (boss) {
            shift += mean;
            s_shift = shift;
          }
          __syncthreads();
          shift = s_shift;
        }
      }
      if (!alive) break;
      // ---- the charges, after a CG in R once more onto sum q = Q
      if (final_shift) {
        if (!exchange1(qi)) { alive = false; break; }
        qi += (cc[CG_Q] - s_tot[0]) * inv_n;
      }
      if (in) {
        A.q[i] = qi;
        A.qr[i] = (R)qi;
      }
      if (T.rank == 0 && boss) {
        cc[CG_M] = mean;
        cc[CG_SHIFT] = shift;
        cc[CG_RESMAX] = bound;
        cc[CG_RES0] = res0;
        // (CG_MU is read by every block at the replica's start, before the last exchanges)
        cc[CG_MU] = -(mean + shift);
      }
    }
    if (T.rank == 0 && threadIdx.x == 0) {
      its += total;   // all of them
      A.conv[rr] = conv;
      A.iters[rr] = its;
      if (!conv) atomicOr(A.err, CT_ERR_CG_MAXITER);
      atomicMax(A.ctl, its);
      __threadfence();
      if (atomicAdd(A.ctl + 1, 1) == A.Rn - 1) {   // the solve is over
        __threadfence();
        const int m = atomicExch(A.ctl, 0);
        A.ctl[1] = 0;
        *A.it = m;
        *A.total += m;
        const int h = *A.hist;
        *A.hist = h < 3 ? h + 1 : 3;
      }
    }
  }
  if constexpr (!CL) {   // the last block to leave clears the counter for the next solve
    __syncthreads();
    if (threadIdx.x == 0) {
      __threadfence();
      if (atomicAdd(A.ctl + 2, 1) == (int)gridDim.x - 1) A.ctl[2] = A.ctl[3] = 0;
    }
  }
}

// ---------------------------------------------------------------- launchers
// Dynamic shared memory of a block: its groups' block inverses, and the
// cluster team's two vectors.
template <class R, bool CL>
static size_t solve_smem(int per, int maxn, int precond) {
  return (precond ? (size_t)per * 1024 * sizeof(typename BlockChunk<R>::BT) : 0) + (CL ? 2 * (size_t)maxn * sizeof(R) : 0);
}

template <class R, bool CL>
static cudaError_t launch_solve(const DevState& S, const SolveArgs<R>& A, cudaStream_t st) {
  cudaLaunchConfig_t cfg = {};
  cfg.gridDim = dim3((unsigned)(CL ? S.R * S.solve_blocks : S.solve_blocks));
  cfg.blockDim = dim3(CS_T);
  cfg.dynamicSmemBytes = solve_smem<R, CL>(S.solve_per, A.maxn, S.precond);
  cfg.stream = st;
  cudaLaunchAttribute at[1];
  if (CL) {
    at[0].id = cudaLaunchAttributeClusterDimension;
    at[0].val.clusterDim.x = (unsigned)S.solve_blocks;
    at[0].val.clusterDim.y = at[0].val.clusterDim.z = 1;
  } else {
    at[0].id = cudaLaunchAttributeCooperative;
    at[0].val.cooperative = 1;
  }
  cfg.attrs = at;
  cfg.numAttrs = 1;
  return cudaLaunchKernelEx(&cfg, k_cg_solve<R, CL>, A);
}

template <class R>
cudaError_t launch_cg_solve(const DevState& S, const TypeParams& T, double tol, int max_iter, const double* rhs,
                            cudaStream_t st) {
  SolveArgs<R> A;
  A.N = S.N; A.ld = S.ld; A.Rn = S.R;
  A.nl = S.nl; A.nmat = S.nmat; A.M = S.M;
  A.Dg = (const R*)S.Dg; A.dinv = (const R*)S.dinv;
  A.dvec = (const R*)(S.precond ? S.bsum : S.dinv);
  A.binv = S.precond ? (const typename BlockStore<R>::T*)S.binv : nullptr;
  A.type = S.type; A.reps = S.reps; A.T = T;
  A.q = S.q; A.h1 = S.cqh1; A.h2 = S.cqh2;
  A.qr = (R*)S.qr; A.y = (R*)S.cy;
  A.cg = S.cg; A.conv = S.cg_conv; A.iters = S.cg_iters; A.it = S.cg_it; A.hist = S.cg_hist; A.total = S.cg_total;
  A.err = S.err; A.tol = tol; A.max_iter = max_iter; A.rhs = rhs;
  A.ctl = S.solve_ctl; A.part = S.solve_part; A.maxn = S.solve_maxn; A.per = S.solve_per; A.Mf = S.Mf;
  return S.solver == SOLVE_CLUSTER ? launch_solve<R, true>(S, A, st) : launch_solve<R, false>(S, A, st);
}

// Whether a batch's clusters beat its launches, by an estimate of the time of an
// iteration in microseconds. All clusters have the size that the largest
// replica wants, `fit` of them run at a time (7 to 14 of 16 blocks), and a small
// replica in a large cluster costs almost as much as a large one, its two
// barriers; so the clusters take one wave of replicas after another, and the
// launches their tails plus the stream of the matrix. Replicas of different size
// also converge at different times: 0.6 of the iterations on average.
// Measured, microseconds per MD step in clusters and by launches:
//   mixed, even: 4, 12, 16, 24 x 8,000 atoms 362 and 502, 812 and 873, 1,152 and
//   1,056, 1,630 and 1,426; 24, 48, 57 x 4,096 750 and 881, 1,454 and 1,499, 1,589
//   and 1,556; 200 x 1,000 1,171 and 1,325; 1,000 x 64 433 and 618;
//   mixed, uneven: 96 replicas of 200 to 3,000 atoms 1,360 and 1,507; 4,096 + 20 x 64
//   209 and 375, + 100 x 64 392 and 388, + 1,000 x 64 2,884 and 782; 8,000 + 500 x 8
//   1,500 and 422; 4,096 + 100 x 512 720 and 611; 1,728 + 500 x 64 425 and 471;
//   FP64: 128 x 1,000 7,915 and 11,677; 4,096 + 100 x 64 2,770 and 2,776, + 1,000 x 64
//   23,362 and 6,597; 1,728 + 500 x 64 3,621 and 4,089.
static bool clusters_pay(bool fp32, int R, int N, double maxn, int size, int fit, int nsm, double row) {
  const double mean = (double)N / R, some = maxn > 1.25 * mean ? 0.6 : 1.0;
  const double barriers = 2.5 + 0.4 * size;
  const double per_atom = 0.036 * std::max((double)fit * size / nsm, 1.0);   // of a block's share; blocks share an SM
  const double waves = std::ceil((double)R / fit);
  const double clusters = std::max(some * waves * (barriers + per_atom * mean / size), barriers + per_atom * maxn / size);
  const double launches = (fp32 ? 35.0 : 66.0) + some * N * row / (fp32 ? 5.2e6 : 2.7e6);
  return clusters < launches;
}

// Which form of the solve a system takes. The whole-solve kernel pays where
// an iteration's time is its launches and tails; where it is the streaming
// of a matrix larger than L2, the per-iteration kernels (every SM, whole
// rows, deep pipelines) are the better form.
//   * replicas of at most CS_CLMAX * CS_W groups of 32 atoms: a cluster
//     each, as large as gives every block work and fills the chip, and large
//     enough that the matrices of the replicas running together stay in L2
//     (a lone replica up to CS_CL_ONE atoms: past that the whole chip's
//     bandwidth and FP64 rate outweigh the cluster's cheaper barrier). Not
//     past 3.5 L2 budgets of matrix in all: 96 replicas, 158,000 atoms take
//     45 us per iteration in clusters against 55 by launches, 288 replicas,
//     1.25 million atoms 0.57 ms against 0.33 (past the line clusters still
//     win with small replicas, 500 x 512 atoms 1,276 us per step against
//     1,557, 4,000 x 64 1,386 against 1,809, and lose with large ones, 72 x
//     4,096 2,011 against 1,903). And not where clusters_pay says that the
//     launches are faster;
//   * one larger replica whose matrix fits L2: the grid-wide team;
//   * anything else: the per-iteration kernels.
// Solve times, microseconds per MD step by launches and with this kernel:
// FP64, 64 atoms 1,000 -> 149 (18 -> 21 iterations, see k_cg_solve's cycles),
// 512 atoms 1,950 -> 240 (31 -> 34), 19,555 atoms 2,820 -> 756 (38 -> 43);
// mixed, 11,491 atoms 520 -> 160 (11), 32 configurations of 64-512 atoms
// 840 -> 140 (20).
template <class R>
cudaError_t plan_cg_solve(DevState& S, const int64_t* off) {
  S.solver = SOLVE_LAUNCHES;
  S.solve_blocks = S.solve_per = S.solve_maxn = 0;
  if (S.N == 0) return cudaSuccess;
  int64_t maxn = 0;
  for (int r = 0; r < S.R; ++r) maxn = std::max(maxn, off[r + 1] - off[r]);
  const int ng = (int)(maxn / 32) + 2;   // groups a replica can touch
  // stored entries per atom: the list's capacity less its headroom and skin
  const double row = 0.65 * S.cap_all * (sizeof(R) == 4 ? 8.0 : 12.0);
  const double l2 = 100e6;
  size_t most_smem = 0;
  cudaError_t e = cudaSuccess;
  const bool many = S.R > 1;
  if (ng <= CS_CLMAX * CS_W && (many ? (double)S.N * row <= 3.5 * l2 : maxn <= CS_CL_ONE)) {
    e = allow_dynamic_smem((const void*)k_cg_solve<R, true>, &most_smem);
    if (e == cudaSuccess)
      e = cudaFuncSetAttribute(k_cg_solve<R, true>, cudaFuncAttributeNonPortableClusterSizeAllowed, 1);
    if (e != cudaSuccess) return e;
    const double mean = (double)S.N / S.R;
    const int slots = S.nsm * (sizeof(R) == 4 ? 2 : 1);
    int size = 1;
    while (size < CS_CLMAX &&
           (ng > size * CS_W ||                                         // every group has a warp
            (size * 2 <= (int)(mean / 32) + 1 &&                        // every block has groups
             ((double)S.R * size < slots ||                             // fill the chip
              slots / size * std::min(mean, (double)maxn) * row > l2))))   // matrices in L2 together
      size *= 2;
    cudaLaunchConfig_t cfg = {};
    cfg.gridDim = dim3((unsigned)(S.R * size));
    cfg.blockDim = dim3(CS_T);
    const int per = (ng + size - 1) / size;
    cfg.dynamicSmemBytes = solve_smem<R, true>(per, (int)maxn, S.precond);
    cudaLaunchAttribute at[1];
    at[0].id = cudaLaunchAttributeClusterDimension;
    at[0].val.clusterDim.x = (unsigned)size;
    at[0].val.clusterDim.y = at[0].val.clusterDim.z = 1;
    cfg.attrs = at;
    cfg.numAttrs = 1;
    int fit = 0;
    if (cfg.dynamicSmemBytes <= most_smem &&
        cudaOccupancyMaxActiveClusters(&fit, k_cg_solve<R, true>, &cfg) == cudaSuccess && fit > 0 &&
        (!many || clusters_pay(sizeof(R) == 4, S.R, S.N, (double)maxn, size, fit, S.nsm, row))) {
      S.solver = SOLVE_CLUSTER;
      S.solve_blocks = size;
      S.solve_per = per;
      S.solve_maxn = (int)maxn;
      return cudaSuccess;
    }
    cudaGetLastError();
  }
  if (!many && (double)S.N * row <= l2) {
    // one block per SM: a second would add to the exchanges more than it
    // takes off the passes
    const int most = std::min(S.nsm, SOLVE_MAX_BLOCKS), per = (ng + most - 1) / most;
    const size_t smem = solve_smem<R, false>(per, 0, S.precond);
    e = allow_dynamic_smem((const void*)k_cg_solve<R, false>, &most_smem);
    if (e != cudaSuccess) return e;
    int occ = 0;
    if (per <= CS_W && smem <= most_smem &&
        cudaOccupancyMaxActiveBlocksPerMultiprocessor(&occ, k_cg_solve<R, false>, CS_T, smem) == cudaSuccess && occ > 0) {
      S.solver = SOLVE_GRID;
      S.solve_blocks = (ng + per - 1) / per;
      S.solve_per = per;
    }
  }
  return cudaSuccess;
}

template cudaError_t launch_cg_solve<float>(const DevState&, const TypeParams&, double, int, const double*, cudaStream_t);
template cudaError_t launch_cg_solve<double>(const DevState&, const TypeParams&, double, int, const double*, cudaStream_t);
template cudaError_t plan_cg_solve<float>(DevState&, const int64_t*);
template cudaError_t plan_cg_solve<double>(DevState&, const int64_t*);

}  // namespace ct
