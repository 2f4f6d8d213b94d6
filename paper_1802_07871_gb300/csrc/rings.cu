// rings.cu — ring statistics of the C network (Sec. 3.3 follows the numbers
// of 5-, 6- and 7-membered C rings and the in-plane orientation of the
// 6-membered ones). The paper gives no ring criterion; the library counts
// primitive rings: closed paths of distinct C atoms joined by C-C bonds
// shorter than a cutoff, whose bond vectors sum to zero (a path around a
// periodic box is no ring), with no shorter path in the graph between any
// two of their atoms (same displacement) than along the ring.
//
// A ring is found from its lowest atom a, in the direction whose second atom
// is below its last. Two kernels: k_ring_graph lists each C atom's C-C bonds
// (partner, vector) in one place; k_rings takes a warp per atom a:
//   1. breadth first from a to half the largest ring: every (atom,
//      displacement) within max_size / 2 bonds of a and its distance D, in a
//      hash table in shared memory;
//   2. the lanes search depth first from a's two-bond paths. In a primitive
//      ring of n atoms the atom t bonds along has D = min(t, n - t), or a
//      shorter walk would join it to a. So a path runs outwards (D = its
//      length) to at most half the largest ring, and once D falls behind it
//      has to come home one bond at a time: what is left of an exhaustive
//      search of up to eight bonds is a few dozen steps;
//   3. a closed path is checked for every other pair of its atoms by walks of
//      at most three bonds, and its record appended.
// Atoms whose surroundings overflow the table (160 places; 121 is the most in
// amorphous carbon at 3 g/cm^3) are queued and searched again with larger
// tables in global memory. Bound by the
// latency of the walks' dependent loads; the exhaustive search by one thread
// per atom, through the strided lists, took 151 ms on 96 replicas (158,391
// atoms) where a call now takes 2.9 ms.
#include <math.h>
#include <algorithm>

#include "ctbop.h"
#include "internal.cuh"
#include "kernels.h"

namespace ct {

#define RING_MAX 8
#define RING_CLOSE2 0.01   // |sum of bond vectors|^2 below which a path closes (0.1 A)

#define RING_SLOTS 256                     // hash slots of a table in shared memory
#define RING_WARPS 4                       // warps per block

__device__ inline float int_bits(int i, float) { return __int_as_float(i); }
__device__ inline double int_bits(int i, double) { return __longlong_as_double((long long)i); }
__device__ inline int bits_int(float x) { return __float_as_int(x); }
__device__ inline int bits_int(double x) { return (int)__double_as_longlong(x); }

// The C-C bonds of every C atom: entry k of atom v at v * cap + k, the bond
// vector and (bits of w) the partner; and the atoms with two or more, which are
// the ones to search.
template <class R>
struct RingGraph {
  typename Vec4<R>::T* bond;
  int* deg;
  int cap;
};

template <class R>
__global__ void k_ring_graph(int N, int ld, int cap, const typename Vec4<R>::T* __restrict__ u,
                             const int* __restrict__ rep, const RepInfo* __restrict__ reps,
                             const int2* __restrict__ nl, const int* __restrict__ ncov, R cut2,
                             typename Vec4<R>::T* __restrict__ bond, int* __restrict__ deg, int* __restrict__ cand,
                             unsigned long long* __restrict__ n_cand) {
  const int v = blockIdx.x * blockDim.x + threadIdx.x, lane = threadIdx.x & 31;
  int n = 0;
  typename Vec4<R>::T uv;
  uv.w = R(0);
  if (v < N) uv = u[v];
  if ((int)uv.w == 1) {
    const RepInfo& ri = reps[rep[v]];
    R hx = ri.hcf[0], hy = ri.hcf[1], hz = ri.hcf[2];
    if (sizeof(R) == 8) { hx = (R)ri.hc[0]; hy = (R)ri.hc[1]; hz = (R)ri.hc[2]; }
    const int nc = min(ncov[v], cap);
    for (int e = 0; e < nc; ++e) {
      const int2 jc = nl[(size_t)e * ld + v];
      const typename Vec4<R>::T uw = u[jc.x];
      if ((int)uw.w != 1) continue;
      int dx, dy, dz;
      unpack_code(jc.y, dx, dy, dz);
      typename Vec4<R>::T b;
      b.x = (uw.x - uv.x) + (R)dx * hx;
      b.y = (uw.y - uv.y) + (R)dy * hy;
      b.z = (uw.z - uv.z) + (R)dz * hz;
      if (b.x * b.x + b.y * b.y + b.z * b.z >= cut2) continue;
      b.w = int_bits(jc.x, R(0));
      bond[(size_t)v * cap + n] = b;
      ++n;
    }
  }
  if (v < N) deg[v] = n;
  const bool c = n >= 2;   // (no ring closes through one bond)
  const unsigned m = __ballot_sync(CT_FULL, c);
  if (m == 0u) return;
  int at = 0;
  if (lane == 0) at = (int)atomicAdd(n_cand, (unsigned long long)__popc(m));
  at = __shfl_sync(CT_FULL, at, 0);
  if (c) cand[at + __popc(m & ((1u << lane) - 1u))] = v;
}

template <class R>
__device__ inline bool same_place(R ax, R ay, R az, R bx, R by, R bz) {
  const R ex = ax - bx, ey = ay - by, ez = az - bz;
  return ex * ex + ey * ey + ez * ez < R(RING_CLOSE2);
}

// A walk of 1..len bonds from s reaching t with displacement (dx, dy, dz)?
template <class R>
__device__ bool shortcut(const RingGraph<R>& G, int s, int t, R dx, R dy, R dz, int len) {
  int node[3], eix[3];
  R px[3], py[3], pz[3];
  int depth = 0;
  node[0] = s;
  eix[0] = 0;
  px[0] = py[0] = pz[0] = R(0);
  while (depth >= 0) {
    const int v = node[depth];
    if (eix[depth] >= G.deg[v]) {
      --depth;
      continue;
    }
    const typename Vec4<R>::T b = G.bond[(size_t)v * G.cap + eix[depth]++];
    const int w = bits_int(b.w);
    const R qx = px[depth] + b.x, qy = py[depth] + b.y, qz = pz[depth] + b.z;
    if (w == t && same_place(qx, qy, qz, dx, dy, dz)) return true;
    if (depth + 1 < len) {
      ++depth;
      node[depth] = w;
      eix[depth] = 0;
      px[depth] = qx;
      py[depth] = qy;
      pz[depth] = qz;
    }
  }
  return false;
}

// A closed path of n atoms from a: if no pair of its atoms (from the s0-th
// on) has a shortcut, its record.
template <class R>
__device__ void ring_found(const RingGraph<R>& G, int n, int s0, const int* path, const R* px, const R* py,
                           const R* pz, const double* __restrict__ x, const int* __restrict__ rep,
                           ctbop_ring* __restrict__ out, long long cap, unsigned long long* __restrict__ count) {
  for (int s = s0; s < n; ++s)
    for (int t = s + 2; t < n; ++t) {
      const int k = min(t - s, n - (t - s));
      if (k >= 2 && shortcut(G, path[s], path[t], px[t] - px[s], py[t] - py[s], pz[t] - pz[s], k - 1)) return;
    }
  const int a = path[0];
  double cx = 0, cy = 0, cz = 0;
  for (int k = 0; k < n; ++k) {
    cx += (double)px[k];
    cy += (double)py[k];
    cz += (double)pz[k];
  }
  double orient = nan("");
  if (n == 6) {
    double sc = 0.0, ss = 0.0;
    for (int k = 0; k < 3; ++k) {
      double psi = 6.0 * atan2((double)(py[k + 3] - py[k]), (double)(px[k + 3] - px[k]));
      sc += cos(psi);
      ss += sin(psi);
    }
    orient = fmod(atan2(ss, sc) / 6.0 * (180.0 / M_PI) + 60.0, 60.0);
  }
  const unsigned long long slot = atomicAdd(count, 1ull);
  if ((long long)slot < cap) {
    ctbop_ring rr;
    rr.replica = rep[a];
    rr.size = n;
    rr.centre[0] = x[3 * a] + cx / n;
    rr.centre[1] = x[3 * a + 1] + cy / n;
    rr.centre[2] = x[3 * a + 2] + cz / n;
    rr.orientation = orient;
    out[slot] = rr;
  }
}

// Hash table of (atom, displacement) and distance, one per warp; at most
// three quarters of its slots are taken.
template <class R>
struct RingTable {
  R *x, *y, *z;
  int* key;          // atom * 8 + distance, -1 free
  int* node;         // slots in order of discovery
  int slots;         // a power of two
  __device__ void place(void* mem, int n) {
    slots = n;
    x = static_cast<R*>(mem);
    y = x + n;
    z = y + n;
    key = reinterpret_cast<int*>(z + n);
    node = key + n;
  }
  __host__ __device__ static size_t bytes(int n) { return (size_t)n * (3 * sizeof(R) + sizeof(int)) + (size_t)n * 3 / 4 * sizeof(int); }
  __device__ static unsigned hash(int atom) { return ((unsigned)atom * 2654435761u) >> 12; }
  // distance of atom w at (qx, qy, qz), 8 if it is not in the table
  __device__ int distance(int w, R qx, R qy, R qz) const {
    for (unsigned h = hash(w);; ++h) {
      h &= slots - 1;
      const int k = key[h];
      if (k < 0) return 8;
      if ((k >> 3) == w && same_place(qx, qy, qz, x[h], y[h], z[h])) return k & 7;
    }
  }
};

// The search from atom a by one warp; false when its table overflows.
template <class R>
__device__ bool ring_search(int a, const RingTable<R>& T, const RingGraph<R>& G, const double* __restrict__ x,
                            const int* __restrict__ rep, int max_size, ctbop_ring* __restrict__ out, long long cap,
                            unsigned long long* __restrict__ count) {
  const int lane = threadIdx.x & 31;
  const unsigned lt = (1u << lane) - 1u;
  const int most = T.slots * 3 / 4;
  const int da = G.deg[a];
  // ---- 1. breadth first
  for (int k = lane; k < T.slots; k += 32) T.key[k] = -1;
  __syncwarp();
  if (lane == 0) {
    const unsigned h = RingTable<R>::hash(a) & (T.slots - 1);
    T.key[h] = a * 8;
    T.x[h] = T.y[h] = T.z[h] = R(0);
    T.node[0] = (int)h;
  }
  __syncwarp();
  int n0 = 0, n1 = 1;   // the frontier: nodes [n0, n1)
  bool full = false;
  for (int d = 1; d <= max_size / 2 && !full; ++d) {
    int n2 = n1;
    // each lane takes a frontier node in turn; its bonds are tried one by one
    for (int f0 = n0; f0 < n1 && !full; f0 += 32) {
      const int f = f0 + lane;
      int v = 0, dv = 0;
      R vx = R(0), vy = R(0), vz = R(0);
      if (f < n1) {
        const int h = T.node[f];
        v = T.key[h] >> 3;
        dv = G.deg[v];
        vx = T.x[h]; vy = T.y[h]; vz = T.z[h];
      }
      const int dmax = (int)__reduce_max_sync(CT_FULL, (unsigned)dv);
      for (int e = 0; e < dmax && !full; ++e) {
        bool todo = e < dv;
        int w = -1;
        R qx = R(0), qy = R(0), qz = R(0);
        if (todo) {
          const typename Vec4<R>::T b = G.bond[(size_t)v * G.cap + e];
          w = bits_int(b.w);
          qx = vx + b.x; qy = vy + b.y; qz = vz + b.z;
        }
        unsigned h = RingTable<R>::hash(w) & (T.slots - 1);
        while (__any_sync(CT_FULL, todo)) {
          // claim a free slot; whoever wins writes its place before anyone compares with it
          bool won = false;
          int k = 0;
          if (todo) {
            k = atomicCAS(T.key + h, -1, w * 8 + d);
            won = k == -1;
            if (won) { T.x[h] = qx; T.y[h] = qy; T.z[h] = qz; }
          }
          __syncwarp();
          const unsigned wins = __ballot_sync(CT_FULL, won);
          if (won) {
            const int at = n2 + __popc(wins & lt);
            T.node[at] = (int)h;   // (at < most: see full)
            todo = false;
          } else if (todo) {
            if ((k >> 3) == w && same_place(qx, qy, qz, T.x[h], T.y[h], T.z[h])) todo = false;   // known already
            else h = (h + 1) & (T.slots - 1);
          }
          n2 += __popc(wins);
          full = n2 > most - 32;   // (at most 32 more a round: neither the table nor the list overruns)
          __syncwarp();
          if (full) break;
        }
      }
    }
    n0 = n1;
    n1 = n2;
  }
  if (full) return false;   // (uniform over the warp)
  // ---- 2. depth first from the two-bond paths, dealt to the lanes
  int dm = 0;
  for (int e = lane; e < da; e += 32) dm = max(dm, G.deg[bits_int(G.bond[(size_t)a * G.cap + e].w)]);
  dm = (int)__reduce_max_sync(CT_FULL, (unsigned)dm);
  for (int t = lane; t < da * dm; t += 32) {
    int path[RING_MAX], eix[RING_MAX], dist[RING_MAX];
    R px[RING_MAX], py[RING_MAX], pz[RING_MAX];
    const typename Vec4<R>::T b1 = G.bond[(size_t)a * G.cap + t / dm];
    path[0] = a;
    path[1] = bits_int(b1.w);
    if (path[1] <= a) continue;
    px[0] = py[0] = pz[0] = R(0);
    px[1] = b1.x; py[1] = b1.y; pz[1] = b1.z;
    dist[0] = 0;
    dist[1] = 1;
    eix[1] = t % dm;
    if (eix[1] >= G.deg[path[1]]) continue;
    const int only = eix[1] + 1;   // this lane's one bond of the second atom
    int depth = 1;
    while (depth >= 1) {
      const int v = path[depth];
      if (eix[depth] >= (depth == 1 ? only : G.deg[v])) {
        --depth;
        continue;
      }
      const typename Vec4<R>::T b = G.bond[(size_t)v * G.cap + eix[depth]++];
      const int w = bits_int(b.w);
      if (w <= a) continue;
      bool seen = false;
      for (int k = 1; k <= depth; ++k) seen = seen || path[k] == w;
      if (seen) continue;
      const R qx = px[depth] + b.x, qy = py[depth] + b.y, qz = pz[depth] + b.z;
      const int D = T.distance(w, qx, qy, qz), len = depth + 1;   // len: bonds from a to w along the path
      // outwards: as far again; on the way home: one nearer. The ring has at least len + D atoms
      if (D == 8 || len + D > max_size || (dist[depth] < depth && D != dist[depth] - 1)) continue;
      path[len] = w;
      px[len] = qx; py[len] = qy; pz[len] = qz;
      if (D == 1) {   // home: w is bonded to a at this place
        if (path[1] < w) ring_found(G, len + 1, 1, path, px, py, pz, x, rep, out, cap, count);
        continue;
      }
      depth = len;
      eix[depth] = 0;
      dist[depth] = D;
    }
  }
  __syncwarp();
  return true;
}

template <class R>
__global__ void __launch_bounds__(RING_WARPS * 32)
    k_rings(const int* __restrict__ cand, RingGraph<R> G, const double* __restrict__ x, const int* __restrict__ rep,
            int max_size, ctbop_ring* __restrict__ out, long long cap, unsigned long long* __restrict__ count,
            int* __restrict__ wide) {
  extern __shared__ __align__(16) unsigned char smem_raw[];
  const int warp = threadIdx.x >> 5, lane = threadIdx.x & 31;
  RingTable<R> T;
  T.place(smem_raw + warp * RingTable<R>::bytes(RING_SLOTS), RING_SLOTS);
  const int n = (int)count[2];
  // (neighbours of the list to one block: they share bonds in L1)
  for (int t = blockIdx.x * RING_WARPS + warp; t < n; t += gridDim.x * RING_WARPS) {
    const int a = cand[t];
    if (!ring_search(a, T, G, x, rep, max_size, out, cap, count) && lane == 0) wide[atomicAdd(count + 1, 1ull)] = a;
    __syncwarp();
  }
}

// The queued atoms, with a table of `slots` in global memory for each warp
// of the launch; those that overflow it too go to the next queue.
template <class R>
__global__ void __launch_bounds__(RING_WARPS * 32)
    k_rings_wide(int n_queue, const int* __restrict__ queue, unsigned char* __restrict__ tables, int slots,
                 RingGraph<R> G, const double* __restrict__ x, const int* __restrict__ rep, int max_size,
                 ctbop_ring* __restrict__ out, long long cap, unsigned long long* __restrict__ count,
                 int* __restrict__ wide) {
  const int w = blockIdx.x * RING_WARPS + (threadIdx.x >> 5);
  RingTable<R> T;
  T.place(tables + (size_t)w * RingTable<R>::bytes(slots), slots);
  for (int t = w; t < n_queue; t += gridDim.x * RING_WARPS) {
    const int a = queue[t];
    if (!ring_search(a, T, G, x, rep, max_size, out, cap, count) && (threadIdx.x & 31) == 0)
      wide[atomicAdd(count + 1, 1ull)] = a;
    __syncwarp();
  }
}

// Scratch of the search, per atom: the bonds in the force slots (Real4 per
// covalent entry; every force pass writes its slots before it reads them), the
// degrees, the two queues and the list of atoms to search in the staging buffer
// (16 of its 24 bytes an atom).
//
// The grid is at most eight times what is resident at once, and strides over the
// listed atoms: a warp per atom of the system, none with anything to do in SiC,
// took 89 us a call on a slab of 397,490 atoms without C-C bonds, where an
// exhaustive search's threads had taken 44; this 42. (The resident blocks alone, or
// warps that fetch one atom after another, lose 3 to 7% where C abounds: uneven
// shares, and neighbours spread over the SMs.) The ensemble of 158,391 atoms
// 2,480 -> 2,145 us, a graphene sheet of 20,088 atoms 444 -> 465.
template <class R>
cudaError_t launch_rings(const DevState& S, double bond_cut, int max_size, ctbop_ring* out, long long cap,
                         unsigned long long* count, cudaStream_t st) {
  if (S.N == 0) return cudaSuccess;
  int* deg = static_cast<int*>(S.stage);
  RingGraph<R> G{(typename Vec4<R>::T*)S.gslot, deg, S.cap_cov};
  k_ring_graph<R><<<(S.N + 255) / 256, 256, 0, st>>>(S.N, S.ld, S.cap_cov, (const typename Vec4<R>::T*)S.u, S.rep,
                                                     S.reps, S.nl, S.ncov, (R)(bond_cut * bond_cut), G.bond, deg,
                                                     deg + (size_t)3 * S.N, count + 2);
  const size_t smem = RING_WARPS * RingTable<R>::bytes(RING_SLOTS);
  int occ = 0;
  cudaError_t e = cudaOccupancyMaxActiveBlocksPerMultiprocessor(&occ, k_rings<R>, RING_WARPS * 32, smem);
  if (e != cudaSuccess) return e;
  const int grid = std::min((S.N + RING_WARPS - 1) / RING_WARPS, 8 * S.nsm * std::max(occ, 1));
  k_rings<R><<<grid, RING_WARPS * 32, smem, st>>>(deg + (size_t)3 * S.N, G, S.x, S.rep, max_size, out, cap, count,
                                                  deg + S.N);
  return cudaGetLastError();
}

size_t rings_wide_bytes(const DevState& S, bool fp32, int slots) {
  return (size_t)S.nsm * RING_WARPS * (fp32 ? RingTable<float>::bytes(slots) : RingTable<double>::bytes(slots));
}

template <class R>
cudaError_t launch_rings_wide(const DevState& S, int pass, int n_queue, int slots, void* tables, int max_size,
                              ctbop_ring* out, long long cap, unsigned long long* count, cudaStream_t st) {
  int* deg = static_cast<int*>(S.stage);
  RingGraph<R> G{(typename Vec4<R>::T*)S.gslot, deg, S.cap_cov};
  int *queue = deg + (size_t)S.N * (1 + pass % 2), *next = deg + (size_t)S.N * (2 - pass % 2);
  k_rings_wide<R><<<S.nsm, RING_WARPS * 32, 0, st>>>(n_queue, queue, static_cast<unsigned char*>(tables), slots, G, S.x,
                                                     S.rep, max_size, out, cap, count, next);
  return cudaGetLastError();
}

template cudaError_t launch_rings_wide<float>(const DevState&, int, int, int, void*, int, ctbop_ring*, long long,
                                              unsigned long long*, cudaStream_t);
template cudaError_t launch_rings_wide<double>(const DevState&, int, int, int, void*, int, ctbop_ring*, long long,
                                               unsigned long long*, cudaStream_t);
template cudaError_t launch_rings<float>(const DevState&, double, int, ctbop_ring*, long long, unsigned long long*,
                                         cudaStream_t);
template cudaError_t launch_rings<double>(const DevState&, double, int, ctbop_ring*, long long, unsigned long long*,
                                          cudaStream_t);

}  // namespace ct
