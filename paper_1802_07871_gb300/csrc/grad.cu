// grad.cu — derivatives of the energy with respect to the potential's
// parameters (the force-matching gradient of the differentiation pattern),
// FP64, with forward-mode tangents along a per-atom direction.
//
// At the charge minimiser the total derivative of E with respect to a
// parameter equals the partial derivative at fixed charges (the charges are
// stationary on sum q = Q, which no parameter changes), so dE/dtheta is a
// sum of per-term partial derivatives:
//   * pair terms 1/2 fc(r) [A e^{-l1 r} - c_ij b_ij B e^{-l2 r}] (A, B, l1,
//     l2, kappa, and R, S through fc);
//   * the bond order b (Eq. 7) through sigma, p, g_l, n_l, recomputing the
//     environment sums zeta_l (Eq. 2) instead of storing them;
//   * zeta_l through the triplet parameters gamma, c, d, h, alpha and through
//     the cutoff fc(r_ik) (R, S of the pair (i, k));
//   * the self energy E0 + chi q + J q^2 and the charge kernel (k_e, r_coul,
//     gamma_c).
// The gradient vector has the layout of ctbop_params (144 doubles); each
// atom's terms are weighted by a per-replica weight, so one pass gives
// sum_r a_r dE_r/dtheta.
//
// The force part of a force-matching gradient needs, for a direction g (one
// 3-vector per atom), the derivative of dE/dtheta along x + e g at fixed
// charges and the derivative of the charge gradient dE/dq = H q + chi along
// the same direction. Both come from the same kernels evaluated on dual
// numbers (value, derivative along g): every quantity that depends on the
// positions carries its exact directional derivative, with no step size.
#include <algorithm>
#include <cmath>

#include "internal.cuh"
#include "kernels.h"
#include "ctbop.h"

namespace ct {

// ------------------------------------------------------------ dual numbers
// A value and its derivative along one direction, in T = float or double.
// Operators take the same T on both sides, so no double constant can slip
// into an FP32 expression.
template <class T> struct DualT {
  T v, d;
  DualT() = default;
  __device__ DualT(T x) : v(x), d(T(0)) {}
  __device__ DualT(T x, T dx) : v(x), d(dx) {}
};
template <class T> __device__ inline DualT<T> operator+(DualT<T> a, DualT<T> b) { return {a.v + b.v, a.d + b.d}; }
template <class T> __device__ inline DualT<T> operator-(DualT<T> a, DualT<T> b) { return {a.v - b.v, a.d - b.d}; }
template <class T> __device__ inline DualT<T> operator-(DualT<T> a) { return {-a.v, -a.d}; }
template <class T> __device__ inline DualT<T> operator*(DualT<T> a, DualT<T> b) {
  return {a.v * b.v, a.d * b.v + a.v * b.d};
}
template <class T> __device__ inline DualT<T> operator/(DualT<T> a, DualT<T> b) {
  const T r = inv(b.v), q = a.v * r;
  return {q, (a.d - q * b.d) * r};
}
template <class T> __device__ inline DualT<T> operator+(DualT<T> a, T b) { return {a.v + b, a.d}; }
template <class T> __device__ inline DualT<T> operator+(T a, DualT<T> b) { return {a + b.v, b.d}; }
template <class T> __device__ inline DualT<T> operator-(DualT<T> a, T b) { return {a.v - b, a.d}; }
template <class T> __device__ inline DualT<T> operator-(T a, DualT<T> b) { return {a - b.v, -b.d}; }
template <class T> __device__ inline DualT<T> operator*(DualT<T> a, T b) { return {a.v * b, a.d * b}; }
template <class T> __device__ inline DualT<T> operator*(T a, DualT<T> b) { return {a * b.v, a * b.d}; }
template <class T> __device__ inline DualT<T> operator/(DualT<T> a, T b) { return {a.v / b, a.d / b}; }
template <class T> __device__ inline DualT<T> operator/(T a, DualT<T> b) {
  const T r = inv(b.v), q = a * r;
  return {q, -q * b.d * r};
}
template <class T> __device__ inline DualT<T>& operator+=(DualT<T>& a, DualT<T> b) { a = a + b; return a; }

__device__ inline double val(double x) { return x; }
__device__ inline float val(float x) { return x; }
template <class T> __device__ inline T val(DualT<T> x) { return x.v; }
__device__ inline double tng(double) { return 0.0; }
__device__ inline float tng(float) { return 0.0f; }
template <class T> __device__ inline T tng(DualT<T> x) { return x.d; }

// elementary functions on T and on DualT<T> (CUDA's own float and double
// routines for the values; the derivatives from their closed forms)
__device__ inline double fexp(double x) { return exp(x); }
__device__ inline float fexp(float x) { return expf(x); }
__device__ inline double flog(double x) { return log(x); }
__device__ inline float flog(float x) { return logf(x); }
__device__ inline double fpow(double x, double n) { return pow(x, n); }
__device__ inline float fpow(float x, float n) { return powf(x, n); }
__device__ inline double fcospi(double x) { return cospi(x); }
__device__ inline float fcospi(float x) { return cospif(x); }
__device__ inline double fsinpi(double x) { return sinpi(x); }
__device__ inline float fsinpi(float x) { return sinpif(x); }
template <class T> __device__ inline DualT<T> fexp(DualT<T> x) { T e = fexp(x.v); return {e, e * x.d}; }
template <class T> __device__ inline DualT<T> flog(DualT<T> x) { return {flog(x.v), x.d * inv(x.v)}; }
template <class T> __device__ inline DualT<T> fpow(DualT<T> x, T n) {   // x.v > 0
  T p = fpow(x.v, n);
  return {p, n * p * inv(x.v) * x.d};
}
template <class T> __device__ inline DualT<T> fcospi(DualT<T> x) {
  return {fcospi(x.v), -T(M_PI) * fsinpi(x.v) * x.d};
}
template <class T> __device__ inline DualT<T> fsinpi(DualT<T> x) {
  return {fsinpi(x.v), T(M_PI) * fcospi(x.v) * x.d};
}

// A value with its derivative (kept for DualT, dropped for a plain T).
template <class S> struct Mk;
template <> struct Mk<double> { __device__ static double f(double v, double) { return v; } };
template <> struct Mk<float> { __device__ static float f(float v, float) { return v; } };
template <class T> struct Mk<DualT<T>> { __device__ static DualT<T> f(T v, T d) { return DualT<T>(v, d); } };

// The parameter struct in the working precision: ctbop_params' fields, in
// the same order, as R.
template <class R> struct ParamsT {
  R A[4], B[4], lambda1[4], lambda2[4], R_[4], S[4], kappa[4];
  R sigma[4], p[4], g[4][2], n[4][2];
  R gamma[8][2], c[8][2], d[8][2], h[8][2], alpha[8][2];
  R E0[2], chi[2], J[2], gamma_c[2], mass[2];
  R r_coul, k_e;
};
static_assert(sizeof(ParamsT<double>) == sizeof(ctbop_params), "ParamsT mirrors ctbop_params");
static_assert(sizeof(ParamsT<float>) * 2 == sizeof(ctbop_params), "ParamsT mirrors ctbop_params");

// Cutoff fc(r) and its derivatives with respect to R and S.
template <class R, class S>
__device__ inline void fc_params(S r, R Rin, R Sc, S& fc, S& dR, S& dS) {
  dR = dS = S(R(0));
  if (val(r) < Rin) { fc = S(R(1)); return; }
  if (val(r) >= Sc) { fc = S(R(0)); return; }
  R w = Sc - Rin;
  // 1/2 [1 + cos(pi t)] as cos^2(pi t / 2), free of the cancellation near
  // t = 1 (the cutoff function of the force kernels does the same)
  S h = R(0.5) * ((r - Rin) / w);
  S c = fcospi(h), sn = fsinpi(h);
  fc = c * c;
  S dfdt = R(-M_PI) * sn * c;
  dR = dfdt * (r - Sc) / (w * w);
  dS = dfdt * (Rin - r) / (w * w);
}

template <class R, class S>
__device__ inline S fc_only(S r, R Rin, R Sc) {
  if (val(r) < Rin) return S(R(1));
  if (val(r) >= Sc) return S(R(0));
  S c = fcospi(R(0.5) * ((r - Rin) / (Sc - Rin)));
  return c * c;
}

// Sums of the covalent terms. A bond feeds 13 parameters of its ordered pair
// and, per type of third atom, 12 more; each with a value and a tangent, in
// FP64 and weighted by the atom's replica. An FP64 warp instruction takes 64
// cycles here, and adding every lane's share to a block sum in shared memory
// (no FP64 instruction there: a compare-and-swap loop whose lanes all want the
// same few words) kept the FP64 pipe busy 81% of the pass. Instead the lanes of
// a warp put up to 32 shares each into a shared tile (working precision), and
// lane s adds up share s of all lanes with a bond, one fused multiply-add per
// lane, into a register per ordered pair: a bond costs three FP64 instructions
// a lane instead of about 74 contended additions. The registers join the block
// sums once per block.
#define PG_TILE 32
template <class R> struct Stage {
  R* tile;             // [PG_TILE][33]: share, lane
  const double* w;     // [32][2]: the lanes' value and tangent weights
  // shares of this lane: value 2 k, tangent 2 k + 1
  __device__ void put(int k, R x) const { tile[(2 * k) * 33 + (threadIdx.x & 31)] = x; }
  __device__ void put(int k, DualT<R> x) const {
    tile[(2 * k) * 33 + (threadIdx.x & 31)] = x.v;
    tile[(2 * k + 1) * 33 + (threadIdx.x & 31)] = x.d;
  }
  // lane s: sums of share s over the lanes of `mask`, by their ordered pair
  template <bool TAN>
  __device__ void sum(unsigned mask, int pb, int n, double (&acc)[4]) const {
    const int s = threadIdx.x & 31;
    const bool used = s < 2 * n && (TAN || !(s & 1));
    __syncwarp();
    for (unsigned m = mask; m; m &= m - 1) {
      const int src = __ffs(m) - 1;
      const int p = __shfl_sync(CT_FULL, pb, src);   // (uniform)
      const double x = used ? (double)tile[s * 33 + src] : 0.0;
      const double ws = w[2 * src + (s & 1)];
      if (p == 0) acc[0] = fma(ws, x, acc[0]);
      else if (p == 1) acc[1] = fma(ws, x, acc[1]);
      else if (p == 2) acc[2] = fma(ws, x, acc[2]);
      else acc[3] = fma(ws, x, acc[3]);
    }
    __syncwarp();
  }
};
template <class S> struct IsDual { static constexpr bool v = false; };
template <class T> struct IsDual<DualT<T>> { static constexpr bool v = true; };

// Lanes per atom: FP32 four, as many as an atom of these systems usually has
// bonds; FP64 eight: there the pass waits for the densest atoms' serial loops
// over third atoms (15 neighbours in the random clusters), not for lanes.
#define PG_T 128     // threads per block; 32 where the entries of its atoms do not fit shared memory
template <class R> struct PgLanes { static constexpr int v = sizeof(R) == 8 ? 8 : 4; };

// What the bond order's parameter derivatives need of the parameters alone,
// per ordered pair: with s_l = g_l^-p, S0 = s_1 + s_2: ln S0, d ln S0 / dp and
// p g_l^(-p-1) / S0.
template <class R> struct PgConst {
  R lnS0[4], dlnS0_dp[4], dg[4][2];
  R id2[8][2];   // 1 / d^2 of the triplets
};

// One covalent list entry as staged in shared memory: the bond's direction,
// length and cutoff, and their derivatives along the direction (zero without
// one).
template <class R> struct __align__(16) Ent {
  R x, y, z, r, fc;
  R tx, ty, tz, tr, tfc;
  R pad[2];
};

template <class R, class S> __device__ inline void ent_vec(const Ent<R>& a, S& x, S& y, S& z, S& r) {
  x = Mk<S>::f(a.x, a.tx); y = Mk<S>::f(a.y, a.ty); z = Mk<S>::f(a.z, a.tz); r = Mk<S>::f(a.r, a.tr);
}

// Bond vector from atom i to the image of j named by the list code, in the
// cell-local coordinates the positions are stored in.
template <class R>
__device__ inline void bond_vec(const typename Vec4<R>::T& ui, const typename Vec4<R>::T& uj, int code,
                                const RepInfo& ri, R& rx, R& ry, R& rz) {
  int dx, dy, dz;
  unpack_code(code, dx, dy, dz);
  R hx = ri.hcf[0], hy = ri.hcf[1], hz = ri.hcf[2];
  if (sizeof(R) == 8) { hx = (R)ri.hc[0]; hy = (R)ri.hc[1]; hz = (R)ri.hc[2]; }
  rx = (uj.x - ui.x) + (R)dx * hx;
  ry = (uj.y - ui.y) + (R)dy * hy;
  rz = (uj.z - ui.z) + (R)dz * hz;
}

// Covalent terms: one lane group per atom, the atom's covalent entries
// staged in shared memory; each lane takes bonds e, the warp in step. Sums by
// Stage, then one atomicAdd per parameter and block. R is the
// working precision, S either R (values only) or DualT<R>: then the entries
// carry their derivatives along dir and the charges theirs along qdir, the
// tangents of every term go to the second half of grad, and (with vout) each
// bond's share of d(Hq + chi)/de goes to vout: the charge-coupling term
// 1/2 fc kappa (q_i - q_j)^2 b_ij f_A contributes +-kappa fc f_A b_ij
// (q_i - q_j) to rows i and j.
template <class R, class S, int NT>
__global__ void __launch_bounds__(NT)
    k_pgrad_cov(int N, int cap_cov, int ld, const typename Vec4<R>::T* __restrict__ u,
                const int* __restrict__ rep, const RepInfo* __restrict__ reps, const int2* __restrict__ nl,
                const int* __restrict__ ncov, const double* __restrict__ q, const double* __restrict__ qdir,
                const double* __restrict__ wval, const double* __restrict__ wtan, const double* __restrict__ dir,
                ParamsT<R> P, PgConst<R> K, double* __restrict__ grad, double* __restrict__ vout) {
  using R4 = typename Vec4<R>::T;
  constexpr int PG_GRP = PgLanes<R>::v, APB = NT / PG_GRP;
  extern __shared__ __align__(32) unsigned char smem_raw[];
  constexpr int NW = NT / 32;
  constexpr bool TAN = IsDual<S>::v;
  __shared__ double s_g[2 * PG_NPARAM], s_w[NW][64];
  __shared__ R s_tile[NW][PG_TILE * 33];
  for (int k = threadIdx.x; k < 2 * PG_NPARAM; k += blockDim.x) s_g[k] = 0.0;
  const int lane = threadIdx.x & 31, warp = threadIdx.x >> 5;
  const Stage<R> stage{s_tile[warp], s_w[warp]};
  double sums[3][4];
#pragma unroll
  for (int k = 0; k < 12; ++k) sums[k / 4][k % 4] = 0.0;
  int g = threadIdx.x / PG_GRP, l = threadIdx.x % PG_GRP;
  Ent<R>* s_e = reinterpret_cast<Ent<R>*>(smem_raw) + (size_t)g * cap_cov;
  int* s_t = reinterpret_cast<int*>(reinterpret_cast<Ent<R>*>(smem_raw) + (size_t)APB * cap_cov) +
             (size_t)g * cap_cov;
  int* s_j = reinterpret_cast<int*>(reinterpret_cast<Ent<R>*>(smem_raw) + (size_t)APB * cap_cov) +
             (size_t)APB * cap_cov + (size_t)g * cap_cov;
  int* s_lv = s_j + (size_t)APB * cap_cov;   // the live bonds (r < S), in list order
  int i = blockIdx.x * APB + g;
  bool live = i < N;
  int nc = 0, ti = 0;
  double wv = 0.0, wt = 0.0;
  S qi = S(R(0));
  if (live) {
    R4 ui = u[i];
    ti = (int)ui.w;
    nc = min(ncov[i], cap_cov);
    const RepInfo& ri = reps[rep[i]];
    wv = wval[rep[i]];
    wt = wtan ? wtan[rep[i]] : 0.0;
    qi = Mk<S>::f((R)q[i], qdir ? (R)qdir[i] : R(0));
    R gix = 0, giy = 0, giz = 0;
    if (dir) { gix = (R)dir[3 * i]; giy = (R)dir[3 * i + 1]; giz = (R)dir[3 * i + 2]; }
    for (int e = l; e < nc; e += PG_GRP) {
      size_t idx = (size_t)e * ld + i;
      int j = nl[idx].x;
      R4 uj = u[j];
      Ent<R> w;
      bond_vec<R>(ui, uj, nl[idx].y, ri, w.x, w.y, w.z);
      w.r = sqrt(w.x * w.x + w.y * w.y + w.z * w.z);
      const R ir = inv(w.r);
      w.x *= ir; w.y *= ir; w.z *= ir;
      w.tx = w.ty = w.tz = w.tr = R(0);
      if (dir) {
        const R tx = (R)dir[3 * j] - gix, ty = (R)dir[3 * j + 1] - giy, tz = (R)dir[3 * j + 2] - giz;
        w.tr = w.x * tx + w.y * ty + w.z * tz;
        w.tx = (tx - w.tr * w.x) * ir; w.ty = (ty - w.tr * w.y) * ir; w.tz = (tz - w.tr * w.z) * ir;
      }
      const int pe = ti * 2 + (int)uj.w;
      const S fe = fc_only(Mk<S>::f(w.r, w.tr), P.R_[pe], P.S[pe]);
      w.fc = val(fe);
      w.tfc = tng(fe);
      s_e[e] = w;
      s_t[e] = (int)uj.w;
      s_j[e] = j;
    }
  }
  __syncthreads();
  // bonds past S have f_c = 0 and no parameter derivative: the loops below
  // run over the live ones only, in list order
  const int nlive = compact_live<PG_GRP>(
      live, nc, l, s_lv, [&](int e) { return s_e[e].r < P.S[ti * 2 + s_t[e]]; }, [](int) {});
  s_w[warp][2 * lane] = wv;
  s_w[warp][2 * lane + 1] = wt;
  __syncwarp();
  const int nmine = live && (wv != 0.0 || wt != 0.0) ? nlive : 0;
  const int rounds = (int)__reduce_max_sync(CT_FULL, (unsigned)((nmine + PG_GRP - 1) / PG_GRP));
  for (int round = 0; round < rounds; ++round) {
    const int b_ = round * PG_GRP + l;
    const int e = b_ < nmine ? s_lv[b_] : -1;
    int pb = 0, tj = 0;
    S ex = S(R(0)), ey = S(R(0)), ez = S(R(0)), re = S(R(0)), fc = S(R(0)), fcR = S(R(0)), fcS = S(R(0));
    if (e >= 0) {
      ent_vec(s_e[e], ex, ey, ez, re);
      tj = s_t[e];
      pb = ti * 2 + tj;
      fc_params(re, P.R_[pb], P.S[pb], fc, fcR, fcS);
    }
    const bool on = e >= 0 && val(fc) != R(0);
    const unsigned mask = __ballot_sync(CT_FULL, on);
    S Ez[2], sA[2][2], sC[2][2], sD[2][2], sH[2][2], sL[2][2], sR[2][2], sS[2][2];
#pragma unroll
    for (int k = 0; k < 4; ++k)
      Ez[k & 1] = sA[k >> 1][k & 1] = sC[k >> 1][k & 1] = sD[k >> 1][k & 1] = sH[k >> 1][k & 1] = sL[k >> 1][k & 1] =
          sR[k >> 1][k & 1] = sS[k >> 1][k & 1] = S(R(0));
    if (on) {
      // environment sums of bond e (recomputed), and with them what the
      // triplet parameters' derivatives need, dE/dzeta_l taken out: sums over
      // the k of each type of E = fc e^{alpha (r_e - r_k)} times
      //   A ang / gamma, C hm^2 / den, D 1/den^2 - 1/d^4, H hm / den^2, L A (r_e - r_k),
      // and of e^{...} ang / gamma times dfc/dR, dfc/dS for k in its taper
      // (hm = h - cos, den = d^2 + hm^2)
#pragma unroll
      for (int tk = 0; tk < 2; ++tk) {
        const int tri = pb * 2 + tk, pk = ti * 2 + tk;
        for (int kk = 0; kk < nlive; ++kk) {
          const int k = s_lv[kk];
          if (k == e || s_t[k] != tk) continue;
          S kx, ky, kz, rk;
          const Ent<R>& ek = s_e[k];
          ent_vec(ek, kx, ky, kz, rk);
          const S fck = Mk<S>::f(ek.fc, ek.tfc);
          const S ct = ex * kx + ey * ky + ez * kz, dr = re - rk;
          // (by the length: just past R the cutoff rounds to 1 while its second derivative has already jumped)
          const bool taper = val(rk) >= P.R_[pk];
          S fkR, fkS, dum;
          if (taper) fc_params(rk, P.R_[pk], P.S[pk], dum, fkR, fkS);
#pragma unroll
          for (int ll = 0; ll < 2; ++ll) {
            const R cc = P.c[tri][ll], dd = P.d[tri][ll], d2 = dd * dd, id2 = K.id2[tri][ll];
            const S hm = P.h[tri][ll] - ct, hm2 = hm * hm;
            const S iden = R(1) / (d2 + hm2), q2 = hm2 * iden, iden2 = iden * iden;
            const S ang = R(1) + (cc * cc * id2) * q2;   // ang / gamma
            const S exl = fexp(P.alpha[tri][ll] * dr), E = exl * fck, EA = E * ang;
            sA[tk][ll] += EA;
            sC[tk][ll] += E * q2;
            sD[tk][ll] += E * (iden2 - id2 * id2);
            sH[tk][ll] += E * (hm * iden2);
            sL[tk][ll] += EA * dr;
            if (taper) {
              const S xa = exl * ang;
              sR[tk][ll] += xa * fkR;
              sS[tk][ll] += xa * fkS;
            }
          }
        }
      }
      S z[2];
      for (int ll = 0; ll < 2; ++ll)
        z[ll] = P.gamma[pb * 2][ll] * sA[0][ll] + P.gamma[pb * 2 + 1][ll] * sA[1][ll];
      // bond order (Eq. 7) and its parameter derivatives, via ln b = e (ln S - ln S0)
      R pp = P.p[pb], sg = P.sigma[pb], ex_ = R(1) / (R(2) * sg * pp);
      S zn[2], Z[2], t[2], lnz[2];
      for (int ll = 0; ll < 2; ++ll) {
        bool pos = val(z[ll]) > R(0);
        zn[ll] = pos ? fpow(z[ll], P.n[pb][ll]) : S(R(0));
        lnz[ll] = pos ? flog(z[ll]) : S(R(0));
        Z[ll] = P.g[pb][ll] + zn[ll];
        t[ll] = fpow(Z[ll], -pp);
      }
      S Ssum = t[0] + t[1];
      S lnb = ex_ * (flog(Ssum) - K.lnS0[pb]);
      S b = fexp(lnb);
      S dq = qi - Mk<S>::f((R)q[s_j[e]], qdir ? (R)qdir[s_j[e]] : R(0));
      S dq2 = dq * dq;
      S cq = R(1) - P.kappa[pb] * dq2;
      S e1 = fexp(-P.lambda1[pb] * re), e2 = fexp(-P.lambda2[pb] * re);
      S fR = P.A[pb] * e1, fA = P.B[pb] * e2;
      S V = fR - cq * b * fA;
      S Eb = R(-0.5) * cq * fc * fA;   // dE/db
      if (vout) {
        double wq = (double)tng(P.kappa[pb] * (fc * fA * b)) * (double)val(dq);
        if (wq != 0.0) {
          atomicAdd(vout + i, wq);
          atomicAdd(vout + s_j[e], -wq);
        }
      }
      // pair parameters
      stage.put(0, R(0.5) * fc * e1);
      stage.put(1, R(-0.5) * cq * fc * b * e2);
      stage.put(2, R(-0.5) * fc * re * fR);
      stage.put(3, R(0.5) * cq * fc * b * fA * re);
      stage.put(4, R(0.5) * dq2 * fc * b * fA);
      stage.put(5, R(0.5) * fcR * V);
      stage.put(6, R(0.5) * fcS * V);
      // bond-order parameters
      S dlnS_dp = -(t[0] * flog(Z[0]) + t[1] * flog(Z[1])) / Ssum;
      S wb = Eb * b;
      stage.put(7, wb * (-lnb / sg));
      stage.put(8, wb * (-lnb / pp + ex_ * (dlnS_dp - K.dlnS0_dp[pb])));
      for (int ll = 0; ll < 2; ++ll) {
        const S tz = (-pp * ex_) * (t[ll] / (Z[ll] * Ssum));   // d ln b / d Z_l
        stage.put(9 + ll, wb * (tz + ex_ * K.dg[pb][ll]));
        const S wt_ = wb * tz;
        stage.put(11 + ll, val(z[ll]) > R(0) ? wt_ * zn[ll] * lnz[ll] : S(R(0)));
        // dE/dzeta_l = Eb db/dzeta_l = Eb b (d ln b / d zeta_l)
        if (val(z[ll]) > R(0)) Ez[ll] = P.n[pb][ll] * (wt_ * (zn[ll] / z[ll]));
      }
    }
    stage.template sum<TAN>(mask, pb, 13, sums[0]);
    // triplet parameters, and the cutoff of the (i, k) pairs inside zeta
#pragma unroll
    for (int tk = 0; tk < 2; ++tk) {
      if (on) {
        const int tri = pb * 2 + tk;
        S tR = S(R(0)), tS = S(R(0));
#pragma unroll
        for (int ll = 0; ll < 2; ++ll) {
          const R cc = P.c[tri][ll], dd = P.d[tri][ll], g2 = R(2) * P.gamma[tri][ll];
          const S gE = P.gamma[tri][ll] * Ez[ll];
          stage.put(0 + ll, Ez[ll] * sA[tk][ll]);
          stage.put(2 + ll, (g2 * cc * K.id2[tri][ll]) * (Ez[ll] * sC[tk][ll]));
          stage.put(4 + ll, (g2 * cc * cc * dd) * (Ez[ll] * sD[tk][ll]));
          stage.put(6 + ll, (g2 * cc * cc) * (Ez[ll] * sH[tk][ll]));
          stage.put(8 + ll, gE * sL[tk][ll]);
          tR += gE * sR[tk][ll];
          tS += gE * sS[tk][ll];
        }
        stage.put(10, tR);
        stage.put(11, tS);
      }
      stage.template sum<TAN>(mask, pb, 12, sums[1 + tk]);
    }
  }
  // the warps' sums into the block's: share s = 2 k (value) or 2 k + 1
  // (tangent) of parameter k of the tile, ordered pair p
  const int k = lane >> 1, half = (lane & 1) * PG_NPARAM;
#pragma unroll
  for (int p = 0; p < 4; ++p) {
    if (k < 13) {
      const int at = k == 0 ? PG_A + p : k == 1 ? PG_B + p : k == 2 ? PG_L1 + p : k == 3 ? PG_L2 + p : k == 4 ? PG_KAPPA + p
                   : k == 5 ? PG_R + p : k == 6 ? PG_S + p : k == 7 ? PG_SIGMA + p : k == 8 ? PG_P + p
                   : k < 11 ? PG_G + 2 * p + (k - 9) : PG_N + 2 * p + (k - 11);
      if (sums[0][p] != 0.0) atomicAdd(&s_g[half + at], sums[0][p]);
    }
    if (k < 12) {
#pragma unroll
      for (int tk = 0; tk < 2; ++tk) {
        const int tri = 2 * p + tk, pk = (p & 2) + tk, ll = k & 1;
        const int at = k < 2 ? PG_GAMMA + 2 * tri + ll : k < 4 ? PG_C + 2 * tri + ll : k < 6 ? PG_D + 2 * tri + ll
                     : k < 8 ? PG_H + 2 * tri + ll : k < 10 ? PG_ALPHA + 2 * tri + ll : k == 10 ? PG_R + pk : PG_S + pk;
        if (sums[1 + tk][p] != 0.0) atomicAdd(&s_g[half + at], sums[1 + tk][p]);
      }
    }
  }
  __syncthreads();
  for (int k = threadIdx.x; k < 2 * PG_NPARAM; k += blockDim.x)
    if (s_g[k] != 0.0) atomicAdd(grad + k, s_g[k]);
}

// Charge-kernel and self-energy parameters, G lanes per atom (each unordered
// pair appears in both atoms' lists, hence the 1/2 of the energy). With
// iD = (r^3 + gamma^-3)^(-1/3), T the taper and x = r / Rc, an entry needs
//   k = T iD                      K = ke k
//   m = -r T'(x) iD / Rc^2        dK/dRc = ke m
//   g = T iD^4                    dK/dgamma = ke gamma^-3 g / (2 gamma)
// (gamma^-3 = (gamma_i gamma_j)^(-3/2)); only their sums over j weighted by q_j
// are kept, g's by the type of j, and the parameters and q_i applied once per
// atom. DIR: distances carry their derivatives tr along dir, and with d/dr of
// the three the sums' tangents follow; vout_i gets the Coulomb share of
// d(Hq + chi)_i/de, ke sum_j q_j k' tr. QDIR: the charges carry theirs. (The
// general dual numbers with a power, a cube root and six divisions per entry,
// one thread per atom, took 6.5 ms in FP64 on 6,278 atoms; this 0.39 along dir,
// 0.28 along q.)
#define PC_T 256
#define PC_G 8
template <class R, bool DIR, bool QDIR>
__global__ void __launch_bounds__(PC_T)
    k_pgrad_coul(int N, int ld, const typename Vec4<R>::T* __restrict__ u, const int* __restrict__ rep,
                 const RepInfo* __restrict__ reps, const int2* __restrict__ nl, const int* __restrict__ nall,
                 const double* __restrict__ q, const double* __restrict__ qdir, const double* __restrict__ wval,
                 const double* __restrict__ wtan, const double* __restrict__ dir, ParamsT<R> P, R gs00, R gs01, R gs11,
                 double* __restrict__ grad, double* __restrict__ vout) {
  using R4 = typename Vec4<R>::T;
  constexpr int AW = 32 / PC_G, AB = PC_T / PC_G;
  constexpr int NV = 4;            // sums of k, m, g (j Si), g (j C)
  constexpr bool TAN = DIR || QDIR;
  __shared__ R s_v[TAN ? 2 * NV : NV][AB];
  const int lane = threadIdx.x & 31, warp = threadIdx.x >> 5, a = lane % AW, l = lane / AW;
  const int i = ((int)blockIdx.x * (PC_T / 32) + warp) * AW + a;
  R v[NV], t[NV];
#pragma unroll
  for (int k = 0; k < NV; ++k) v[k] = t[k] = R(0);
  double vi = 0.0;
  bool on = i < N;
  if (on) on = wval[rep[i]] != 0.0 || (wtan && wtan[rep[i]] != 0.0);
  if (on) {
    const R4 ui = u[i];
    const int ti = (int)ui.w;
    const R g0 = ti ? gs01 : gs00, g1 = ti ? gs11 : gs01;
    const RepInfo& ri = reps[rep[i]];
    const R rc = P.r_coul, irc = R(1) / rc, irc2 = irc * irc, rc2 = rc * rc;
    R gix = 0, giy = 0, giz = 0;
    if (DIR) { gix = (R)dir[3 * i]; giy = (R)dir[3 * i + 1]; giz = (R)dir[3 * i + 2]; }
    const int na = nall[i];
    for (int e = l; e < na; e += PC_G) {
      const int2 jc = __ldg(nl + (size_t)e * ld + i);
      const int j = jc.x;
      const R4 uj = u[j];
      const R qj = (R)q[j], qt = QDIR ? (R)qdir[j] : R(0);
      R rx, ry, rz;
      bond_vec<R>(ui, uj, jc.y, ri, rx, ry, rz);
      const R r2 = rx * rx + ry * ry + rz * rz;
      if (past_cut(r2, rc2)) continue;
      const R ir = ct_rsqrt<R>(r2), r = r2 * ir;
      const bool cj = uj.w != R(0);
      const R x = r * irc, x2 = x * x, xm = x - R(1), xm2 = xm * xm;
      const R T = R(1) + (x2 * x2) * (R(-35) + x * (R(84) + x * (R(-70) + R(20) * x)));
      const R dT = R(140) * (x2 * x) * (xm2 * xm);   // dT/dx
      const R iD = ct_rcbrt<R>(r2 * r + (cj ? g1 : g0)), iD2 = iD * iD, iD4 = iD2 * iD2;
      const R k = T * iD, m = -irc2 * (r * dT) * iD, g = T * iD4;
      v[0] += qj * k;
      v[1] += qj * m;
      const R qg = qj * g;
      v[2] += cj ? R(0) : qg;
      v[3] += cj ? qg : R(0);
      if (QDIR) {
        t[0] += qt * k;
        t[1] += qt * m;
        const R tg = qt * g;
        t[2] += cj ? R(0) : tg;
        t[3] += cj ? tg : R(0);
      }
      if (DIR) {
        const R tr = (rx * ((R)dir[3 * j] - gix) + ry * ((R)dir[3 * j + 1] - giy) + rz * ((R)dir[3 * j + 2] - giz)) * ir;
        // d/dr: iD' = -r^2 iD^4, T' = dT / Rc, (dT)' = 420 x^2 (x - 1)^2 (2 x - 1) / Rc
        const R Tp = dT * irc, r2D3 = r2 * (iD2 * iD);
        const R kp = iD * (Tp - T * r2D3);
        const R mp = -irc2 * iD * (dT + r * (R(420) * irc) * (x2 * xm2) * (x + xm) - r * dT * r2D3);
        const R gp = iD4 * (Tp - R(4) * T * r2D3);
        const R qr = qj * tr;
        t[0] += qr * kp;
        t[1] += qr * mp;
        const R tg = qr * gp;
        t[2] += cj ? R(0) : tg;
        t[3] += cj ? tg : R(0);
        vi += (double)(kp * tr) * (double)qj;
      }
    }
  }
#pragma unroll
  for (int o = AW; o < 32; o <<= 1) {
#pragma unroll
    for (int k = 0; k < NV; ++k) {
      v[k] += __shfl_xor_sync(CT_FULL, v[k], o);
      if (TAN) t[k] += __shfl_xor_sync(CT_FULL, t[k], o);
    }
    if (DIR) vi += __shfl_xor_sync(CT_FULL, vi, o);
  }
  if (l == 0) {
#pragma unroll
    for (int k = 0; k < NV; ++k) {
      s_v[k][warp * AW + a] = v[k];
      if (TAN) s_v[NV + k][warp * AW + a] = t[k];
    }
    if (DIR && vout && on && vi != 0.0) atomicAdd(vout + i, (double)P.k_e * vi);
  }
  __syncthreads();
  // one warp: the block's atoms (AB = 32), a lane each, in FP64
  if (warp != 0) return;
  const int ie = (int)blockIdx.x * AB + lane;
  double wv = 0.0, wt = 0.0, qi = 0.0, qd = 0.0;
  int ti = 0;
  if (ie < N) {
    wv = wval[rep[ie]];
    wt = TAN && wtan ? wtan[rep[ie]] : 0.0;
    qi = q[ie];
    qd = QDIR ? qdir[ie] : 0.0;
    ti = (int)u[ie].w;
  }
  const double ke = (double)P.k_e, ga = (double)P.gamma_c[0], gb = (double)P.gamma_c[1];
  // sum over j of w K-like terms with w = q_i q_j / 2 (and its tangent)
  auto term = [&](int k, double& val, double& tan) {
    val = 0.5 * qi * (double)s_v[k][lane];
    tan = TAN ? 0.5 * (qd * (double)s_v[k][lane] + qi * (double)s_v[NV + (TAN ? k : 0)][lane]) : 0.0;
  };
  auto put = [&](int at, double val, double tan) {
    const double sv = pair_sum(wv * val, TAN ? wt * tan : 0.0);   // lanes 0..15 the value, 16..31 the tangent
    if (lane == 0 && sv != 0.0) atomicAdd(grad + at, sv);
    if (TAN && lane == 16 && sv != 0.0) atomicAdd(grad + PG_NPARAM + at, sv);
  };
  double a0, b0, a1, b1;
  term(0, a0, b0);
  put(PG_KE, a0, b0);
  term(1, a0, b0);
  put(PG_RCOUL, ke * a0, ke * b0);
  // gamma: the pair (t_i, t_j) feeds both atoms' types
  term(2, a0, b0);
  term(3, a1, b1);
  const double c0 = 0.5 * ke * (double)(ti ? gs01 : gs00), c1 = 0.5 * ke * (double)(ti ? gs11 : gs01);
  a0 *= c0; b0 *= c0; a1 *= c1; b1 *= c1;
  put(PG_GAMMA_C, (ti == 0 ? 2.0 * a0 + a1 : a0) / ga, (ti == 0 ? 2.0 * b0 + b1 : b0) / ga);
  put(PG_GAMMA_C + 1, (ti == 1 ? 2.0 * a1 + a0 : a1) / gb, (ti == 1 ? 2.0 * b1 + b0 : b1) / gb);
#pragma unroll
  for (int ty = 0; ty < 2; ++ty) {
    const double is = ie < N && ti == ty ? 1.0 : 0.0;
    put(PG_E0 + ty, is, 0.0);
    put(PG_CHI + ty, is * qi, is * qd);
    put(PG_J + ty, is * qi * qi, is * 2.0 * qi * qd);
  }
}

// The force part of the loss and its derivative with respect to the forces.
__global__ void k_force_residual(int N, const double* __restrict__ F, const double* __restrict__ F_ref,
                                 const int* __restrict__ order, const int* __restrict__ rep,
                                 const double* __restrict__ wF, double* __restrict__ g, double* __restrict__ out) {
  const int i = blockIdx.x * blockDim.x + threadIdx.x;
  double loss = 0.0, m = 0.0;
  if (i < N) {
    const size_t k = order ? (size_t)order[i] : (size_t)i;
    const double w = wF[rep[i]];
    double d2 = 0.0;
#pragma unroll
    for (int c = 0; c < 3; ++c) {
      const double d = F[3 * (size_t)i + c] - F_ref[3 * k + c], gi = 2.0 * w * d;
      g[3 * (size_t)i + c] = gi;
      m = fmax(m, fabs(gi));
      d2 += d * d;
    }
    loss = w * d2;
  }
  loss = warp_sum(loss);
  m = warp_max(m);
  __shared__ double s_l[8], s_m[8];
  const int lane = threadIdx.x & 31, warp = threadIdx.x >> 5;
  if (lane == 0) {
    s_l[warp] = loss;
    s_m[warp] = m;
  }
  __syncthreads();
  if (threadIdx.x == 0) {
    for (int w = 1; w < 8; ++w) {
      loss += s_l[w];
      m = fmax(m, s_m[w]);
    }
    atomicAdd(out, loss);
    atomic_max_nonneg(out + 1, m);
  }
}

__global__ void k_adjoint_rhs(int N, int R, double* __restrict__ v, double* __restrict__ vmax, double* __restrict__ cg,
                              int* __restrict__ hist) {
  const int i = blockIdx.x * blockDim.x + threadIdx.x;
  double m = 0.0;
  if (i < N) {
    v[i] = -v[i];
    m = fabs(v[i]);
  }
  m = warp_max(m);
  if ((threadIdx.x & 31) == 0 && m > 0.0) atomic_max_nonneg(vmax, m);
  if (i < R) cg[(size_t)i * CG_STRIDE + CG_Q] = 0.0;
  if (i == 0) *hist = 0;
}

// ---------------------------------------------------------------- launchers
void launch_force_residual(const DevState& S, const double* F_ref, const int* order, const double* wF, double* g,
                           double* out, cudaStream_t st) {
  if (S.N == 0) return;
  k_force_residual<<<(S.N + 255) / 256, 256, 0, st>>>(S.N, S.F, F_ref, order, S.rep, wF, g, out);
}

void launch_adjoint_rhs(const DevState& S, double* v, double* vmax, cudaStream_t st) {
  const int n = std::max(S.N, S.R);
  k_adjoint_rhs<<<(n + 255) / 256, 256, 0, st>>>(S.N, S.R, v, vmax, S.cg, S.cg_hist);
}

template <class R, class S>
static cudaError_t pgrad_launch(const DevState& D, const ParamsT<R>& P, const ctbop_params& P64, const double* wval, const double* wtan,
                                const double* dir, const double* qdir, double* grad, double* vout,
                                cudaStream_t st) {
  using R4 = typename Vec4<R>::T;
  PgConst<R> K;
  for (int k = 0; k < 4; ++k) {
    const double p = P64.p[k], g0 = P64.g[k][0], g1 = P64.g[k][1], s0 = std::pow(g0, -p), s1 = std::pow(g1, -p), S0 = s0 + s1;
    K.lnS0[k] = (R)std::log(S0);
    K.dlnS0_dp[k] = (R)(-(s0 * std::log(g0) + s1 * std::log(g1)) / S0);
    K.dg[k][0] = (R)(p * std::pow(g0, -p - 1.0) / S0);
    K.dg[k][1] = (R)(p * std::pow(g1, -p - 1.0) / S0);
  }
  for (int t = 0; t < 8; ++t)
    for (int l = 0; l < 2; ++l) K.id2[t][l] = (R)(1.0 / (P64.d[t][l] * P64.d[t][l]));
  // blocks of 128 threads, or of 32 where the covalent entries of their atoms
  // need more shared memory than a block can have
  auto cov = [&](auto kernel, int threads, bool& fits) -> cudaError_t {
    const int apb = threads / PgLanes<R>::v;
    const size_t sm = (size_t)apb * D.cap_cov * (sizeof(Ent<R>) + 3 * sizeof(int));
    size_t most = 0;
    cudaError_t e = allow_dynamic_smem((const void*)kernel, &most);
    if (e != cudaSuccess) return e;
    fits = sm <= most;
    if (!fits) return threads > 32 ? cudaSuccess : cudaErrorInvalidValue;
    kernel<<<(D.N + apb - 1) / apb, threads, sm, st>>>(D.N, D.cap_cov, D.ld, (const R4*)D.u, D.rep, D.reps, D.nl,
                                                          D.ncov, D.q, qdir, wval, wtan, dir, P, K, grad, vout);
    return cudaGetLastError();
  };
  bool fits = false;
  cudaError_t e = cov(k_pgrad_cov<R, S, PG_T>, PG_T, fits);
  if (e == cudaSuccess && !fits) e = cov(k_pgrad_cov<R, S, 32>, 32, fits);
  if (e != cudaSuccess) return e;
  // gamma^-3 of the pair types
  const double ga = P64.gamma_c[0], gb = P64.gamma_c[1];
  const R gs00 = (R)std::pow(ga * ga, -1.5), gs01 = (R)std::pow(ga * gb, -1.5), gs11 = (R)std::pow(gb * gb, -1.5);
  auto coul = [&](auto kernel) {
    kernel<<<(D.N + PC_T / PC_G - 1) / (PC_T / PC_G), PC_T, 0, st>>>(D.N, D.ld, (const R4*)D.u, D.rep, D.reps, D.nl, D.nall,
                                                                   D.q, qdir, wval, wtan, dir, P, gs00, gs01, gs11, grad,
                                                                   vout);
  };
  if (dir && qdir) coul(k_pgrad_coul<R, true, true>);
  else if (dir) coul(k_pgrad_coul<R, true, false>);
  else if (qdir) coul(k_pgrad_coul<R, false, true>);
  else coul(k_pgrad_coul<R, false, false>);
  return cudaGetLastError();
}

template <class R>
static cudaError_t pgrad_prec(const DevState& D, const ctbop_params& P, const double* wval, const double* wtan,
                              const double* dir, const double* qdir, double* grad, double* vout,
                              cudaStream_t st) {
  ParamsT<R> Pr;
  const double* src = reinterpret_cast<const double*>(&P);
  R* dst = reinterpret_cast<R*>(&Pr);
  for (int k = 0; k < PG_NPARAM; ++k) dst[k] = (R)src[k];
  if (dir || qdir) return pgrad_launch<R, DualT<R>>(D, Pr, P, wval, wtan, dir, qdir, grad, vout, st);
  return pgrad_launch<R, R>(D, Pr, P, wval, nullptr, nullptr, nullptr, grad, nullptr, st);
}

cudaError_t launch_param_grad(const DevState& D, const ctbop_params& P, bool fp32, const double* wval,
                              const double* wtan, const double* dir, const double* qdir, double* grad,
                              double* vout, cudaStream_t st) {
  cudaError_t e = cudaMemsetAsync(grad, 0, sizeof(double) * 2 * PG_NPARAM, st);
  if (e == cudaSuccess && vout) e = cudaMemsetAsync(vout, 0, sizeof(double) * std::max(D.N, 1), st);
  if (e != cudaSuccess || D.N == 0) return e;
  if (fp32) return pgrad_prec<float>(D, P, wval, wtan, dir, qdir, grad, vout, st);
  return pgrad_prec<double>(D, P, wval, wtan, dir, qdir, grad, vout, st);
}

}  // namespace ct
