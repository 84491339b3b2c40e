// diff1d.cu - the three-stage diffusion solver of Sec. 2 on the GPU (sm_103a), batched
// over independent 1D instances; FP64.
//
// One step (Eq. limit_U_dis1 - Eq. limit_UT_dis3, fully discrete as Eq. dis-diff; for
// sigma_0/T^3 the fully discrete form after Eq. marshak-diff2):
//   stage 1 (prediction)  (U*_j - U_j)/dt = f_j [k_{j+1} (U*_{j+1} - U*_j) - k_j (U*_j - U*_{j-1})],
//                         f = 4T^3/(4aT^3 + C_v), k_i = a c kappa_i / (D sigma_i dx^2) at node i,
//                         kappa_i = 1 (sigma(x)) or the node mean of T^3 (sigma_0/T^3),
//                         sigma_i the harmonic node mean, k = 0 at the two walls (zero flux):
//                         one tridiagonal solve per instance;
//   stage 2 (correction)  a (T^4 - T_n^4)/dt + C_v (T - T_n)/dt = k*_{j+1} (U*_{j+1} - U*_j) - k*_j (U*_j - U*_{j-1}),
//                         k* with kappa* = the node mean of max(U*, 0)^{3/4} (sigma_0/T^3) or k:
//                         a per-cell quartic, solved by monotone Newton;
//   stage 3 (projection)  U = T^4.
// Instances of up to kFN kFQ = 8192 cells run k_diff: one cluster per instance, all three
// stages of many steps in one launch, the state in registers.  Larger ones run three
// launches per step: k_dcoef (per cell: U, f, node k), k_dsolve (one CTA per instance: the
// partitioned tridiagonal solver of tridiag.cuh, unknowns in global memory), k_dcorr (per
// cell: the correction's flux and Newton).
#include <cooperative_groups.h>
#include <cuda_runtime.h>

#include <algorithm>
#include <cmath>
#include <new>
#include <string>
#include <vector>

#include "../../include/grte.h"
#include "tridiag.cuh"

namespace cg = cooperative_groups;

namespace grte {
namespace {

constexpr int kDT = 256;   // threads per solve CTA

struct DInst {
  int64_t N, off;          // cells, offset into the cell arrays
  int64_t foff, roff;      // factor / reduced-system offsets
  double dt, dx, a, c, Cv, Dd;
  int kind;
};

struct DDev {
  const DInst* inst;
  double *sig, *T, *U, *f, *k, *Us, *x, *F, *Rd;
  int* status;
};

// u^{3/4} for u >= 0 as u u^{-1/4}: r = u^{-1/4} from binary32 and one third-order step,
// r (1-e)^{-1/4} = r (1 + e/4 + 5 e^2/32 + ...), e = 1 - u r^4 < 2^-19; outside the
// binary32 range the library power.
__device__ __forceinline__ double d_pow34(double u) {
  const float f = (float)u;
  if (!(f > 1e-30f && f < 1e30f)) return u > 0.0 ? pow(u, 0.75) : 0.0;
  const double r = (double)rsqrtf(sqrtf(f));
  const double r2 = r * r;
  const double e = fma(-u * r2, r2, 1.0);
  return u * fma(r, e * fma(e, 0.15625, 0.25), r);
}

// The positive root of t^4 + beta t = R (beta, R > 0): Newton from
// T_hi = min(R^{1/4}, R/beta), monotone (convex increasing left side).  T_hi is at most 1.381
// times the root (at beta = R^{3/4}, t^4 + t = 1), from where exact Newton errors go 0.10,
// 9.3e-3, 7.8e-5, 5.5e-9: within the binary32 range five steps there reach its rounding, and two
// binary64 steps, their slope's reciprocal in binary32, finish: 2e-7 -> 6e-14 -> rounding (worst
// 4.4e-16 over 2e6 arguments of the whole range).  Elsewhere all steps are binary64, until t
// stops decreasing; false if maxit steps do not suffice.
__device__ __forceinline__ bool d_root(double beta, double R, int maxit, double& t) {
  const float rf = (float)R, bf = (float)beta;
  if (rf > 1e-20f && rf < 1e20f && bf > 1e-20f && bf < 1e20f) {
    float tf = fminf(sqrtf(sqrtf(rf)), __fdividef(rf, bf));
#pragma unroll
    for (int it = 0; it < 5; ++it) {
      const float t3 = tf * tf * tf;
      tf -= __fdividef(tf * (t3 + bf) - rf, 4.0f * t3 + bf);
    }
    if (tf > 1e-20f) {
      t = (double)tf;
#pragma unroll
      for (int it = 0; it < 2; ++it) {
        const double t3 = t * t * t;
        const double f = fma(t, t3 + beta, -R);
        t = fma(-f, (double)__frcp_rn((float)fma(4.0, t3, beta)), t);
      }
      return true;
    }
  }
  t = fmin(sqrt(sqrt(R)), R / beta);
  int it = 0;
  for (; it < maxit; ++it) {
    const double t2 = t * t;
    const double tn = t - (t2 * t2 + beta * t - R) / (4.0 * t2 * t + beta);
    if (!(tn < t)) break;
    t = tn;
  }
  return it < maxit;
}

// The correction's root at one cell and its statuses: a (T^4 - T_n^4) + C_v (T - T_n) = dt flux
// as T^4 + beta T = U_n + beta T_n + dt flux/a, beta = C_v/a.
__device__ __forceinline__ double d_correct(double beta, double R, int maxit, int& status) {
  double t = 0.0;
  if (!(R > 0.0)) {
    status |= 1 << (R <= 0.0 ? GRTE_ENEGATIVE : GRTE_ENAN);
  } else if (!d_root(beta, R, maxit, t)) {
    status |= 1 << GRTE_ENONCONV;
  }
  if (!isfinite(t)) status |= 1 << GRTE_ENAN;
  return t;
}

__device__ __forceinline__ int inst_of(const DInst* in, int n, int64_t g) {
  int lo = 0, hi = n - 1;
  while (lo < hi) {
    const int mid = (lo + hi + 1) >> 1;
    if (in[mid].off <= g) lo = mid; else hi = mid - 1;
  }
  return lo;
}

// per cell: U = T^4, f = 4T^3/(4aT^3 + Cv), k at the cell's left node (0 at the wall)
__global__ void k_dcoef(DDev D, int n_inst, int64_t ncell) {
  const int64_t g = blockIdx.x * (int64_t)blockDim.x + threadIdx.x;
  if (g >= ncell) return;
  const DInst I = D.inst[inst_of(D.inst, n_inst, g)];
  const int64_t j = g - I.off;
  const double T = D.T[g], T3 = T * T * T;
  D.U[g] = T3 * T;
  D.f[g] = 4.0 * T3 / (4.0 * I.a * T3 + I.Cv);
  double k = 0.0;
  if (j >= 1) {
    const double sl = D.sig[g - 1], sr = D.sig[g];
    const double sn = 2.0 * sl * sr / (sl + sr);
    double kap = 1.0;
    if (I.kind == GRTE_SIGMA_T3) {
      const double Tl = D.T[g - 1];
      kap = 0.5 * (Tl * Tl * Tl + T3);
    }
    k = I.a * I.c * kap / (I.Dd * sn * I.dx * I.dx);
  }
  D.k[g] = k;
  D.x[g] = D.U[g] / I.dt;   // right-hand side of stage 1
}

struct DCoef {   // stage-1 matrix of one instance
  const double *f, *k;
  double idt;
  int64_t N;
  __device__ double kr(int64_t j) const { return j + 1 < N ? k[j + 1] : 0.0; }
  __device__ double a(int64_t j) const { return j > 0 ? -f[j] * k[j] : 0.0; }
  __device__ double c(int64_t j) const { return j + 1 < N ? -f[j] * k[j + 1] : 0.0; }
  __device__ double b(int64_t j) const { return idt + f[j] * (k[j] + kr(j)); }
};

__global__ void __launch_bounds__(kDT) k_dsolve(DDev D) {
  extern __shared__ __align__(16) unsigned char dsm[];
  const DInst I = D.inst[blockIdx.x];
  DCoef cf{D.f + I.off, D.k + I.off, 1.0 / I.dt, I.N};
  XAcc<double, false> xa{D.x + I.off};
  tri_solve<true>(cf, I.N, xa, D.F + I.foff, D.Rd + I.roff, (double*)dsm);
}

// per cell: the correction's flux at U*, then (a/dt) T^4 + (C_v/dt) T = (a/dt) U_n + (C_v/dt) T_n + flux
__global__ void k_dcorr(DDev D, int n_inst, int64_t ncell, int maxit) {
  const int64_t g = blockIdx.x * (int64_t)blockDim.x + threadIdx.x;
  if (g >= ncell) return;
  const int ii = inst_of(D.inst, n_inst, g);
  const DInst I = D.inst[ii];
  const int64_t j = g - I.off, N = I.N;
  const double* Us = D.x + I.off;   // the solution of stage 1
  auto knode = [&](int64_t i) -> double {   // k* at node i (cells i-1, i)
    if (i < 1 || i > N - 1) return 0.0;
    if (I.kind != GRTE_SIGMA_T3) return D.k[I.off + i];
    const double sl = D.sig[I.off + i - 1], sr = D.sig[I.off + i];
    const double sn = 2.0 * sl * sr / (sl + sr);
    const double kap = 0.5 * (d_pow34(fmax(Us[i - 1], 0.0)) + d_pow34(fmax(Us[i], 0.0)));
    return I.a * I.c * kap / (I.Dd * sn * I.dx * I.dx);
  };
  const double uj = Us[j];
  double flux = 0.0;
  if (j + 1 < N) flux += knode(j + 1) * (Us[j + 1] - uj);
  if (j >= 1) flux -= knode(j) * (uj - Us[j - 1]);
  D.Us[g] = uj;
  const double Tn = D.T[g];
  const double beta = I.Cv / I.a;
  int status = 0;
  const double t = d_correct(beta, D.U[g] + beta * Tn + I.dt / I.a * flux, maxit, status);
  if (status) atomicOr(D.status, status);
  D.T[g] = t;
}

// ----------------------------------------------------------------------------- one kernel
constexpr int kFT = 128;           // threads per CTA
constexpr int kFC = 4;             // cells per thread
constexpr int kFN = kFT * kFC;     // cells per CTA
constexpr int kFQ = 16;            // largest cluster
constexpr int kFSteps = 64;        // steps per launch at most
constexpr int64_t kStageCells = 1 << 20;   // pinned staging of at most 8 MB per handle

struct DSmem {
  double A[kFT], B[kFT], C[kFT], R[kFT];   // separator rows
  double n0[kFT], n1[kFT], n2[kFT];        // each thread's first unknown in terms of its separators
  double sep[kFT + 1];                     // [0]: the separator left of this CTA
  double xf[kFT], vf[kFT], vl[kFT];        // U* and V of each thread's first cell, V of its last
  double ef[kFT], el[kFT];                 // T^3 of each thread's first and last cell
  double cx;                               // coupling of the last separator to the next CTA's first cell
  double nxt;                              // U* of the next CTA's first cell
  double pub[7];                           // published to the cluster: f0 f1 f2, A B R of the CTA's row, cx
};

// Eliminate the first three of four consecutive unknowns: x_u = rc_u - cc_u x_3 - ac_u x_L
// (x_L: the unknown left of the four); A, B, R: row 3 with x_2 inserted (its coupling to
// the right is still c[3]).
struct DChunk { double rc[3], cc[3], ac[3]; };
__device__ __forceinline__ void d_eliminate(const double* a, const double* b, const double* c, const double* r,
                                            DChunk& k, double& A, double& B, double& R) {
  double inv = rcp64(b[0]);
  k.ac[0] = a[0] * inv;
  k.cc[0] = c[0] * inv;
  k.rc[0] = r[0] * inv;
#pragma unroll
  for (int u = 1; u < 3; ++u) {
    inv = rcp64(fma(-a[u], k.cc[u - 1], b[u]));
    k.ac[u] = -a[u] * k.ac[u - 1] * inv;
    k.cc[u] = c[u] * inv;
    k.rc[u] = fma(-a[u], k.rc[u - 1], r[u]) * inv;
  }
#pragma unroll
  for (int u = 1; u >= 0; --u) {
    const double q = k.cc[u];
    k.rc[u] = fma(-q, k.rc[u + 1], k.rc[u]);
    k.ac[u] = fma(-q, k.ac[u + 1], k.ac[u]);
    k.cc[u] = -q * k.cc[u + 1];
  }
  A = -a[3] * k.ac[2];
  B = fma(-a[3], k.cc[2], b[3]);
  R = fma(-a[3], k.rc[2], r[3]);
}

// The power of two s with 1 <= den s < 2 (den > 0; at the ends of the range the nearest one).
__device__ __forceinline__ double d_inv_scale(double den) {
  const int e = __double2hiint(den) & 0x7ff00000;
  return __hiloint2double(max(0x7fe00000 - e, 0x00100000), 0);
}

// Whether T >= 0 lies outside [2^-128, 2^128) (integer operations only; false for 0 and denormals,
// whose T^3 and T^4 are 0).
__device__ __forceinline__ bool d_far(double T) {
  const int h = __double2hiint(T) >> 20;
  return h > 0 && (unsigned)(h - 1023 + 128) >= 256u;
}

// Parallel cyclic reduction over lanes [0, n) of a warp, rows with unit diagonal:
// x_i + a x_{i-1} + c x_{i+1} = r.  A coupling beyond either end is kept: afterwards
// x_i = r - a x_{-1} - c x_n.
__device__ __forceinline__ void d_pcr(int lane, int n, double& a, double& c, double& r) {
  for (int s = 1; s < n; s <<= 1) {
    const double aL = __shfl_up_sync(~0u, a, s), cL = __shfl_up_sync(~0u, c, s), rL = __shfl_up_sync(~0u, r, s);
    const double aR = __shfl_down_sync(~0u, a, s), cR = __shfl_down_sync(~0u, c, s),
                 rR = __shfl_down_sync(~0u, r, s);
    const bool hasL = lane >= s, hasR = lane + s < n;
    double b = 1.0, an = a, cn = c;
    if (hasL) {
      b = fma(-a, cL, b);
      r = fma(-a, rL, r);
      an = -a * aL;
    }
    if (hasR) {
      b = fma(-c, aR, b);
      r = fma(-c, rR, r);
      cn = -c * cR;
    }
    const double inv = rcp64(b);
    a = an * inv;
    c = cn * inv;
    r *= inv;
  }
}

// nsteps steps of one instance per cluster of Q = ceil(N/512) CTAs: CTA q holds cells
// [512 q, 512 q + 512), four consecutive ones per thread, T and the node factors in registers.
// Stage 1 multiplied by dt (a T^3 + C_v/4) = dt den needs no division per cell:
//   [den + T^3 (k_j + k_{j+1})] U*_j - T^3 (k_j U*_{j-1} + k_{j+1} U*_{j+1}) = den U_j,
// or, where den U_j ~ T^7 might leave the range before U_j does, that row scaled by a power of two
// (a branch on exponents: scaling always takes 2.7% more, the check 0.4%, with the same bits).
// Four levels of elimination, the last unknown of each group kept as its separator: 4 cells
// per thread; 4 threads' separators per lane of warp 0; 31 lanes by cyclic reduction with the
// couplings to both ends carried along; one row per CTA, gathered by every CTA's warp 0.
//
// Bound: the binary64 pipe (2 lanes a clock and SM), about 75 operations per cell and step;
// hence the binary32 starts of reciprocals, powers and Newton, and one warp for the
// separators (a reduction over all four warps costs four times the issue slots).  Two
// cluster barriers a step (T^3 of the neighbour cells, the CTA rows); a cluster of one has
// none.  512 cells per CTA so that uneven batches spread over the SMs and the longest
// instance over 16 of them.
// 64 uneven runs (155,000 cells), 50 steps: 14.8 ms as three launches a step (171 us in the
// correction, 108 in the solve, 18 in the coefficients), 1.87 ms as one kernel; 20 us a
// step is the binary64 rate for those operations, 37 are taken (2 or 3 CTAs an SM).
__global__ void __launch_bounds__(kFT) k_diff(DDev D, int first, int Q, int nsteps, int maxit) {
  __shared__ DSmem sm;
  cg::cluster_group cl = cg::this_cluster();
  const int t = threadIdx.x, lane = t & 31, q = blockIdx.x % Q;
  const DInst I = D.inst[first + blockIdx.x / Q];
  const bool t3k = I.kind == GRTE_SIGMA_T3;
  const int64_t j0 = (int64_t)q * kFN + t * kFC;
  const double beta = I.Cv / I.a, c4 = 0.25 * I.Cv, ia = 1.0 / I.a;
  double T[kFC], g[kFC + 1];   // g: node factors dt a c/(D sigma dx^2) (halved for the mean of T^3)
  const double gc = I.dt / (I.Dd * I.dx * I.dx) * (t3k ? 0.25 : 0.5);
#pragma unroll
  for (int u = 0; u < kFC; ++u) T[u] = j0 + u < I.N ? D.T[I.off + j0 + u] : 0.0;
#pragma unroll
  for (int u = 0; u <= kFC; ++u) {
    const int64_t i = j0 + u;
    g[u] = 0.0;
    if (i >= 1 && i < I.N) {
      const double sl = D.sig[I.off + i - 1], sr = D.sig[I.off + i];
      g[u] = gc * (I.a * I.c * (sl + sr) / (sl * sr));   // (no product of more than two sigma)
    }
  }
  // what no T in [2^-128, 2^128) needs the scaled rows for
  bool far0 = !(I.a > 0x1p-100 && I.a < 0x1p100 && c4 > 0x1p-100 && c4 < 0x1p100);
#pragma unroll
  for (int u = 0; u <= kFC; ++u) far0 = far0 || !(g[u] < 0x1p100);
  int status = 0;
  for (int n = 0; n < nsteps; ++n) {
    DChunk k;
    double A, B, R, U[kFC], cx;
    {
      double T3[kFC], kn[kFC + 1];
      bool far = far0;
#pragma unroll
      for (int u = 0; u < kFC; ++u) {
        T3[u] = T[u] * T[u] * T[u];
        U[u] = T3[u] * T[u];
        far = far || d_far(T[u]);
      }
      if (t3k) {
        sm.ef[t] = T3[0];
        sm.el[t] = T3[kFC - 1];
      }
      if (Q > 1) cl.sync();
      else __syncthreads();
#pragma unroll
      for (int u = 0; u <= kFC; ++u) kn[u] = g[u];
      if (t3k) {
        const double eL = t > 0 ? sm.el[t - 1] : (q > 0 ? cl.map_shared_rank(sm.el, q - 1)[kFT - 1] : 0.0);
        const double eR = t < kFT - 1 ? sm.ef[t + 1] : (q < Q - 1 ? cl.map_shared_rank(sm.ef, q + 1)[0] : 0.0);
#pragma unroll
        for (int u = 0; u <= kFC; ++u) kn[u] *= (u > 0 ? T3[u - 1] : eL) + (u < kFC ? T3[u] : eR);
      }
      double a[kFC], b[kFC], c[kFC], r[kFC];
#pragma unroll
      for (int u = 0; u < kFC; ++u) {
        const double den = fma(I.a, T3[u], c4);
        a[u] = -T3[u] * kn[u];
        c[u] = -T3[u] * kn[u + 1];
        b[u] = den - (a[u] + c[u]);
        r[u] = den * U[u];
      }
      if (far) {
        // the rows times the power of two that brings den to [1, 2): exact, and den U* stays in
        // range wherever U* does
#pragma unroll
        for (int u = 0; u < kFC; ++u) {
          const double den = fma(I.a, T3[u], c4), s = d_inv_scale(den), T3s = T3[u] * s, dens = den * s;
          a[u] = -T3s * kn[u];
          c[u] = -T3s * kn[u + 1];
          b[u] = dens - (a[u] + c[u]);
          r[u] = dens * U[u];
        }
      }
      d_eliminate(a, b, c, r, k, A, B, R);
      cx = c[kFC - 1];
    }
    sm.n0[t] = k.rc[0];
    sm.n1[t] = k.cc[0];
    sm.n2[t] = k.ac[0];
    __syncthreads();
    double C = 0.0;
    if (t < kFT - 1) {
      R = fma(-cx, sm.n0[t + 1], R);
      C = -cx * sm.n1[t + 1];
      B = fma(-cx, sm.n2[t + 1], B);
    } else {
      sm.cx = cx;
    }
    sm.A[t] = A;
    sm.B[t] = B;
    sm.C[t] = C;
    sm.R[t] = R;
    __syncthreads();
    DChunk kb;
    double la = 0.0, lc = 0.0, lr = 0.0;
    if (t < 32) {
      double a[4], b[4], c[4], r[4];
#pragma unroll
      for (int v = 0; v < 4; ++v) {
        a[v] = sm.A[4 * lane + v];
        b[v] = sm.B[4 * lane + v];
        c[v] = sm.C[4 * lane + v];
        r[v] = sm.R[4 * lane + v];
      }
      d_eliminate(a, b, c, r, kb, A, B, R);
      const double m0 = __shfl_down_sync(~0u, kb.rc[0], 1), m1 = __shfl_down_sync(~0u, kb.cc[0], 1),
                   m2 = __shfl_down_sync(~0u, kb.ac[0], 1);
      if (lane < 31) {   // lane 31's separator is the CTA's: its row stays as it is
        const double inv = rcp64(fma(-c[3], m2, B));
        la = A * inv;
        lc = -c[3] * m1 * inv;
        lr = fma(-c[3], m0, R) * inv;
      }
      d_pcr(lane, 31, la, lc, lr);
      // lane i < 31: s_i = lr - la S_{q-1} - lc S_q; row 31: A s_30 + B S_q + cx F_{q+1} = R
      const double y = __shfl_up_sync(~0u, lr, 1), ga = __shfl_up_sync(~0u, la, 1), gc = __shfl_up_sync(~0u, lc, 1);
      if (lane == 31) {
        sm.pub[3] = -A * ga;
        sm.pub[4] = fma(-A, gc, B);
        sm.pub[5] = fma(-A, y, R);
        sm.pub[6] = sm.cx;
      }
      if (lane == 0) {   // the CTA's first cell: F = f0 - f1 S_{q-1} - f2 S_q
        const double p0 = fma(-kb.cc[0], lr, kb.rc[0]), p1 = fma(-kb.cc[0], la, kb.ac[0]), p2 = -kb.cc[0] * lc;
        sm.pub[0] = fma(-k.cc[0], p0, k.rc[0]);
        sm.pub[1] = fma(-k.cc[0], p1, k.ac[0]);
        sm.pub[2] = -k.cc[0] * p2;
      }
      __syncwarp();
    }
    if (Q > 1) cl.sync();
    if (t < 32) {
      double S, SL = 0.0;
      if (Q > 1) {
        double a = 0.0, b = 1.0, c = 0.0, r = 0.0, f0 = 0.0, f1 = 0.0, f2 = 0.0;
        if (lane < Q) {
          const double* p = cl.map_shared_rank(sm.pub, lane);
          a = p[3];
          b = p[4];
          r = p[5];
          if (lane < Q - 1) {
            const double* p2 = cl.map_shared_rank(sm.pub, lane + 1);
            const double x = p[6];
            f0 = p2[0];
            f1 = p2[1];
            f2 = p2[2];
            b = fma(-x, f1, b);
            c = -x * f2;
            r = fma(-x, f0, r);
          }
        }
        const double inv = rcp64(b);
        a *= inv;
        c *= inv;
        r *= inv;
        d_pcr(lane, Q, a, c, r);
        const double F = f0 - f1 * r - f2 * __shfl_down_sync(~0u, r, 1);
        const double nx = __shfl_sync(~0u, F, q);
        S = __shfl_sync(~0u, r, q);
        SL = __shfl_sync(~0u, r, q > 0 ? q - 1 : 0);
        if (q == 0) SL = 0.0;
        if (lane == 0) sm.nxt = q < Q - 1 ? nx : 0.0;
      } else {
        S = sm.pub[5] * rcp64(sm.pub[4]);
        if (lane == 0) sm.nxt = 0.0;
      }
      const double s = lane < 31 ? lr - la * SL - lc * S : S;
      double sL = __shfl_up_sync(~0u, s, 1);
      if (lane == 0) {
        sL = SL;
        sm.sep[0] = SL;
      }
#pragma unroll
      for (int v = 0; v < 3; ++v) sm.sep[1 + 4 * lane + v] = kb.rc[v] - kb.cc[v] * s - kb.ac[v] * sL;
      sm.sep[4 + 4 * lane] = s;
    }
    __syncthreads();
    // U* of the thread's cells, then the fluxes at its five nodes and the correction
    double x[kFC], V[kFC];
    const double xL = sm.sep[t];
    x[kFC - 1] = sm.sep[t + 1];
#pragma unroll
    for (int u = 0; u < 3; ++u) x[u] = k.rc[u] - k.cc[u] * x[kFC - 1] - k.ac[u] * xL;
    if (t3k) {
#pragma unroll
      for (int u = 0; u < kFC; ++u) V[u] = d_pow34(fmax(x[u], 0.0));
      sm.vf[t] = V[0];
      sm.vl[t] = V[kFC - 1];
    }
    sm.xf[t] = x[0];
    __syncthreads();
    const double xR = t < kFT - 1 ? sm.xf[t + 1] : sm.nxt;
    double fl[kFC + 1];
#pragma unroll
    for (int u = 0; u <= kFC; ++u) fl[u] = g[u] * ((u < kFC ? x[u] : xR) - (u > 0 ? x[u - 1] : xL));
    if (t3k) {
      const double VL = t > 0 ? sm.vl[t - 1] : d_pow34(fmax(xL, 0.0));
      const double VR = t < kFT - 1 ? sm.vf[t + 1] : d_pow34(fmax(xR, 0.0));
#pragma unroll
      for (int u = 0; u <= kFC; ++u) fl[u] *= (u > 0 ? V[u - 1] : VL) + (u < kFC ? V[u] : VR);
    }
#pragma unroll
    for (int u = 0; u < kFC; ++u) {
      const bool live = j0 + u < I.N;
      if (live) T[u] = d_correct(beta, fma(ia, fl[u + 1] - fl[u], fma(beta, T[u], U[u])), maxit, status);
      if (live && n == nsteps - 1) {
        D.Us[I.off + j0 + u] = x[u];
        D.T[I.off + j0 + u] = T[u];
      }
    }
  }
  if (status) atomicOr(D.status, status);
  if (Q > 1) cl.sync();   // no CTA leaves while another may still read its shared memory
}

void diff_config(cudaLaunchConfig_t& cfg, cudaLaunchAttribute* at, int Q, int count, cudaStream_t st) {
  cfg = {};
  cfg.gridDim = dim3((unsigned)(count * Q));
  cfg.blockDim = dim3(kFT);
  cfg.stream = st;
  at[0].id = cudaLaunchAttributeClusterDimension;
  at[0].val.clusterDim.x = (unsigned)Q;
  at[0].val.clusterDim.y = at[0].val.clusterDim.z = 1;
  cfg.attrs = at;
  cfg.numAttrs = 1;
}

}  // namespace
}  // namespace grte

using namespace grte;

struct grte_diff_ctx {
  int n_inst = 0;
  int64_t ncell = 0;
  std::vector<DInst> inst;           // in the caller's order
  int n_big = 0;                     // instances beyond k_diff: the first of the device's order
  int64_t big_cells = 0;
  int fcnt[kFQ + 1] = {}, foff[kFQ + 1] = {};   // per cluster size: instances, first of them
  cudaStream_t side[kFQ] = {};       // launches of the smaller cluster sizes
  cudaEvent_t ev_fork = nullptr, ev_join[kFQ] = {};
  int* h_status = nullptr;           // pinned
  // pinned staging of the state, one slot per instance (null above kStageCells cells: then the
  // copies go to and from the caller's memory); a slot set since the last synchronisation
  // (stamp == epoch) may still be read by its copy
  double* h_state = nullptr;
  std::vector<int64_t> stamp;
  int64_t epoch = 0;
  DDev D{};
  DInst* d_inst = nullptr;
  cudaStream_t stream = nullptr;
  bool own_stream = false;
  std::vector<void*> allocs;
  std::string err;
  int newton_maxit = 60;
};

static grte_status dfail(grte_diff_t h, grte_status s, const std::string& m) {
  if (h) h->err = m;
  return s;
}
#define DCK(call)                                                                  \
  do {                                                                             \
    cudaError_t e_ = (call);                                                       \
    if (e_ != cudaSuccess) return dfail(h, GRTE_ECUDA, cudaGetErrorString(e_));    \
  } while (0)

template <typename T>
static bool dalloc_d(grte_diff_t h, T** p, int64_t n) {
  void* q = nullptr;
  if (cudaMalloc(&q, sizeof(T) * (size_t)std::max<int64_t>(n, 1)) != cudaSuccess) return false;
  h->allocs.push_back(q);
  *p = (T*)q;
  return true;
}

extern "C" {

void grte_diff_destroy(grte_diff_t h) {
  if (!h) return;
  if (h->stream) cudaStreamSynchronize(h->stream);
  for (void* p : h->allocs) cudaFree(p);
  for (cudaStream_t s : h->side) if (s) cudaStreamDestroy(s);
  for (cudaEvent_t e : h->ev_join) if (e) cudaEventDestroy(e);
  if (h->ev_fork) cudaEventDestroy(h->ev_fork);
  if (h->h_status) cudaFreeHost(h->h_status);
  if (h->h_state) cudaFreeHost(h->h_state);
  if (h->own_stream && h->stream) cudaStreamDestroy(h->stream);
  delete h;
}

const char* grte_diff_last_error(grte_diff_t h) { return h ? h->err.c_str() : "null handle"; }

grte_status grte_diff_create(int n_inst, const grte_diffusion1d* in, void* stream, grte_diff_t* out) {
  if (!out) return GRTE_EINVAL;
  *out = nullptr;
  if (n_inst <= 0 || !in) return GRTE_EINVAL;
  grte_diff_t h = new (std::nothrow) grte_diff_ctx();
  if (!h) return GRTE_ENOMEM;
  *out = h;
  for (int i = 0; i < n_inst; ++i) {
    const grte_diffusion1d& p = in[i];
    if (p.nx < 2 || p.nx > (1 << 24)) return dfail(h, GRTE_EINVAL, "nx must be in [2, 2^24]");
    if (!p.sigma) return dfail(h, GRTE_EINVAL, "sigma is NULL");
    if (p.sigma_kind != GRTE_SIGMA_CONST && p.sigma_kind != GRTE_SIGMA_T3) return dfail(h, GRTE_EINVAL, "bad sigma_kind");
    if (!(p.x1 > p.x0) || !(p.dt > 0) || !(p.a > 0) || !(p.c > 0) || !(p.Cv > 0))
      return dfail(h, GRTE_EINVAL, "x1 > x0, dt, a, c, Cv must be positive");
    for (int64_t j = 0; j < p.nx; ++j)
      if (!(p.sigma[j] > 0.0) || !std::isfinite(p.sigma[j])) return dfail(h, GRTE_EINVAL, "sigma must be positive");
    DInst I{};
    I.N = p.nx;
    I.dt = p.dt;
    I.dx = (p.x1 - p.x0) / (double)p.nx;
    I.a = p.a;
    I.c = p.c;
    I.Cv = p.Cv;
    I.Dd = p.dd > 0 ? p.dd : 3.0;
    I.kind = p.sigma_kind;
    h->inst.push_back(I);
  }
  // device order: the instances beyond k_diff, then the cluster sizes, largest first
  bool fits[kFQ + 1];   // a cluster of this size can be resident
  DCK(cudaFuncSetAttribute((const void*)k_diff, cudaFuncAttributeNonPortableClusterSizeAllowed, 1));
  for (int c = 1; c <= kFQ; ++c) {
    cudaLaunchConfig_t cfg;
    cudaLaunchAttribute at[1];
    diff_config(cfg, at, c, 1, nullptr);
    int n = 0;
    fits[c] = cudaOccupancyMaxActiveClusters(&n, (const void*)k_diff, &cfg) == cudaSuccess && n >= 1;
    if (!fits[c]) cudaGetLastError();
  }
  auto ctas = [&](int i) -> int {   // 0: beyond k_diff
    const int64_t c = (h->inst[i].N + kFN - 1) / kFN;
    return c <= kFQ && fits[c] ? (int)c : 0;
  };
  std::vector<int> order(n_inst);
  for (int i = 0; i < n_inst; ++i) order[i] = i;
  std::stable_sort(order.begin(), order.end(), [&](int x, int y) {
    const int a = ctas(x), b = ctas(y);
    return (a ? kFQ - a : -1) < (b ? kFQ - b : -1);
  });
  int64_t off = 0, foff = 0, roff = 0;
  std::vector<DInst> dev;
  for (int i : order) {
    DInst& I = h->inst[i];
    const int c = ctas(i);
    I.off = off;
    I.foff = foff;
    I.roff = roff;
    off += I.N;
    if (c == 0) {
      foff += tri_fac_size(I.N, kDT);
      roff += tri_red_size(I.N, kDT);
      h->n_big += 1;
      h->big_cells = off;
    } else if (h->fcnt[c]++ == 0) {
      h->foff[c] = (int)dev.size();
    }
    dev.push_back(I);
  }
  h->n_inst = n_inst;
  h->ncell = off;
  if (stream) {
    h->stream = (cudaStream_t)stream;
  } else {
    DCK(cudaStreamCreateWithFlags(&h->stream, cudaStreamNonBlocking));
    h->own_stream = true;
  }
  DDev& D = h->D;
  const int64_t nc = off, nb = h->big_cells;
  if (!(dalloc_d(h, &h->d_inst, n_inst) && dalloc_d(h, &D.sig, nc) && dalloc_d(h, &D.T, nc) &&
        dalloc_d(h, &D.U, nb) && dalloc_d(h, &D.f, nb) && dalloc_d(h, &D.k, nb) && dalloc_d(h, &D.Us, nc) &&
        dalloc_d(h, &D.x, nb) && dalloc_d(h, &D.F, foff) && dalloc_d(h, &D.Rd, roff) &&
        dalloc_d(h, &D.status, 1)))
    return dfail(h, GRTE_ENOMEM, "cudaMalloc failed");
  D.inst = h->d_inst;
  DCK(cudaMemcpyAsync(h->d_inst, dev.data(), sizeof(DInst) * n_inst, cudaMemcpyHostToDevice, h->stream));
  for (int i = 0; i < n_inst; ++i)
    DCK(cudaMemcpyAsync(D.sig + h->inst[i].off, in[i].sigma, sizeof(double) * in[i].nx, cudaMemcpyHostToDevice,
                        h->stream));
  DCK(cudaMallocHost(&h->h_status, sizeof(int)));
  if (nc <= kStageCells && cudaMallocHost(&h->h_state, sizeof(double) * nc) != cudaSuccess) {
    h->h_state = nullptr;
    cudaGetLastError();
  }
  h->stamp.assign(n_inst, -1);
  int classes = h->n_big > 0 ? 1 : 0;
  for (int c = 1; c <= kFQ; ++c) classes += h->fcnt[c] > 0;
  if (classes > 1) {
    DCK(cudaEventCreateWithFlags(&h->ev_fork, cudaEventDisableTiming));
    for (int i = 0; i < classes - 1; ++i) {
      DCK(cudaStreamCreateWithFlags(&h->side[i], cudaStreamNonBlocking));
      DCK(cudaEventCreateWithFlags(&h->ev_join[i], cudaEventDisableTiming));
    }
  }
  DCK(cudaMemsetAsync(D.status, 0, sizeof(int), h->stream));
  DCK(cudaMemsetAsync(D.T, 0, sizeof(double) * nc, h->stream));
  DCK(cudaStreamSynchronize(h->stream));
  return GRTE_OK;
}

grte_status grte_diff_set_T(grte_diff_t h, int inst, const double* T, size_t len) {
  if (!h) return GRTE_EINVAL;
  if (inst < 0 || inst >= h->n_inst || !T) return dfail(h, GRTE_EINVAL, "bad instance or NULL T");
  const DInst& I = h->inst[inst];
  if (len != (size_t)I.N) return dfail(h, GRTE_EINVAL, "len must equal nx");
  for (size_t j = 0; j < len; ++j)
    if (!(T[j] >= 0.0) || !std::isfinite(T[j])) return dfail(h, GRTE_EINVAL, "T must be finite and >= 0");
  // the caller may reuse T on return: it is copied to its slot, so that setting a batch does
  // not wait for each copy (64 uneven runs: 0.96 ms with a wait each)
  cudaStreamCaptureStatus cap = cudaStreamCaptureStatusNone;
  DCK(cudaStreamIsCapturing(h->stream, &cap));
  if (h->h_state && cap == cudaStreamCaptureStatusNone) {   // (a capture must not hold a slot)
    if (h->stamp[inst] == h->epoch) {
      DCK(cudaStreamSynchronize(h->stream));
      ++h->epoch;
    }
    std::copy(T, T + len, h->h_state + I.off);
    DCK(cudaMemcpyAsync(h->D.T + I.off, h->h_state + I.off, sizeof(double) * I.N, cudaMemcpyHostToDevice, h->stream));
    h->stamp[inst] = h->epoch;
    return GRTE_OK;
  }
  DCK(cudaMemcpyAsync(h->D.T + I.off, T, sizeof(double) * I.N, cudaMemcpyHostToDevice, h->stream));
  DCK(cudaStreamSynchronize(h->stream));
  return GRTE_OK;
}

// The launches of one block of steps.  Cluster sizes have no data in common: the first
// (largest) class runs on the handle's stream, the others on side streams between a fork
// and a join, so that a class of few instances does not hold the chip alone.
static grte_status diff_block(grte_diff_t h, int nsteps) {
  int cls = 0;
  if (h->ev_fork) DCK(cudaEventRecord(h->ev_fork, h->stream));
  if (h->n_big > 0) {
    const unsigned cb = 256, cg = (unsigned)((h->big_cells + cb - 1) / cb);
    const size_t smem = (size_t)tri_smem_bytes(kDT, true, 8);
    for (int n = 0; n < nsteps; ++n) {
      k_dcoef<<<cg, cb, 0, h->stream>>>(h->D, h->n_big, h->big_cells);
      k_dsolve<<<(unsigned)h->n_big, kDT, smem, h->stream>>>(h->D);
      k_dcorr<<<cg, cb, 0, h->stream>>>(h->D, h->n_big, h->big_cells, h->newton_maxit);
    }
    DCK(cudaGetLastError());
    ++cls;
  }
  for (int c = kFQ; c >= 1; --c) {
    if (!h->fcnt[c]) continue;
    cudaStream_t st = cls ? h->side[cls - 1] : h->stream;
    if (cls) DCK(cudaStreamWaitEvent(st, h->ev_fork, 0));
    cudaLaunchConfig_t cfg;
    cudaLaunchAttribute at[1];
    diff_config(cfg, at, c, h->fcnt[c], st);
    DCK(cudaLaunchKernelEx(&cfg, k_diff, h->D, h->foff[c], c, nsteps, h->newton_maxit));
    if (cls) DCK(cudaEventRecord(h->ev_join[cls - 1], st));
    ++cls;
  }
  for (int i = 0; i + 1 < cls; ++i) DCK(cudaStreamWaitEvent(h->stream, h->ev_join[i], 0));
  return GRTE_OK;
}

grte_status grte_diff_step(grte_diff_t h, int64_t nsteps) {
  if (!h) return GRTE_EINVAL;
  if (nsteps < 0) return dfail(h, GRTE_EINVAL, "nsteps < 0");
  for (int64_t n = 0; n < nsteps; n += kFSteps) {
    const grte_status s = diff_block(h, (int)std::min<int64_t>(kFSteps, nsteps - n));
    if (s != GRTE_OK) return s;
  }
  DCK(cudaGetLastError());
  return GRTE_OK;
}

static grte_status dstatus(grte_diff_t h) {
  DCK(cudaMemcpyAsync(h->h_status, h->D.status, sizeof(int), cudaMemcpyDeviceToHost, h->stream));
  DCK(cudaStreamSynchronize(h->stream));
  ++h->epoch;
  const int s = *h->h_status;
  for (int code : {GRTE_ENAN, GRTE_ENONCONV, GRTE_ENEGATIVE})
    if (s & (1 << code)) return dfail(h, (grte_status)code, "device reported status " + std::to_string(code));
  return GRTE_OK;
}

grte_status grte_diff_sync(grte_diff_t h) {
  if (!h) return GRTE_EINVAL;
  const grte_status s = dstatus(h);
  if (s != GRTE_OK && s != GRTE_ECUDA) DCK(cudaMemset(h->D.status, 0, sizeof(int)));
  return s;
}

static grte_status dget(grte_diff_t h, int inst, const double* src, double* out, size_t len) {
  if (!h) return GRTE_EINVAL;
  if (inst < 0 || inst >= h->n_inst || !out) return dfail(h, GRTE_EINVAL, "bad instance or NULL output");
  const DInst& I = h->inst[inst];
  if (len != (size_t)I.N) return dfail(h, GRTE_EINVAL, "len must equal nx");
  // the values and the status come back behind one synchronisation
  double* to = h->h_state ? h->h_state + I.off : out;
  DCK(cudaMemcpyAsync(to, src + I.off, sizeof(double) * I.N, cudaMemcpyDeviceToHost, h->stream));
  const grte_status s = dstatus(h);
  if (s != GRTE_ECUDA && to != out) std::copy(to, to + I.N, out);
  return s;
}

grte_status grte_diff_get_T(grte_diff_t h, int inst, double* T, size_t len) {
  return h ? dget(h, inst, h->D.T, T, len) : GRTE_EINVAL;
}
grte_status grte_diff_get_Ustar(grte_diff_t h, int inst, double* U, size_t len) {
  return h ? dget(h, inst, h->D.Us, U, len) : GRTE_EINVAL;
}

}  // extern "C"
