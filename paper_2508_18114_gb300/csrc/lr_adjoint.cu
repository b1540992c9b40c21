// Discrete adjoint of the RK4 integration of Eq. S5: gradient of the
// assignment errors (Sec. S3.A) with respect to the pulse parameters.
//
// Loss and cotangents. eps_a = erfc(SNR/2)/2 + tau gamma/2 with
// SNR = sqrt(2 eta kappa S), S = dt sum_n w_n |beta_e(n) - beta_g(n)|^2
// (trapezoid weights w_n). With d eps/d S = -exp(-SNR^2/4) eta kappa /
// (2 sqrt(pi) SNR), the readout signal beta(n) = tr(Z_n^dag r Z_n) of
// trajectory e receives the complex cotangent g(n) = dL/dRe + i dL/dIm =
// dL/d eps * d eps/d S * dt * w_n * 2 (beta_e - beta_g)(n), and g -> -g for g.
// For a real loss with dL = Re tr(Zbar^dag dZ), beta contributes
// Zbar += conj(g) r Z + g r^dag Z.
//
// RK4 (stage inputs U_0 = Z, U_1 = Z + h/2 K_1, U_2 = Z + h/2 K_2,
// U_3 = Z + h K_3, K_{s+1} = F(U_s)) reversed: with Zbar' = lambda,
//   Kbar_4 = h/6 lambda,               Ubar_3 = J(U_3)^dag Kbar_4
//   Kbar_3 = h/3 lambda + h   Ubar_3,  Ubar_2 = J(U_2)^dag Kbar_3
//   Kbar_2 = h/3 lambda + h/2 Ubar_2,  Ubar_1 = J(U_1)^dag Kbar_2
//   Kbar_1 = h/6 lambda + h/2 Ubar_1,  Ubar_0 = J(U_0)^dag Kbar_1
//   lambda_n = lambda + sum_s Ubar_s + (beta(n) cotangent).
//
// Vector-Jacobian product of F(U) = -i H_eff U + sum_k 1/2 a_k (l_k U) X_k'^dag,
// X_k' = G^-1 U^dag l_k U (L_k = sqrt(a_k) l_k, a = kappa, gamma), for a
// cotangent Fbar (derived from dF with dG = dU^dag U + U^dag dU):
//   E_k' = (l_k U)^dag Fbar G^-1,   P_k' = X_k' E_k' + (X_k' E_k')^dag,
//   Ubar = i H_eff^dag Fbar + sum_k a_k/2 [ l_k^dag (Fbar X_k' + U E_k'^dag)
//          + (l_k U) E_k' - U P_k' ].
// The pulse enters only through c(t) (r + r^dag): theta_bar_i +=
// Im tr(Fbar^dag (r + r^dag) U) dc/dtheta_i at the stage time.
//
// Forward stages run the plain engine's kernels. States are stored every `ckpt_every` steps; a segment is recomputed once,
// keeping every stage input U_s, G^-1 and X_k' of its steps where the caller's workspace
// has room for them, else step by step (the same kernels on the same inputs: the gradient
// does not depend on it), and the last segment is kept by the forward pass itself.
//
// Bound by the FP64 pipe (2 FMA/clk/SM; a warp instruction holds it for 16 cycles
// whatever the number of its active lanes), so what counts is the number of FP64
// instructions: square roots of the ladder operators come from a table, Fbar is
// formed once, the P_k' are added before they are applied (28 FMAs per entry and l in
// the VJP), partial sums are added across the chip and the pulse is evaluated once
// per segment. 12 trajectories of N = 2000, M = 20, 16 steps: see adj_vjp.
//
// Precision follows the context. FP64 context: everything in complex128 /
// FP64. FP32-bulk context: the states, stage inputs, cotangents and every
// per-element product (operator apply, projection terms, the VJP rows, the
// partial sums of (l_k U)^dag Fbar and T_k) in complex64 / FP32; the Gram
// matrix summed from exact products of the FP32 entries in double-word FP32;
// G^-1, X_k', E_k', P_k' (M x M) in FP64 (rounded once to FP32 for the
// per-element kernels); the readout signal, the trapezoid weights and the
// pulse-parameter gradient accumulated in FP64.
#include <algorithm>
#include <climits>
#include <cmath>
#include <string>
#include <utility>
#include <vector>

#include "lr_internal.cuh"

namespace lr {
namespace adj {

constexpr int AT = 256;
constexpr int AR = 16;   // rows per partial block (as the plain engine)
constexpr int MR2 = LR_MAX_RANK * LR_MAX_RANK;

struct Ptrs {
  const TrajDev* traj;
  const PulseDev* pulse;
  unsigned* err;
  double2* Xs;      // [4][n_traj][2][MR2]  X_k' of each stage of the step (row-major M x M)
  double2* Gi;      // [4][n_traj][MR2]     G^-1 of each stage
  double2* EP;      // [n_traj][4][MR2]     E_r', E_b', X_r' E_r', X_b' E_b'
  double* bpart;
  double* thbar;    // [n_traj][8]
  double2* beta;
  long bstride;     // beta entries per trajectory
  double* coef;     // [n_cand][3 K] c(t) at t_n, t_n + h/2, t_n + h of the segment's steps
  int cstride;
  const double* gcoef;   // [n_cand]
  int n_traj;
  double tau, dt;
};

__device__ __forceinline__ double2 cmul(double2 a, double2 b) { return mk(fma(a.x, b.x, -a.y * b.y), fma(a.x, b.y, a.y * b.x)); }
__device__ __forceinline__ double2 cmulc(double2 a, double2 b) { return mk(fma(a.x, b.x, a.y * b.y), fma(a.x, b.y, -a.y * b.x)); }  // conj(a) b
__device__ __forceinline__ double2 cadd(double2 a, double2 b) { return mk(a.x + b.x, a.y + b.y); }
// s + a b
template <typename T2>
__device__ __forceinline__ T2 cmac(T2 a, T2 b, T2 s) {
  return mkc<T2>(fma(a.x, b.x, fma(-a.y, b.y, s.x)), fma(a.x, b.y, fma(a.y, b.x, s.y)));
}
// s + a conj(b)
template <typename T2>
__device__ __forceinline__ T2 cmac_c(T2 a, T2 b, T2 s) {
  return mkc<T2>(fma(a.x, b.x, fma(a.y, b.y, s.x)), fma(a.y, b.x, fma(-a.x, b.y, s.y)));
}

// c(t) at the stage times of steps s0 .. s0 + len - 1, one thread each (the FP64 pulse
// shape takes ~12k cycles; once per segment here, not in every block of every stage).
__global__ void adj_drive(Ptrs a, int n_cand, long s0, int len) {
  const int i = blockIdx.x * blockDim.x + threadIdx.x;
  if (i >= 3 * len * n_cand) return;
  const int c = i / (3 * len), r = i - c * 3 * len, k = r % 3;
  const double t = (double)(s0 + r / 3) * a.dt + (k == 0 ? 0.0 : (k == 2 ? a.dt : 0.5 * a.dt));
  a.coef[(size_t)c * a.cstride + r] = pulse_coefficient(a.pulse[c], a.tau, t);
}

// Fbar = ca lam + cb Un (cb == 0: Un unused), kept in Fb, and partial sums of B_k' =
// (l_k U)^dag Fbar and w = tr(Fbar^dag (r + r^dag) U) per row block. B_k' in the bulk
// arithmetic, w in FP64.
template <typename T2>
__global__ void __launch_bounds__(AT) adj_bpart(Ptrs a, const T2* __restrict__ U, const T2* __restrict__ lam,
                                                const T2* __restrict__ Un, double ca_d, double cb_d,
                                                T2* __restrict__ Fb, const __grid_constant__ SqTab sq) {
  using T = typename real_of<T2>::type;
  const TrajDev d = a.traj[blockIdx.y];
  const int b = blockIdx.x;
  if (b >= d.nblk) return;
  __shared__ T2 sF[AR][LR_MAX_RANK], sR[AR][LR_MAX_RANK], sB[AR][LR_MAX_RANK];
  __shared__ double2 wpart[AT / 32];
  const int M = d.M, ld = d.ld, r0 = b * AR, rows = min(AR, d.N - r0);
  const size_t off = d.z_off;
  const int st = d.Nr * d.Nf;
  const T ca = (T)ca_d, cb = (T)cb_d;
  double2 wsum = mk(0.0, 0.0);
  for (int e = threadIdx.x; e < AR * M; e += AT) {
    const int i = e / M, m = e - (e / M) * M;
    T2 f = mkc<T2>(0, 0), zr = mkc<T2>(0, 0), zb = mkc<T2>(0, 0);
    if (i < rows) {
      const int n = r0 + i;
      const size_t o = off + (size_t)n * ld + m;
      const T2 l0 = lam[o];
      f = mkc<T2>(ca * l0.x, ca * l0.y);
      if (cb_d != 0.0) {
        const T2 u0 = Un[o];
        f = mkc<T2>(fma(cb, u0.x, f.x), fma(cb, u0.y, f.y));
      }
      Fb[o] = f;
      const RowIdx ri = row_index(d, n);
      const int iro = readout_index(d, ri), dro = readout_dim(d);
      T2 xd = mkc<T2>(0, 0);
      if (iro + 1 < dro) {
        const T c = (T)sq_of(sq, iro + 1);
        const T2 v = U[o + ld];
        zr = mkc<T2>(c * v.x, c * v.y);
        xd = zr;
      }
      if (iro >= 1) {
        const T c = (T)sq_of(sq, iro);
        const T2 v = U[o - ld];
        xd = mkc<T2>(fma(c, v.x, xd.x), fma(c, v.y, xd.y));
      }
      if (ri.it + 1 < d.Nt) {
        const T c = (T)sq_of(sq, ri.it + 1);
        const T2 v = U[o + (size_t)st * ld];
        zb = mkc<T2>(c * v.x, c * v.y);
      }
      // conj(f) xd, summed in FP64
      wsum = cadd(wsum, cmulc(mk((double)f.x, (double)f.y), mk((double)xd.x, (double)xd.y)));
    }
    sF[i][m] = f;
    sR[i][m] = zr;
    sB[i][m] = zb;
  }
  for (int o = 16; o > 0; o >>= 1)
    wsum = mk(wsum.x + __shfl_down_sync(0xffffffffu, wsum.x, o), wsum.y + __shfl_down_sync(0xffffffffu, wsum.y, o));
  if ((threadIdx.x & 31) == 0) wpart[threadIdx.x >> 5] = wsum;
  __syncthreads();
  double* out = a.bpart + d.p_off + (size_t)b * plain_pstride(M);
  const int MM = M * M;
  for (int e = threadIdx.x; e < 2 * MM; e += AT) {
    const int k = e / MM, ij = e - k * MM, i = ij / M, j = ij - (ij / M) * M;
    T re = 0, im = 0;
    for (int r = 0; r < rows; ++r) {
      const T2 x = k == 0 ? sR[r][i] : sB[r][i], y = sF[r][j];   // conj(x) y
      re = fma(x.x, y.x, fma(x.y, y.y, re));
      im = fma(x.x, y.y, fma(-x.y, y.x, im));
    }
    out[2 * e] = (double)re;
    out[2 * e + 1] = (double)im;
  }
  if (threadIdx.x == 0) {
    double2 w = mk(0.0, 0.0);
    for (int t = 0; t < AT / 32; ++t) w = cadd(w, wpart[t]);
    out[4 * MM] = w.x;
    out[4 * MM + 1] = w.y;
  }
}

// From the sums of B_k' and w in the trajectory's first row block: E_k' = B_k' G^-1
// and X_k' E_k', block (2 x + k) on columns BC x .. of jump k (one SM would take 62k
// cycles for the 16 M^3 FMAs at M = 20); in the last block theta_bar += Im(w)
// dc/dtheta at the stage time.
constexpr int BC = 4;
__global__ void __launch_bounds__(AT) adj_bsolve(Ptrs a, int stage, double t_stage) {
  const int tj = blockIdx.y, tid = threadIdx.x;
  const TrajDev d = a.traj[tj];
  const int M = d.M, MM = M * M;
  const double2* P = reinterpret_cast<const double2*>(a.bpart + d.p_off);
  if (blockIdx.x == gridDim.x - 1) {
    if (tid == 0) {
      const double im = P[2 * MM].y;
      double dc[8];
      pulse_coefficient_grad(a.pulse[d.cand], a.tau, t_stage, dc);
      for (int i = 0; i < 8; ++i) a.thbar[(size_t)tj * 8 + i] += im * dc[i];
    }
    return;
  }
  const int k = blockIdx.x & 1, j0 = (blockIdx.x >> 1) * BC, nc = min(BC, M - j0);
  if (nc <= 0) return;
  __shared__ double2 E[LR_MAX_RANK][BC];
  const double2* Gi = a.Gi + ((size_t)stage * a.n_traj + tj) * MR2;
  const double2* X = a.Xs + (((size_t)stage * a.n_traj + tj) * 2 + k) * MR2;
  double2* EP = a.EP + (size_t)tj * 4 * MR2;
  const int i = tid / BC, c = tid % BC;   // LR_MAX_RANK * BC <= AT threads, one entry each
  const bool in = i < M && c < nc;
  if (in) {
    double2 s = mk(0.0, 0.0);
    for (int l = 0; l < M; ++l) s = cmac(P[k * MM + i * M + l], Gi[l * M + j0 + c], s);
    E[i][c] = s;
    EP[k * MR2 + i * M + j0 + c] = s;
  }
  __syncthreads();
  if (in) {
    double2 s = mk(0.0, 0.0);
    for (int l = 0; l < M; ++l) s = cmac(X[i * M + l], E[l][c], s);
    EP[(2 + k) * MR2 + i * M + j0 + c] = s;
  }
}

// Ubar_s for the cotangent Fbar (Fb). Thread: one row, the columns m and m + 1, with
// the M x M factors in shared memory (rows of M | 1 entries: no bank conflicts along
// a column either): 28 FMAs per column and l on the FP64 pipe, 448 us a stage at its
// rate for 12 trajectories of N = 2000, M = 20; 522 us with the ~60 others (ncu).
constexpr int VT = 128;
template <typename T2>
__global__ void __launch_bounds__(VT) adj_vjp(Ptrs a, const T2* __restrict__ U, const T2* __restrict__ Fb, int stage,
                                              const double* __restrict__ coef, T2* __restrict__ Ub,
                                              const __grid_constant__ SqTab sq) {
  using T = typename real_of<T2>::type;
  constexpr bool f32 = sizeof(T) == 4;
  extern __shared__ __align__(16) unsigned char vjp_sm[];
  const int tj = blockIdx.y;
  const TrajDev d = a.traj[tj];
  const int M = d.M, ld = d.ld, np = (M + 1) / 2, ldx = M | 1;
  const long total = (long)d.N * np;
  if ((long)blockIdx.x * VT >= total) return;
  const size_t off = d.z_off;
  const int st = d.Nr * d.Nf, sr = d.Nf;
  const double ak[2] = {d.kappa, d.gamma};
  T2* sm = reinterpret_cast<T2*>(vjp_sm);   // X_r', X_b', E_r', E_b', sum_k a_k/2 P_k'
  {
    const double2* EP = a.EP + (size_t)tj * 4 * MR2;
    const double2* Xt = a.Xs + (((size_t)stage * a.n_traj + tj) * 2) * MR2;
    for (int e = threadIdx.x; e < M * M; e += VT) {
      const int i = e / M, j = e - i * M, o = i * ldx + j, et = j * M + i;
      double px = 0.0, py = 0.0;
#pragma unroll
      for (int k = 0; k < 2; ++k) {
        const double2 x = Xt[k * MR2 + e], v = EP[k * MR2 + e];
        sm[k * M * ldx + o] = mkc<T2>((T)x.x, (T)x.y);
        sm[(2 + k) * M * ldx + o] = mkc<T2>((T)v.x, (T)v.y);
        if (ak[k] == 0.0) continue;
        const double2 p = EP[(2 + k) * MR2 + e], q = EP[(2 + k) * MR2 + et];   // P = XE + (XE)^dag
        px = fma(0.5 * ak[k], p.x + q.x, px);
        py = fma(0.5 * ak[k], p.y - q.y, py);
      }
      sm[4 * M * ldx + o] = mkc<T2>((T)px, (T)py);
    }
  }
  __syncthreads();
  const long idx = (long)blockIdx.x * VT + threadIdx.x;
  if (idx >= total) return;
  const int n = (int)(idx / np), m = 2 * (int)(idx - (long)n * np);
  const bool two = m + 1 < M;
  const int mc[2] = {m, two ? m + 1 : m};
  const T cf = (T)coef[(size_t)d.cand * a.cstride];
  const RowIdx ri = row_index(d, n);
  const T2* f = Fb + off + (size_t)n * ld;
  const T2* u = U + off + (size_t)n * ld;
  double dre, dim_;
  heff_diag(d, ri, 0.0, dre, dim_);   // the adjoint runs in the lab frame
  // i H_eff^dag Fbar: diagonal i conj(h) = i dre + dim
  T2 acc[2];
#pragma unroll
  for (int q = 0; q < 2; ++q) {
    const T2 f0 = f[mc[q]];
    if constexpr (f32) {
      const T dh = (T)dre, dl = (T)(dre - (double)dh), di = (T)dim_;
      acc[q] = mkc<T2>(fma(-dh, f0.y, fma(-dl, f0.y, di * f0.x)), fma(dh, f0.x, fma(dl, f0.x, di * f0.y)));
    } else {
      acc[q] = mkc<T2>(fma(-dre, f0.y, dim_ * f0.x), fma(dre, f0.x, dim_ * f0.y));
    }
  }
  // + i (real off-diagonal H entries times Fbar)
  auto add_row = [&](int o, T w) {
    const T2* v = f + (long)o * ld;
#pragma unroll
    for (int q = 0; q < 2; ++q) {
      const T2 x = v[mc[q]];
      acc[q] = mkc<T2>(fma(-w, x.y, acc[q].x), fma(w, x.x, acc[q].y));
    }
  };
#pragma unroll
  for (int sa = -1; sa <= 1; sa += 2) {
    const int it2 = ri.it + sa;
    if (it2 < 0 || it2 >= d.Nt) continue;
    const double ct = sq_of(sq, max(ri.it, it2));
#pragma unroll
    for (int sb = -1; sb <= 1; sb += 2) {
      const int ir2 = ri.ir + sb;
      if (ir2 < 0 || ir2 >= d.Nr) continue;
      add_row(sa * st + sb * sr, (T)(d.g * ct * sq_of(sq, max(ri.ir, ir2))));
    }
  }
  if (d.n_modes == 3) {
#pragma unroll
    for (int sa = -1; sa <= 1; sa += 2) {
      const int ir2 = ri.ir + sa;
      if (ir2 < 0 || ir2 >= d.Nr) continue;
      const double cr = sq_of(sq, max(ri.ir, ir2));
#pragma unroll
      for (int sb = -1; sb <= 1; sb += 2) {
        const int if2 = ri.iff + sb;
        if (if2 < 0 || if2 >= d.Nf) continue;
        add_row(sa * sr + sb, (T)(d.J * cr * sq_of(sq, max(ri.iff, if2))));
      }
    }
  }
  const int iro = readout_index(d, ri), dro = readout_dim(d);
#pragma unroll
  for (int sa = -1; sa <= 1; sa += 2) {
    const int i2 = iro + sa;
    if (i2 < 0 || i2 >= dro) continue;
    add_row(sa, cf * (T)sq_of(sq, max(iro, i2)));
  }
  // projection terms, k = r (stride 1, readout index), k = b (stride st, transmon index)
  const T2 zero = mkc<T2>(0, 0);
#pragma unroll
  for (int k = 0; k < 2; ++k) {
    if (ak[k] == 0.0) continue;
    const int idx_k = k == 0 ? iro : ri.it;
    const int dim_k = k == 0 ? dro : d.Nt;
    const long s_k = (long)(k == 0 ? 1 : st) * ld;
    const T2* Xk = sm + k * M * ldx;
    const T2* Ek = sm + (2 + k) * M * ldx;
    if (idx_k >= 1) {          // l_k^dag (Fbar X_k' + U E_k'^dag) at row n - s_k
      const T2 *fm = f - s_k, *um = u - s_k;
      T2 s1[2] = {zero, zero};
      for (int l = 0; l < M; ++l) {
        const T2 x = fm[l], y = um[l];
#pragma unroll
        for (int q = 0; q < 2; ++q)
          s1[q] = cmac_c(y, Ek[mc[q] * ldx + l], cmac(x, Xk[l * ldx + mc[q]], s1[q]));
      }
      const T c = (T)(0.5 * ak[k] * sq_of(sq, idx_k));
#pragma unroll
      for (int q = 0; q < 2; ++q) acc[q] = mkc<T2>(fma(c, s1[q].x, acc[q].x), fma(c, s1[q].y, acc[q].y));
    }
    if (idx_k + 1 < dim_k) {   // (l_k U) E_k'
      const T2* up = u + s_k;
      T2 s2[2] = {zero, zero};
      for (int l = 0; l < M; ++l) {
        const T2 y = up[l];
#pragma unroll
        for (int q = 0; q < 2; ++q) s2[q] = cmac(y, Ek[l * ldx + mc[q]], s2[q]);
      }
      const T c = (T)(0.5 * ak[k] * sq_of(sq, idx_k + 1));
#pragma unroll
      for (int q = 0; q < 2; ++q) acc[q] = mkc<T2>(fma(c, s2[q].x, acc[q].x), fma(c, s2[q].y, acc[q].y));
    }
  }
  {                            // - U sum_k a_k/2 P_k'
    const T2* Pk = sm + 4 * M * ldx;
    T2 s3[2] = {zero, zero};
    for (int l = 0; l < M; ++l) {
      const T2 y = u[l];
#pragma unroll
      for (int q = 0; q < 2; ++q) s3[q] = cmac(y, Pk[l * ldx + mc[q]], s3[q]);
    }
#pragma unroll
    for (int q = 0; q < 2; ++q) acc[q] = mkc<T2>(acc[q].x - s3[q].x, acc[q].y - s3[q].y);
  }
  T2* out = Ub + off + (size_t)n * ld;
  out[m] = acc[0];
  if (two) out[m + 1] = acc[1];
}

// lam_new = lam + sum_s Ubar_s + conj(g) r Z + g r^dag Z (readout cotangent of step n).
template <typename T2>
__global__ void __launch_bounds__(AT) adj_update(Ptrs a, const T2* __restrict__ Z, const T2* __restrict__ lam,
                                                 const T2* __restrict__ U0, const T2* __restrict__ U1,
                                                 const T2* __restrict__ U2, const T2* __restrict__ U3,
                                                 T2* __restrict__ lam_new, long step, long S, int with_sum,
                                                 const __grid_constant__ SqTab sq) {
  using T = typename real_of<T2>::type;
  const int tj = blockIdx.y;
  const TrajDev d = a.traj[tj];
  const int M = d.M, ld = d.ld;
  const size_t off = d.z_off;
  const int c = d.cand;
  const double2 be = a.beta[(size_t)(2 * c + 1) * a.bstride + step];
  const double2 bg = a.beta[(size_t)(2 * c) * a.bstride + step];
  const double w = (step == 0 || step == S) ? 0.5 : 1.0;
  const double sg = (tj & 1) ? 1.0 : -1.0;
  const double gs = sg * a.gcoef[c] * w;
  const T gx = (T)(gs * (be.x - bg.x)), gy = (T)(gs * (be.y - bg.y));
  const long total = (long)d.N * M;
  for (long idx = (long)blockIdx.x * blockDim.x + threadIdx.x; idx < total; idx += (long)gridDim.x * blockDim.x) {
    const int n = (int)(idx / M), m = (int)(idx - (long)n * M);
    const size_t o = off + (size_t)n * ld + m;
    T vx = 0, vy = 0;
    if (with_sum) {
      const T2 l0 = lam[o], a0 = U0[o], a1 = U1[o], a2 = U2[o], a3 = U3[o];
      vx = l0.x + ((a0.x + a1.x) + (a2.x + a3.x));
      vy = l0.y + ((a0.y + a1.y) + (a2.y + a3.y));
    }
    const RowIdx ri = row_index(d, n);
    const int iro = readout_index(d, ri), dro = readout_dim(d);
    if (iro + 1 < dro) {   // conj(g) r Z
      const T cc = (T)sq_of(sq, iro + 1);
      const T2 z = Z[o + ld];
      const T zx = cc * z.x, zy = cc * z.y;
      vx += gx * zx + gy * zy;
      vy += gx * zy - gy * zx;
    }
    if (iro >= 1) {        // g r^dag Z
      const T cc = (T)sq_of(sq, iro);
      const T2 z = Z[o - ld];
      const T zx = cc * z.x, zy = cc * z.y;
      vx += gx * zx - gy * zy;
      vy += gx * zy + gy * zx;
    }
    lam_new[o] = mkc<T2>(vx, vy);
  }
}

// gcoef[c] = dL/deps_c * d eps/dS * dt * 2 from the recomputed readout signals.
__global__ void adj_gcoef(Ptrs a, const double* __restrict__ deps, double eta, long S, double* gcoef) {
  const int c = blockIdx.x;
  __shared__ double sh[AT];
  const double2* bg = a.beta + (size_t)(2 * c) * a.bstride;
  const double2* be = a.beta + (size_t)(2 * c + 1) * a.bstride;
  double acc = 0.0;
  for (long i = threadIdx.x; i <= S; i += AT) {
    const double dx = be[i].x - bg[i].x, dy = be[i].y - bg[i].y;
    acc += ((i == 0 || i == S) ? 0.5 : 1.0) * (dx * dx + dy * dy);
  }
  sh[threadIdx.x] = acc;
  __syncthreads();
  if (threadIdx.x == 0) {
    double s = 0.0;
    for (int t = 0; t < AT; ++t) s += sh[t];
    const TrajDev d = a.traj[2 * c];
    const double Sint = a.dt * s;
    const double snr = sqrt(2.0 * eta * d.kappa * Sint);
    double dEdS = 0.0;
    if (snr > 0.0) dEdS = -exp(-0.25 * snr * snr) * eta * d.kappa / (2.0 * sqrt(M_PI) * snr);
    gcoef[c] = deps[c] * dEdS * a.dt * 2.0;
  }
}

}  // namespace adj

// ------------------------------------------------------------------ driver

namespace {
// Stage inputs and factors of a whole segment are kept up to this size (3% of HBM), in
// a workspace that has the room; else every step of the reverse pass recomputes its own.
constexpr size_t KEEP_BYTES = (size_t)8 << 30;
}  // namespace

BwdLayout bwd_layout(long long tot, int n_traj, int n_cand, size_t part_doubles, long S, int K, int fp32, int keep) {
  BwdLayout L{};
  size_t o = 0;
  auto take = [&](size_t bytes) {
    const size_t at = o;
    o = (o + bytes + 255) / 256 * 256;
    return at;
  };
  const size_t T = (fp32 ? sizeof(float2) : sizeof(double2)) * (size_t)tot;
  const size_t fac = sizeof(double2) * 4 * 3 * adj::MR2 * (size_t)n_traj;   // X_k' and G^-1 of a step's stages
  L.K = std::min<long>(K, S);
  L.fp32 = fp32;
  L.n_seg = (S + L.K - 1) / L.K;
  L.slots = keep && (size_t)L.K <= KEEP_BYTES / (3 * T + fac) ? L.K : 1;
  L.ck = take(T * L.n_seg);
  L.seg = take(T * (L.K + 1));
  L.cur = take(T);
  L.acc = take(T);
  L.U = take(T * 3 * L.slots);
  L.Ub = take(T * 4);
  L.Fb = take(T);
  L.lam = take(T);
  L.lamn = take(T);
  L.part = take(sizeof(double) * part_doubles);
  L.Xs = take(fac / 3 * 2 * L.slots);
  L.Gi = take(fac / 3 * L.slots);
  L.EP = take(sizeof(double2) * 4 * adj::MR2 * n_traj);
  L.bpart = take(sizeof(double) * part_doubles);
  L.beta = take(sizeof(double2) * n_traj * (size_t)(S + 1));
  L.coef = take(sizeof(double) * n_cand * 3 * L.K);
  L.gcoef = take(sizeof(double) * n_cand);
  L.deps = take(sizeof(double) * n_cand);
  L.thbar = take(sizeof(double) * 8 * n_traj);
  L.total = o;
  return L;
}

namespace {

template <typename T2>
cudaError_t backward_t(const DevPtrs& main, const RunParams& rp0, char* ws, const BwdLayout& L, long long tot,
                       int max_nblk, int max_N, int max_M, long S, const void* z0, int z0_fp32, const double* deps_host,
                       double* dtheta_host, cudaStream_t s) {
  constexpr bool f32 = sizeof(T2) == sizeof(float2);
  const size_t T = sizeof(T2) * (size_t)tot;
  auto P2 = [&](size_t off) { return reinterpret_cast<double2*>(ws + off); };
  auto PS = [&](size_t off) { return reinterpret_cast<T2*>(ws + off); };
  cudaError_t e;
  // plain-engine pointers for the forward stages
  DevPtrs p{};
  p.traj = main.traj;
  p.pulse = main.pulse;
  p.err = main.err;
  p.acc = ws + L.acc;
  p.part = reinterpret_cast<double*>(ws + L.part);
  p.beta = P2(L.beta);
  RunParams rp = rp0;
  rp.max_steps = S;
  adj::Ptrs a{};
  a.traj = main.traj;
  a.pulse = main.pulse;
  a.err = main.err;
  a.EP = P2(L.EP);
  a.bpart = reinterpret_cast<double*>(ws + L.bpart);
  a.thbar = reinterpret_cast<double*>(ws + L.thbar);
  a.beta = P2(L.beta);
  a.bstride = S + 1;
  a.coef = reinterpret_cast<double*>(ws + L.coef);
  a.cstride = 3 * (int)L.K;
  a.gcoef = reinterpret_cast<double*>(ws + L.gcoef);
  a.n_traj = rp.n_traj;
  a.tau = rp.tau;
  a.dt = rp.dt;
  const double h = rp.dt;
  const size_t fx = (size_t)rp.n_traj * 4 * adj::MR2;   // G^-1 entries of a step; X_k' has twice as many
  const double cs[4] = {0.0, 0.5, 0.5, 1.0};
  const int cc[4] = {0, 1, 1, 2};   // column of the drive table by stage
  // M x M factors and stage inputs of slot i
  auto at_slot = [&](long i) {
    a.Xs = P2(L.Xs) + 2 * fx * i;
    a.Gi = P2(L.Gi) + fx * i;
  };
  auto Uat = [&](long i, T2* Z, int st) { return st == 0 ? Z : PS(L.U) + ((size_t)i * 3 + st - 1) * tot; };
  auto gram = [&](const T2* U) {
    plain_gram_launch(p, rp, max_nblk, U, s);
    plain_reduce_launch(p.traj, rp.n_traj, LR_MAX_RANK, p.part, 6, 0, s);
  };
  // forward stages of step n (i of its segment) from Z into slot sl; Z_{n+1} into Zout unless null
  auto forward = [&](long n, long i, long sl, T2* Z, T2* Zout) {
    at_slot(sl);
    DevPtrs q = p;
    q.Zn = Z;
    for (int st = 0; st < 4; ++st) {
      T2* u = Uat(sl, Z, st);
      gram(u);
      q.X = a.Xs + (size_t)st * rp.n_traj * 2 * adj::MR2;
      plain_solve_launch(q, rp, a.Gi + (size_t)st * rp.n_traj * adj::MR2, n, st, 0, 1, -1.0, s);
      T2* out = st < 3 ? Uat(sl, Z, st + 1) : Zout;
      if (!out) break;
      plain_rhs_launch(q, rp, max_N, u, out, st, a.coef + 3 * i + cc[st], a.cstride, s);
    }
  };
  auto drive = [&](long s0, long len) {
    const int nd = (int)(3 * len * rp.n_cand);
    adj::adj_drive<<<(nd + 63) / 64, 64, 0, s>>>(a, rp.n_cand, s0, (int)len);
  };
  T2* seg = PS(L.seg);
  T2* cur = PS(L.cur);
  const bool keep = L.slots > 1 || L.K == 1;
  // the states of a segment from seg[0]: seg[1 .. len]
  auto fill = [&](long s0, long len, bool end) {
    for (long i = 0; i < len; ++i)
      if (keep || i + 1 < len || end)
        forward(s0 + i, i, keep ? i : 0, seg + (size_t)i * tot, i + 1 < len || end ? seg + (size_t)(i + 1) * tot : nullptr);
  };

  // initial state into the first checkpoint (in the adjoint's state type)
  if (z0_fp32 == (int)f32)
    e = cudaMemcpyAsync(PS(L.ck), z0, T, cudaMemcpyDeviceToDevice, s);
  else
    e = launch_convert(z0, PS(L.ck), tot, f32 ? 1 : 0, s);
  if (e != cudaSuccess) return e;
  if ((e = cudaMemsetAsync(ws + L.thbar, 0, sizeof(double) * 8 * rp.n_traj, s)) != cudaSuccess) return e;
  if ((e = cudaMemcpyAsync(ws + L.deps, deps_host, sizeof(double) * rp.n_cand, cudaMemcpyHostToDevice, s)) !=
      cudaSuccess)
    return e;
  // forward pass: checkpoints and the readout signal; the last segment is filled
  for (long sg = 0; sg < L.n_seg; ++sg) {
    const long s0 = sg * L.K, len = std::min<long>(L.K, S - s0);
    const bool last = sg + 1 == L.n_seg;
    drive(s0, len);
    if ((e = cudaMemcpyAsync(last ? seg : cur, PS(L.ck) + (size_t)sg * tot, T, cudaMemcpyDeviceToDevice, s)) !=
        cudaSuccess)
      return e;
    if (last) {
      fill(s0, len, true);
    } else {
      for (long i = 0; i < len; ++i) forward(s0 + i, i, 0, cur, cur);
      if ((e = cudaMemcpyAsync(PS(L.ck) + (size_t)(sg + 1) * tot, cur, T, cudaMemcpyDeviceToDevice, s)) != cudaSuccess)
        return e;
    }
    if ((e = cudaGetLastError()) != cudaSuccess) return e;
  }
  const T2* zS = seg + (size_t)(S - (L.n_seg - 1) * L.K) * tot;
  gram(zS);
  plain_solve_launch(p, rp, nullptr, S, 0, 0, 0, -1.0, s);
  adj::adj_gcoef<<<rp.n_cand, adj::AT, 0, s>>>(a, reinterpret_cast<double*>(ws + L.deps), rp.eta, S,
                                                reinterpret_cast<double*>(ws + L.gcoef));
  const dim3 egrid((unsigned)std::min<long>(((long)max_N * LR_MAX_RANK + adj::AT - 1) / adj::AT, 4096), rp.n_traj);
  const dim3 vgrid((unsigned)(((long)max_N * (LR_MAX_RANK / 2) + adj::VT - 1) / adj::VT), rp.n_traj);
  const dim3 pgrid(max_nblk, rp.n_traj);
  const dim3 bgrid(2 * (LR_MAX_RANK / adj::BC) + 1, rp.n_traj);
  const int vsm = 5 * LR_MAX_RANK * (LR_MAX_RANK + 1) * (int)sizeof(T2);
  if ((e = cudaFuncSetAttribute(adj::adj_vjp<T2>, cudaFuncAttributeMaxDynamicSharedMemorySize, vsm)) != cudaSuccess)
    return e;
  const int vuse = 5 * max_M * (max_M | 1) * (int)sizeof(T2);
  T2* lam = PS(L.lam);
  T2* lamn = PS(L.lamn);
  T2* Fb = PS(L.Fb);
  // lambda_S: readout cotangent of the final state
  adj::adj_update<T2><<<egrid, adj::AT, 0, s>>>(a, zS, lam, lam, lam, lam, lam, lam, S, S, 0, sq_table());
  T2* Ub[4] = {PS(L.Ub), PS(L.Ub) + tot, PS(L.Ub) + 2 * tot, PS(L.Ub) + 3 * tot};
  const double ca[4] = {h / 6.0, h / 3.0, h / 3.0, h / 6.0};
  const double cb[4] = {h / 2.0, h / 2.0, h, 0.0};
  for (long sg = L.n_seg - 1; sg >= 0; --sg) {
    const long s0 = sg * L.K, len = std::min<long>(L.K, S - s0);
    if (sg + 1 < L.n_seg) {
      drive(s0, len);
      if ((e = cudaMemcpyAsync(seg, PS(L.ck) + (size_t)sg * tot, T, cudaMemcpyDeviceToDevice, s)) != cudaSuccess)
        return e;
      fill(s0, len, false);
    }
    for (long i = len - 1; i >= 0; --i) {
      const long n = s0 + i;
      const double tn = (double)n * h;
      T2* Z = seg + (size_t)i * tot;
      const long sl = keep ? i : 0;
      if (!keep) forward(n, i, 0, Z, nullptr);
      at_slot(sl);
      // reverse stages
      for (int st = 3; st >= 0; --st) {
        const T2* un = st < 3 ? Ub[st + 1] : Ub[0];
        const T2* u = Uat(sl, Z, st);
        adj::adj_bpart<T2><<<pgrid, adj::AT, 0, s>>>(a, u, lam, un, ca[st], st < 3 ? cb[st] : 0.0, Fb, sq_table());
        plain_reduce_launch(a.traj, rp.n_traj, LR_MAX_RANK, a.bpart, 4, 2, s);
        adj::adj_bsolve<<<bgrid, adj::AT, 0, s>>>(a, st, tn + cs[st] * h);
        adj::adj_vjp<T2><<<vgrid, adj::VT, vuse, s>>>(a, u, Fb, st, a.coef + 3 * i + cc[st], Ub[st], sq_table());
      }
      adj::adj_update<T2><<<egrid, adj::AT, 0, s>>>(a, Z, lam, Ub[0], Ub[1], Ub[2], Ub[3], lamn, n, S, 1, sq_table());
      std::swap(lam, lamn);
      if ((e = cudaGetLastError()) != cudaSuccess) return e;
    }
  }
  // theta_bar per candidate = g + e trajectories
  std::vector<double> th(8 * (size_t)rp.n_traj);
  if ((e = cudaMemcpyAsync(th.data(), ws + L.thbar, sizeof(double) * th.size(), cudaMemcpyDeviceToHost, s)) !=
      cudaSuccess)
    return e;
  if ((e = cudaStreamSynchronize(s)) != cudaSuccess) return e;
  for (int c = 0; c < rp.n_cand; ++c)
    for (int i = 0; i < 8; ++i) dtheta_host[8 * c + i] = th[8 * (2 * c) + i] + th[8 * (2 * c + 1) + i];
  return cudaSuccess;
}

}  // namespace

cudaError_t backward_run(const DevPtrs& main, const RunParams& rp, char* ws, const BwdLayout& L, long long tot,
                         int max_nblk, int max_N, int max_M, long S, const void* z0, int z0_fp32, const double* deps_host,
                         double* dtheta_host, cudaStream_t s) {
  if (L.fp32)
    return backward_t<float2>(main, rp, ws, L, tot, max_nblk, max_N, max_M, S, z0, z0_fp32, deps_host, dtheta_host, s);
  return backward_t<double2>(main, rp, ws, L, tot, max_nblk, max_N, max_M, S, z0, z0_fp32, deps_host, dtheta_host, s);
}

}  // namespace lr
