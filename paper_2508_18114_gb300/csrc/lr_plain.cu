// PLAIN engine: straightforward FP64 kernels with the state in HBM.
//
// One RK4 stage of Eq. S5 is four launches:
//   plain_gram  - per row block, partial sums of G = Z^dag Z (upper triangle),
//                 T_r = Z^dag r Z and T_b = Z^dag b Z, plus level populations
//                 and readout photons at recording steps;
//   plain_reduce - the partials added in a fixed order, a warp per 32 entries and share;
//   plain_solve - a few blocks per trajectory: record beta = tr(T_r) at stage 1 of
//                 each step, G^-1 by symmetric sweeps, X_r = G^-1 T_r, X_b = G^-1 T_b;
//   plain_rhs   - per element: F = -i H_eff Z + 1/2 kappa (rZ) X_r^dag
//                 + 1/2 gamma (bZ) X_b^dag, then the RK4 stage update.
// With Y_k = L_k Z the projection term of Eq. S5 is 1/2 sum_k Y_k (Z^+ Y_k)^dag
// = 1/2 kappa (rZ)(G^-1 Z^dag r Z)^dag + 1/2 gamma (bZ)(G^-1 Z^dag b Z)^dag,
// and -1/2 sum_k L_k^dag L_k Z is folded into the diagonal of H_eff.
//
// The state type is a template parameter: complex128 (the reference path), or
// complex64 for the FP32-bulk recomputation inside the adjoint and for the wide
// schedule of the fused engine (wide_integrate: the same kernels, the step counter on
// the device). With complex64 the Gram matrix is summed from the exact products of
// the FP32 entries in double-word FP32 (FP64-class), G^-1 and X_k are FP64 in the
// adjoint and double-word FP32 in the wide schedule (as in the fused kernel), and the
// operator apply, T_k, the projection term and the RK4 update run in FP32 (the
// diagonal energies and the step sizes split into hi + lo floats so that FP32 does
// not round the mode frequencies or dt; the couplings rounded once).
#include <algorithm>
#include <cmath>
#include <type_traits>

#include "lr_mm.cuh"

namespace lr {

const SqTab& sq_table() {
  static const SqTab t = [] {
    SqTab x;
    for (int k = 0; k < SQ_N; ++k) x.v[k] = std::sqrt((double)k);
    return x;
  }();
  return t;
}

// sqrt(k) = hi + lo (x, y), for the weights of a complex64 state.
struct SqTabF {
  float2 v[SQ_N];
};
static const SqTabF& sq_table_f() {
  static const SqTabF t = [] {
    SqTabF x;
    for (int k = 0; k < SQ_N; ++k) {
      const double v = std::sqrt((double)k);
      x.v[k].x = (float)v;
      x.v[k].y = (float)(v - (double)x.v[k].x);
    }
    return x;
  }();
  return t;
}

// A matrix element g sqrt(k) .. sqrt(l), rounded once to the state's type. FP32 state:
// the factors as hi + lo floats (exact products by FMA, ~2^-46 before the rounding),
// so that no coupling is off by several roundings in every step, without FP64.
template <typename T>
struct Weight;
template <>
struct Weight<double> {
  using Tab = SqTab;
  double v;
  __device__ __forceinline__ Weight(double g, float2) : v(g) {}
  __device__ __forceinline__ Weight times(const Tab& t, int k) const { return Weight(v * sq_of(t, k), float2()); }
  __device__ __forceinline__ double round() const { return v; }
};
template <>
struct Weight<float> {
  using Tab = SqTabF;
  float hi, lo;
  __device__ __forceinline__ Weight(double, float2 g) : hi(g.x), lo(g.y) {}
  __device__ __forceinline__ Weight times(const Tab& t, int k) const {
    Weight s(*this);
    float2 q;
    if (k < SQ_N) {
      q = t.v[k];
    } else {
      const double v = sqrt((double)k);
      q.x = (float)v;
      q.y = (float)(v - (double)q.x);
    }
    s.hi = hi * q.x;
    s.lo = fmaf(hi, q.x, -s.hi) + fmaf(hi, q.y, lo * q.x);
    return s;
  }
  __device__ __forceinline__ float round() const { return hi + lo; }
};
static const SqTab& weight_table(double) { return sq_table(); }
static const SqTabF& weight_table(float) { return sq_table_f(); }

constexpr int PR = 16;        // rows per Gram block
constexpr int PT = 256;       // threads per block

__host__ __device__ inline size_t pstride(int M) { return plain_pstride(M); }

int plain_rows_per_block() { return PR; }
size_t plain_partial_doubles(int M) { return pstride(M); }

// The RK4 step of a launch on the device: *dstep + k of a run of n steps (the wide
// schedule, which may be replayed from a graph); dstep null: the host's arguments.
struct StepRef {
  const long long* dstep = nullptr;
  long k = 0, n = 0;
  const long long* loop = nullptr;   // device loop: k counts from loop[0], and n is loop[2]
  __device__ __forceinline__ long at() const { return loop ? (long)loop[0] + k : k; }
  __device__ __forceinline__ bool fits(long max_steps) const {
    return *dstep >= 0 && *dstep + (loop ? (long)loop[2] : n) <= max_steps;
  }
};

template <typename T2>
__global__ void __launch_bounds__(PT) plain_gram(const TrajDev* __restrict__ traj, const T2* __restrict__ Zin,
                                                 double* __restrict__ part, int with_obs, StepRef sr, int pop_every,
                                                 const __grid_constant__ SqTab sq) {
  using T = typename real_of<T2>::type;
  const TrajDev d = traj[blockIdx.y];
  const int b = blockIdx.x;
  if (b >= d.nblk) return;
  __shared__ T2 sZ[PR][LR_MAX_RANK], sR[PR][LR_MAX_RANK], sB[PR][LR_MAX_RANK];
  __shared__ double sw[PR];
  __shared__ int slev[PR], sro[PR];
  const int M = d.M, ld = d.ld;
  const int r0 = b * PR;
  const int rows = min(PR, d.N - r0);
  const T2* Z = Zin + d.z_off;
  const int st = d.Nr * d.Nf;
  for (int e = threadIdx.x; e < PR * M; e += blockDim.x) {
    const int i = e / M, m = e - (e / M) * M;
    T2 z = mkc<T2>(0, 0), zr = mkc<T2>(0, 0), zb = mkc<T2>(0, 0);
    if (i < rows) {
      const int n = r0 + i;
      z = Z[(size_t)n * ld + m];
      const RowIdx ri = row_index(d, n);
      const int iro = readout_index(d, ri);
      if (iro + 1 < readout_dim(d)) {
        const T c = (T)sq_of(sq, iro + 1);
        const T2 v = Z[(size_t)(n + 1) * ld + m];
        zr = mkc<T2>(c * v.x, c * v.y);
      }
      if (ri.it + 1 < d.Nt) {
        const T c = (T)sq_of(sq, ri.it + 1);
        const T2 v = Z[(size_t)(n + st) * ld + m];
        zb = mkc<T2>(c * v.x, c * v.y);
      }
      if (m == 0) {
        slev[i] = ri.it;
        sro[i] = iro;
      }
    }
    sZ[i][m] = z;
    sR[i][m] = zr;
    sB[i][m] = zb;
  }
  __syncthreads();
  double* out = part + d.p_off + (size_t)b * pstride(M);
  const int MM = M * M, ne = M * (M + 1) / 2;
  // entries in a row without the lower triangle: an FP64 instruction takes a warp's
  // time however many of its lanes are in use
  for (int e0 = threadIdx.x; e0 < ne + 2 * MM; e0 += blockDim.x) {
    int mat = 0, i, j;
    if (e0 < ne) {
      tri_entry(e0, i, j);
    } else {
      const int e1 = e0 - ne;
      mat = 1 + e1 / MM;
      const int ij = e1 - (mat - 1) * MM;
      i = ij / M;
      j = ij - i * M;
    }
    const int e = mat * MM + i * M + j;
    if (sizeof(T) == 4 && mat == 0) {
      // FP32 state: exact FP32 products (FMA TwoProduct) in double-word sums
      // (Knuth TwoSum), ~2^-48 relative: the FP64-class Gram on the FP32 pipes
      float rh = 0.f, rl = 0.f, ih = 0.f, il = 0.f;
      auto acc2 = [](float& hi, float& lo, float a, float b) {
        const float p = a * b, e = fmaf(a, b, -p), t = hi + p, bp = t - hi;
        lo += ((hi - (t - bp)) + (p - bp)) + e;
        hi = t;
      };
      for (int r = 0; r < rows; ++r) {
        const T2 a = sZ[r][i], c = sZ[r][j];
        acc2(rh, rl, (float)a.x, (float)c.x);      // conj(a) * c
        acc2(rh, rl, (float)a.y, (float)c.y);
        acc2(ih, il, (float)a.x, (float)c.y);
        acc2(ih, il, -(float)a.y, (float)c.x);
      }
      out[2 * e] = (double)rh + (double)rl;
      out[2 * e + 1] = (double)ih + (double)il;
    } else if (sizeof(T) == 8 || mat == 0) {
      // FP64 sums
      double re = 0.0, im = 0.0;
      for (int r = 0; r < rows; ++r) {
        const T2 a = sZ[r][i];
        const T2 c = mat == 0 ? sZ[r][j] : (mat == 1 ? sR[r][j] : sB[r][j]);
        const double ax = a.x, ay = a.y, cx = c.x, cy = c.y;
        re = fma(ax, cx, fma(ay, cy, re));      // conj(a) * c
        im = fma(ax, cy, fma(-ay, cx, im));
      }
      out[2 * e] = re;
      out[2 * e + 1] = im;
    } else {
      T re = 0, im = 0;
      for (int r = 0; r < rows; ++r) {
        const T2 a = sZ[r][i];
        const T2 c = mat == 1 ? sR[r][j] : sB[r][j];
        re = fma(a.x, c.x, fma(a.y, c.y, re));
        im = fma(a.x, c.y, fma(-a.y, c.x, im));
      }
      out[2 * e] = (double)re;
      out[2 * e + 1] = (double)im;
    }
  }
  if (with_obs && sr.dstep) with_obs = (*sr.dstep + sr.at()) % pop_every == 0;
  if (with_obs) {
    for (int i = threadIdx.x; i < PR; i += blockDim.x) {
      double w = 0.0;
      if (i < rows)
        for (int m = 0; m < M; ++m) {
          const double x = sZ[i][m].x, y = sZ[i][m].y;
          w += x * x + y * y;
        }
      sw[i] = w;
    }
    __syncthreads();
    if (threadIdx.x < LR_MAX_NT + 1) {
      const int t = threadIdx.x;
      double acc = 0.0;
      for (int i = 0; i < rows; ++i) {
        if (t < LR_MAX_NT) acc += (slev[i] == t) ? sw[i] : 0.0;
        else acc += sro[i] * sw[i];
      }
      out[6 * MM + t] = acc;
    }
  }
}

// Entry o < a M^2 + b of every trajectory: the row blocks' partial sums into block
// 0's, warp w of a block adding blocks w, w + 8, ... of 32 entries, then the eight warps
// in order. Bound by the latency of the loads, eight of a thread in flight: ~2 us for
// the 125 blocks of N = 2000 (one thread per entry: ~5 us; in the one block per
// trajectory that solves, 3e5 FP64 adds at M = 20, ~75 us of one SM).
__global__ void __launch_bounds__(PT) plain_reduce(const TrajDev* __restrict__ traj, double* __restrict__ part, int a,
                                                   int b) {
  __shared__ double sh[PT / 32][32];
  const TrajDev d = traj[blockIdx.y];
  const int lane = threadIdx.x & 31, warp = threadIdx.x >> 5, o = blockIdx.x * 32 + lane, no = a * d.M * d.M + b;
  if ((int)blockIdx.x * 32 >= no) return;
  double* P = part + d.p_off + o;
  const size_t ps = pstride(d.M);
  double s = 0.0;
  if (o < no)
    for (int k0 = warp; k0 < d.nblk; k0 += 64) {
      double v[8];
#pragma unroll
      for (int u = 0; u < 8; ++u) v[u] = k0 + 8 * u < d.nblk ? P[(size_t)(k0 + 8 * u) * ps] : 0.0;
#pragma unroll
      for (int u = 0; u < 8; ++u) s += v[u];
    }
  sh[warp][lane] = s;
  __syncthreads();
  if (warp == 0 && o < no) {
    for (int w = 1; w < PT / 32; ++w) s += sh[w][lane];
    P[0] = s;
  }
}

void plain_reduce_launch(const TrajDev* traj, int n_traj, int max_M, double* part, int a, int b, cudaStream_t s) {
  plain_reduce<<<dim3((a * max_M * max_M + b + 31) / 32, n_traj), PT, 0, s>>>(traj, part, a, b);
}

// Two doubles of the reduced sums carry the drive coefficient from plain_solve to
// plain_rhs: the one after the populations, and the imaginary part of G_00.
__device__ __forceinline__ double* drive_slot(double* P, int M, int c) { return P + (c ? 1 : 6 * M * M + LR_MAX_NT + 1); }

// From the sums in the trajectory's first row block: G^-1 by symmetric sweeps and X_k
// = G^-1 T_k (G^-1 to Gi unless null); at stage 0 the readout signal and the records;
// the drive coefficient of the stage time t. Every block of a trajectory forms G^-1
// (latency, ~1000 cycles a sweep in FP64) and its share of X_k, whose 8 M^3 FMAs
// take one SM 31k cycles at M = 20: 28 us in FP64, 16 us in double-word FP32 (two
// trajectories, M = 20, cold caches). It replaces a Cholesky factorisation and two
// triangular sweeps over 2 M columns in one block, ~70 barriers of FP64 latency.
// A: WidePivot; in the wide schedule F64Arith, or DwArith for the FP32 state.
// StepRef: the step and the record are the device counter's.
template <typename A>
__global__ void __launch_bounds__(ST) plain_solve(DevPtrs p, RunParams rp, double2* __restrict__ Gi, long step, int stage,
                                                  int record, int do_solve, double t, StepRef sr) {
  if (sr.dstep) {
    if (!sr.fits(rp.max_steps)) {   // every launch of the schedule leaves
      if (blockIdx.x == 0 && blockIdx.y == 0 && threadIdx.x == 0) set_error(p.err, DEV_CAPACITY);
      return;
    }
    step = (long)*sr.dstep + sr.at();
    record = stage == 0 && step % rp.pop_every == 0;
    t = __dadd_rn(__dmul_rn((double)step, rp.dt), t);   // as the host forms it
  }
  const int tj = blockIdx.y, g = blockIdx.x;
  const TrajDev d = p.traj[tj];
  const int M = d.M, MM = M * M, tid = threadIdx.x, ldg = M | 1;
  __shared__ typename A::C Gs[LR_MAX_RANK * (LR_MAX_RANK + 1)];
  __shared__ short2 tri[LR_MAX_RANK * (LR_MAX_RANK + 1) / 2];
  __shared__ MmShared<A> mm;
  __shared__ XColumns<A> xc;
  double* Pd = p.part + d.p_off;
  const double2* P = reinterpret_cast<const double2*>(Pd);   // p_off and the block size are even
  if (g == 0 && stage == 0) {
    if (tid >= ST - 32) {   // tr T_r, one lane per diagonal entry
      const int i = tid - (ST - 32);
      double2 b = i < M ? P[MM + i * M + i] : mk(0.0, 0.0);
      for (int o = 16; o > 0; o >>= 1)
        b = mk(b.x + __shfl_xor_sync(0xffffffffu, b.x, o), b.y + __shfl_xor_sync(0xffffffffu, b.y, o));
      if (i == 0) {
        p.beta[(size_t)tj * (rp.max_steps + 1) + step] = b;
        if (!isfinite(b.x) || !isfinite(b.y)) set_error(p.err, DEV_NONFINITE);
      }
    }
    if (record) {
      const long rec = step / rp.pop_every;
      if (tid < LR_MAX_NT + 1) {
        const double v = Pd[6 * MM + tid];
        if (tid < rp.nt_max) p.pops[((size_t)tj * rp.n_rec + rec) * rp.nt_max + tid] = tid < d.Nt ? v : 0.0;
        if (tid == LR_MAX_NT) p.nphot[(size_t)tj * rp.n_rec + rec] = v;
      }
      if (tid == 32) {
        double tr = 0.0;
        for (int i = 0; i < M; ++i) tr += P[i * M + i].x;
        p.trace[(size_t)tj * rp.n_rec + rec] = tr;
      }
      if (p.gsnap) {
        double2* gs = p.gsnap + ((size_t)tj * rp.n_rec + rec) * rp.snap_m * rp.snap_m;
        for (int e = tid; e < MM; e += ST) {
          const int i = e / M, j = e - i * M;
          const double2 v = P[min(i, j) * M + max(i, j)];
          gs[i * rp.snap_m + j] = mk(v.x, i == j ? 0.0 : (i < j ? v.y : -v.y));
        }
      }
    }
  }
  if (!do_solve) return;
  // the drive coefficient: ~12k cycles of FP64 latency, beside the sweeps of the warps
  // that hold entries where one is left (M < 32)
  const int nw = mm_warps(M, ST / 32);
  auto drive = [&]() {
    if (g != (gridDim.x > 1 ? 1 : 0) || tid != ST - 1 || t < 0.0) return;
    const PulseDev pulse = p.pulse[d.cand];
    if (rp.frame) {
      const double2 w = pulse_rwa_drive(pulse, rp.tau, t);
      *drive_slot(Pd, M, 0) = w.x;
      *drive_slot(Pd, M, 1) = w.y;
    } else {
      *drive_slot(Pd, M, 0) = pulse_coefficient(pulse, rp.tau, t);
    }
  };
  const int per = (2 * M + gridDim.x - 1) / gridDim.x, c_lo = g * per, c_hi = min(2 * M, c_lo + per);
  xc.load(P + MM, M, c_lo, min(XC, c_hi - c_lo), tid);
  if (tid == 0) mm.bad = 0;
  if (tid < M * (M + 1) / 2) {
    int i, j;
    tri_entry(tid, i, j);
    tri[tid] = make_short2((short)j, (short)i);
  }
  __syncthreads();
  if (tid / 32 < nw) {
    typename A::C e[2] = {A::zero(), A::zero()};   // the sums hold the upper triangle
    if (tid < M * (M + 1) / 2) {
      const int i = tri[tid].x, j = tri[tid].y;
      const double2 v = P[j * M + i];
      to_entry(mk(v.x, i == j ? 0.0 : -v.y), e[0]);
    }
    mm_invert<A, ST>(e, Gs, ldg, mm, tri, M, tid);
    if (nw == ST / 32) drive();
  } else {
    drive();
  }
  __syncthreads();
  if (g == 0) {
    if (tid == 0 && mm.bad) set_error(p.err, DEV_NOT_PD);
    if (Gi)
      for (int e = tid; e < MM; e += ST)
        Gi[(size_t)tj * LR_MAX_RANK * LR_MAX_RANK + e] = A::value(Gs[(e / M) * ldg + e % M]);
  }
  double2* X = p.X + (size_t)tj * 2 * LR_MAX_RANK * LR_MAX_RANK;
  x_columns<A>(xc, Gs, ldg, P + MM, M, c_lo, c_hi, tid, [&](int k, int i, int j, double2 v) {
    X[k * LR_MAX_RANK * LR_MAX_RANK + i * M + j] = v;
  });
}

// a trajectory's share of two blocks per SM, at most eight
static int solve_blocks(const RunParams& rp, int do_solve) {
  return do_solve ? std::max(1, std::min(8, 2 * SMS / rp.n_traj)) : 1;
}
void plain_solve_launch(const DevPtrs& p, const RunParams& rp, double2* Gi, long step, int stage, int record, int do_solve,
                        double t, cudaStream_t s) {
  plain_solve<WidePivot><<<dim3(solve_blocks(rp, do_solve), rp.n_traj), ST, 0, s>>>(p, rp, Gi, step, stage, record,
                                                                                    do_solve, t, StepRef{});
}

// Thread: one row, the columns m and m + 1. Bound by the FP64 pipe for the
// complex128 state: 8 FMAs per column and l of the two projections, ~45 others; 182 us
// for 12 trajectories of N = 2000, M = 20 (160 us at the pipe's rate). For a few
// complex64 trajectories bound by the latency of its loads (16 us for two): the ten
// neighbours' and eight l's are in flight together.
constexpr int RT = 128;   // threads per block

template <typename T2>
__global__ void __launch_bounds__(RT) plain_rhs(DevPtrs p, RunParams rp, const T2* __restrict__ Zin,
                                                T2* __restrict__ Zout, int stage,
                                                const double* __restrict__ ctab, int cstride, StepRef ref,
                                                const __grid_constant__
                                                typename Weight<typename real_of<T2>::type>::Tab sq) {
  if (ref.dstep && !ref.fits(rp.max_steps)) return;
  using T = typename real_of<T2>::type;
  constexpr bool f32 = sizeof(T) == 4;
  const int tj = blockIdx.y;
  const TrajDev d = p.traj[tj];
  const int M = d.M, MM = M * M, ld = d.ld, np = (M + 1) / 2;
  const long total = (long)d.N * np;
  if ((long)blockIdx.x * RT >= total) return;
  __shared__ T2 sX[2][LR_MAX_RANK * LR_MAX_RANK];
  __shared__ double coef, coef_i, wfr;
  const double2* X = p.X + (size_t)tj * 2 * LR_MAX_RANK * LR_MAX_RANK;
  // transposed in shared memory, sX[k][l * M + m] = X_k[m][l]: the threads of a
  // warp (consecutive m) then read consecutive words (no bank conflicts)
  for (int e = threadIdx.x; e < 2 * MM; e += RT) {
    const int k = e / MM, ij = e - k * MM, i = ij / M, j = ij - i * M;
    const double2 x = X[k * LR_MAX_RANK * LR_MAX_RANK + ij];
    sX[k][j * M + i] = mkc<T2>((T)x.x, (T)x.y);
  }
  if (threadIdx.x == 0) {
    double* P = p.part + d.p_off;
    coef = ctab ? ctab[(size_t)d.cand * cstride] : *drive_slot(P, M, 0);
    coef_i = rp.frame ? *drive_slot(P, M, 1) : 0.0;
    wfr = rp.frame ? pulse_drive_frequency(p.pulse[d.cand]) : 0.0;
  }
  __syncthreads();
  const long idx = (long)blockIdx.x * RT + threadIdx.x;
  if (idx >= total) return;
  const T2* Z = Zin + d.z_off;
  T2* Zn = reinterpret_cast<T2*>(p.Zn) + d.z_off;
  T2* acc = reinterpret_cast<T2*>(p.acc) + d.z_off;
  T2* Zo = Zout ? Zout + d.z_off : Zn;
  const int st = d.Nr * d.Nf, sr = d.Nf;
  const T c = (T)coef, ci = (T)coef_i;
  const double dt = rp.dt;
  // step sizes as hi + lo (FP32 state; lo = 0 in FP64)
  const double hsd = stage == 2 ? dt : 0.5 * dt, h6d = dt / 6.0;
  const T hs_hi = (T)hsd, hs_lo = (T)(hsd - (double)hs_hi), h6_hi = (T)h6d, h6_lo = (T)(h6d - (double)h6_hi);
  const bool rwa = rp.frame != 0;
  const int n = (int)(idx / np), m = 2 * (int)(idx - (long)n * np);
  const bool two = m + 1 < M;
  const int m1 = two ? m + 1 : m;
  const RowIdx ri = row_index(d, n);
  double dre, dim_;
  heff_diag(d, ri, wfr, dre, dim_);
  const T2* zrow = Z + (size_t)n * ld;
  T hr[2], hi[2];
  {
    // diagonal energy as hi + lo floats: FP32 does not round the mode frequencies
    const T dh = (T)dre, dl = (T)(dre - (double)dh), di = (T)dim_;
    const T2 z[2] = {zrow[m], zrow[m1]};
#pragma unroll
    for (int u = 0; u < 2; ++u) {
      if constexpr (f32) {
        hr[u] = fma(dh, z[u].x, fma(dl, z[u].x, -di * z[u].y));
        hi[u] = fma(dh, z[u].y, fma(dl, z[u].y, di * z[u].x));
      } else {
        hr[u] = fma(dh, z[u].x, -di * z[u].y);
        hi[u] = fma(dh, z[u].y, di * z[u].x);
      }
    }
  }
  // The neighbours' offsets and weights first (an absent one is the row itself with
  // weight zero), so that their loads are in flight together: complex weights on the
  // readout mode in the rotating frame only.
  int off[10];
  T w[10];
  T wi = 0;
  int na = 0;
  auto add = [&](bool on, int o, T wt) {
    off[na] = on ? o : 0;
    w[na++] = on ? wt : (T)0;
  };
  using W = Weight<T>;
  // g (b + b^dag)(a + a^dag); RWA keeps g (b^dag a + b a^dag) only
#pragma unroll
  for (int a = -1; a <= 1; a += 2) {
    const int it2 = ri.it + a;
    const bool ot = it2 >= 0 && it2 < d.Nt;
    const W ct = W(d.g, d.rate32[0]).times(sq, max(ri.it, it2));
#pragma unroll
    for (int bb = -1; bb <= 1; bb += 2) {
      const int ir2 = ri.ir + bb;
      add(ot && ir2 >= 0 && ir2 < d.Nr && !(rwa && a == bb), a * st + bb * sr, ct.times(sq, max(ri.ir, ir2)).round());
    }
  }
  // J (a + a^dag)(f + f^dag); RWA keeps J (a^dag f + a f^dag) only
#pragma unroll
  for (int a = -1; a <= 1; a += 2) {
    const int ir2 = ri.ir + a;
    const bool or2 = d.n_modes == 3 && ir2 >= 0 && ir2 < d.Nr;
    const W cr = W(d.J, d.rate32[1]).times(sq, max(ri.ir, ir2));
#pragma unroll
    for (int bb = -1; bb <= 1; bb += 2) {
      const int if2 = ri.iff + bb;
      add(or2 && if2 >= 0 && if2 < d.Nf && !(rwa && a == bb), a * sr + bb, cr.times(sq, max(ri.iff, if2)).round());
    }
  }
  // drive on the readout mode (stride 1): lab frame c(t) (r + r^dag); RWA
  // w r + conj(w) r^dag with w = c + i ci (row n gets r from n+1, r^dag from n-1)
  const int iro = readout_index(d, ri), dro = readout_dim(d);
  T sd[2];
#pragma unroll
  for (int a = -1; a <= 1; a += 2) {
    const int i2 = iro + a;
    const bool on = i2 >= 0 && i2 < dro;
    const T s = on ? W(1.0, make_float2(1.f, 0.f)).times(sq, max(iro, i2)).round() : (T)0;
    sd[a > 0] = s;
    add(on, a, c * s);
  }
#pragma unroll
  for (int q = 0; q < 10; ++q) {
    const T2* v = zrow + (long)off[q] * ld;
    const T2 v0 = v[m], v1 = v[m1];
    hr[0] = fma(w[q], v0.x, hr[0]);
    hi[0] = fma(w[q], v0.y, hi[0]);
    hr[1] = fma(w[q], v1.x, hr[1]);
    hi[1] = fma(w[q], v1.y, hi[1]);
    if (q >= 8 && rwa) {
      wi = (q == 9 ? ci : -ci) * sd[q - 8];
      hr[0] = fma(-wi, v0.y, hr[0]);
      hi[0] = fma(wi, v0.x, hi[0]);
      hr[1] = fma(-wi, v1.y, hr[1]);
      hi[1] = fma(wi, v1.x, hi[1]);
    }
  }
  // F = -i H_eff Z
  T fr[2] = {hi[0], hi[1]}, fi[2] = {-hr[0], -hr[1]};
  // + 1/2 kappa (rZ) X_r^dag + 1/2 gamma (bZ) X_b^dag
  auto project = [&](const T2* y, const T2* x, T s) {
    T pr[2] = {0, 0}, pi[2] = {0, 0};
#pragma unroll 8
    for (int l = 0; l < M; ++l) {
      const T2 v = y[l], x0 = x[l * M + m], x1 = x[l * M + m1];   // v conj(x)
      pr[0] = fma(v.x, x0.x, fma(v.y, x0.y, pr[0]));
      pi[0] = fma(v.y, x0.x, fma(-v.x, x0.y, pi[0]));
      pr[1] = fma(v.x, x1.x, fma(v.y, x1.y, pr[1]));
      pi[1] = fma(v.y, x1.x, fma(-v.x, x1.y, pi[1]));
    }
#pragma unroll
    for (int u = 0; u < 2; ++u) {
      fr[u] = fma(s, pr[u], fr[u]);
      fi[u] = fma(s, pi[u], fi[u]);
    }
  };
  if (iro + 1 < dro) project(zrow + ld, sX[0], W(0.5 * d.kappa, d.rate32[2]).times(sq, iro + 1).round());
  if (ri.it + 1 < d.Nt) project(zrow + (size_t)st * ld, sX[1], W(0.5 * d.gamma, d.rate32[3]).times(sq, ri.it + 1).round());
  // RK4 (weights 1/6, 1/3, 1/3, 1/6)
#pragma unroll
  for (int u = 0; u < 2; ++u) {
    if (u == 1 && !two) break;
    const size_t o = (size_t)n * ld + m + u;
    const T2 zn = Zn[o];
    T sx = fr[u], sy = fi[u];
    if (stage > 0) {
      const T2 a = acc[o];
      const T w = stage < 3 ? (T)2 : (T)1;
      sx = fma(w, sx, a.x);
      sy = fma(w, sy, a.y);
    }
    if (stage < 3) {
      acc[o] = mkc<T2>(sx, sy);
      Zo[o] = f32 ? mkc<T2>(zn.x + fma(hs_lo, fr[u], hs_hi * fr[u]), zn.y + fma(hs_lo, fi[u], hs_hi * fi[u]))
                  : mkc<T2>(fma(hs_hi, fr[u], zn.x), fma(hs_hi, fi[u], zn.y));
    } else {
      Zo[o] = f32 ? mkc<T2>(zn.x + fma(h6_lo, sx, h6_hi * sx), zn.y + fma(h6_lo, sy, h6_hi * sy))
                  : mkc<T2>(fma(h6_hi, sx, zn.x), fma(h6_hi, sy, zn.y));
    }
  }
}

void plain_gram_launch(const DevPtrs& p, const RunParams& rp, int max_nblk, const double2* zin, cudaStream_t s) {
  plain_gram<double2><<<dim3(max_nblk, rp.n_traj), PT, 0, s>>>(p.traj, zin, p.part, 0, StepRef{}, 1, sq_table());
}
void plain_gram_launch(const DevPtrs& p, const RunParams& rp, int max_nblk, const float2* zin, cudaStream_t s) {
  plain_gram<float2><<<dim3(max_nblk, rp.n_traj), PT, 0, s>>>(p.traj, zin, p.part, 0, StepRef{}, 1, sq_table());
}

template <typename T2>
void rhs_launch(const DevPtrs& p, const RunParams& rp, int max_N, const T2* zin, T2* zout, int stage,
                const double* coef, int cstride, StepRef ref, cudaStream_t s) {
  const int blocks = (int)(((long)max_N * (LR_MAX_RANK / 2) + RT - 1) / RT);   // those past a trajectory's rank leave at once
  plain_rhs<T2><<<dim3(blocks, rp.n_traj), RT, 0, s>>>(p, rp, zin, zout, stage, coef, cstride, ref,
                                                         weight_table(typename real_of<T2>::type()));
}
void plain_rhs_launch(const DevPtrs& p, const RunParams& rp, int max_N, const double2* zin, double2* zout, int stage,
                      const double* coef, int cstride, cudaStream_t s) {
  rhs_launch(p, rp, max_N, zin, zout, stage, coef, cstride, StepRef{}, s);
}
void plain_rhs_launch(const DevPtrs& p, const RunParams& rp, int max_N, const float2* zin, float2* zout, int stage,
                      const double* coef, int cstride, cudaStream_t s) {
  rhs_launch(p, rp, max_N, zin, zout, stage, coef, cstride, StepRef{}, s);
}

cudaError_t plain_integrate(const DevPtrs& p, const RunParams& rp, int max_nblk, int max_N, long step0, long n_steps,
                            cudaStream_t s) {
  using T2 = double2;
  T2* Zn = reinterpret_cast<T2*>(p.Zn);
  T2* Za = reinterpret_cast<T2*>(p.Za);
  T2* Zb = reinterpret_cast<T2*>(p.Zb);
  const dim3 ggrid(max_nblk, rp.n_traj);
  for (long st = step0; st < step0 + n_steps; ++st) {
    const double tn = (double)st * rp.dt;
    const int record = (st % rp.pop_every) == 0;
    for (int stage = 0; stage < 4; ++stage) {
      const T2* zin = stage == 0 ? Zn : (stage == 2 ? Zb : Za);
      T2* zout = stage == 1 ? Zb : (stage == 3 ? nullptr : Za);
      const double ts = tn + (stage == 0 ? 0.0 : (stage == 3 ? rp.dt : 0.5 * rp.dt));
      plain_gram<T2><<<ggrid, PT, 0, s>>>(p.traj, zin, p.part, stage == 0 && record, StepRef{}, 1, sq_table());
      plain_reduce_launch(p.traj, rp.n_traj, LR_MAX_RANK, p.part, 6, stage == 0 && record ? LR_MAX_NT + 1 : 0, s);
      plain_solve_launch(p, rp, nullptr, st, stage, stage == 0 && record, 1, ts, s);
      rhs_launch(p, rp, max_N, zin, zout, stage, nullptr, 0, StepRef{}, s);
    }
    cudaError_t e = cudaGetLastError();
    if (e != cudaSuccess) return e;
  }
  // observables of the final state
  const long se = step0 + n_steps;
  const int record = (se % rp.pop_every) == 0;
  plain_gram<T2><<<ggrid, PT, 0, s>>>(p.traj, Zn, p.part, record, StepRef{}, 1, sq_table());
  plain_reduce_launch(p.traj, rp.n_traj, LR_MAX_RANK, p.part, 6, record ? LR_MAX_NT + 1 : 0, s);
  plain_solve_launch(p, rp, nullptr, se, 0, record, 0, 0.0, s);
  return cudaGetLastError();
}

constexpr long LOOP_STEPS = 4;   // steps in the body of a device loop

// The wide schedule of the fused engine: the step counter on the device, for the
// complex64 state the double-word Gram and M x M phase. The buffers of p are the caller's.
template <typename T2>
static cudaError_t wide_t(const DevPtrs& p, const RunParams& rp, int max_nblk, int max_N, long n_steps, LoopRef loop,
                          cudaStream_t s) {
  // the team kernel's arithmetic and limits of a pivot: one context refuses the same
  // states whichever schedule it runs
  using A = typename std::conditional<sizeof(T2) == sizeof(float2), DwArith, F64Arith>::type;
  T2* Z[4] = {reinterpret_cast<T2*>(p.Zn), reinterpret_cast<T2*>(p.Za), reinterpret_cast<T2*>(p.Zb),
              reinterpret_cast<T2*>(p.Za)};
  const dim3 ggrid(max_nblk, rp.n_traj);
  const double c[4] = {0.0, 0.5 * rp.dt, 0.5 * rp.dt, rp.dt};
  // step k, or step lp[0] + k of a device loop; the last one records only
  auto step = [&](long k, const long long* lp, bool last, cudaStream_t st) {
    const StepRef ref{p.dstep, k, n_steps, lp};
    for (int stage = 0; stage < (last ? 1 : 4); ++stage) {
      plain_gram<T2><<<ggrid, PT, 0, st>>>(p.traj, Z[stage], p.part, stage == 0, ref, rp.pop_every, sq_table());
      plain_reduce_launch(p.traj, rp.n_traj, LR_MAX_RANK, p.part, 6, stage == 0 ? LR_MAX_NT + 1 : 0, st);
      plain_solve<A><<<dim3(solve_blocks(rp, !last), rp.n_traj), ST, 0, st>>>(p, rp, nullptr, 0, stage, 0, !last, c[stage],
                                                                              ref);
      if (!last) rhs_launch(p, rp, max_N, Z[stage], stage < 3 ? Z[stage + 1] : nullptr, stage, nullptr, 0, ref, st);
    }
    return cudaGetLastError();
  };
  long k = 0;
  if (loop.c && 16 * n_steps >= LOOP_LAUNCHES) {
    const long n = n_steps - n_steps % LOOP_STEPS;
    const cudaError_t e = device_loop(loop, rp.dt, rp.tau, LoopCount{0, n, n_steps}, LOOP_STEPS, [&](cudaStream_t st) {
      for (long i = 0; i < LOOP_STEPS; ++i) {
        const cudaError_t ei = step(i, loop.c, false, st);
        if (ei != cudaSuccess) return ei;
      }
      return cudaSuccess;
    }, s);
    if (e == cudaSuccess)
      k = n;
    else
      cudaGetLastError();   // no memory for the graph, say: the same launches from the host
  }
  for (; k <= n_steps; ++k) {
    const cudaError_t e = step(k, nullptr, k == n_steps, s);
    if (e != cudaSuccess) return e;
  }
  return cudaSuccess;
}
cudaError_t wide_integrate(const DevPtrs& p, const RunParams& rp, int max_nblk, int max_N, long n_steps, int fp32,
                           LoopRef loop, cudaStream_t s) {
  return fp32 ? wide_t<float2>(p, rp, max_nblk, max_N, n_steps, loop, s)
              : wide_t<double2>(p, rp, max_nblk, max_N, n_steps, loop, s);
}

}  // namespace lr
