// Kernels shared by the engines: fixed-rank initial state (Sec. S1.A),
// assignment-error epilogue (Sec. S3.A) and state precision conversion.
#include <cooperative_groups.h>

#include <algorithm>

#include "lr_internal.cuh"

namespace lr {

constexpr int IT = 512;   // threads of the initial-state kernel
constexpr int ET = 256;   // threads of the epilogue kernel
constexpr unsigned long long GOLDEN = 0x9E3779B97F4A7C15ull;

// SplitMix64 (Steele, Lea & Flood 2014): k-th output for a seed.
__device__ __forceinline__ unsigned long long mix64(unsigned long long z) {
  z = (z ^ (z >> 30)) * 0xBF58476D1CE4E5B9ull;
  z = (z ^ (z >> 27)) * 0x94D049BB133111EBull;
  return z ^ (z >> 31);
}
__device__ __forceinline__ unsigned long long splitmix64(unsigned long long seed, unsigned long long k) {
  return mix64(seed + (k + 1ull) * GOLDEN);
}
__device__ __forceinline__ double uniform_open0(unsigned long long seed, unsigned long long k) {
  return ((double)(splitmix64(seed, k) >> 11) + 1.0) * 0x1.0p-53;
}

// Fixed-order block reduction (deterministic for a fixed block size).
template <int NT>
__device__ double block_sum(double v, double* sh) {
  for (int o = 16; o > 0; o >>= 1) v += __shfl_down_sync(0xffffffffu, v, o);
  if ((threadIdx.x & 31) == 0) sh[threadIdx.x >> 5] = v;
  __syncthreads();
  if (threadIdx.x == 0) {
    double r = 0.0;
    for (int w = 0; w < NT / 32; ++w) r += sh[w];
    sh[32] = r;
  }
  __syncthreads();
  const double r = sh[32];
  __syncthreads();
  return r;
}

// Fixed-rank initial state (Sec. S1.A): psi with weight 1 - (M-1) eps and M - 1
// padding columns sqrt(eps) q_j, the q_j the Gram-Schmidt orthonormalisation of
// Gaussian columns against psi and each other. psi is a basis state, so its
// component is removed by zeroing one row; the rest is Cholesky QR: G = W^dag W
// = L L^dag over the M - 1 Gaussian columns, Q = W L^-dag, which has the same q_j
// (a QR factor with a positive diagonal is unique). Everything is FP64. A second
// round brings the orthogonality from cond(W)^2 2^-53 to 2^-53; there is one where it
// cannot be seen (FP32 states with N >= 4 M: cond(W) < ~3).
//
// A cluster of CTAs per trajectory. The rows go in up to IV parts, chosen by N alone, so
// that the state does not depend on the batch around it; a CTA takes whole parts, in
// tiles of ITR rows in shared memory: draws and Gram sums of a tile in one sweep, the
// parts' G added in their order over distributed shared memory, the M x M factor in
// every CTA, then Q tile by tile. Bound by the FP64 pipe (2 FMA/clk/SM): the draws
// (~100 FP64 instructions a pair) and the 8 N M^2 FMAs of the two products. Column
// by column Gram-Schmidt in one block per trajectory took a block sum and a sweep
// of L2 per column pair: 512 trajectories of N = 2000, M = 20 took 31.5 ms, here
// 6.3 ms; two trajectories 5.7 ms, here 0.3 ms.
constexpr int ITR = 128;            // rows per tile
constexpr int IM = LR_MAX_RANK - 1; // most padding columns
constexpr int IV = 8;               // most parts (the portable cluster size)

__host__ __device__ inline int init_ldt(int m1) { return m1 | 1; }   // odd row stride: no bank conflicts down a column
// parts whose sums a CTA of a team of C keeps (alone it adds them as they come)
inline int init_slots(int C) { return C == 1 ? 1 : (IV + C - 1) / C; }
inline size_t init_smem(int m1, int slots) {
  return sizeof(double2) *
         ((size_t)ITR * init_ldt(m1) + IT + 2 * (size_t)m1 * init_ldt(m1) + (size_t)slots * m1 * (m1 + 1) / 2);
}

template <typename T2>
__global__ void __launch_bounds__(IT) initial_state_kernel(const TrajDev* __restrict__ traj, double2* __restrict__ Wbase,
                                                           T2* __restrict__ Zbase, unsigned long long seed, double eps,
                                                           int max_m1) {
  extern __shared__ __align__(16) unsigned char init_sm[];
  namespace cg = cooperative_groups;
  cg::cluster_group cluster = cg::this_cluster();
  const int C = (int)cluster.num_blocks(), q = (int)cluster.block_rank(), tj = blockIdx.x / C;
  const TrajDev d = traj[tj];
  const int N = d.N, M = d.M, ld = d.ld, M1 = M - 1, ldt = init_ldt(M1);
  const int tid = threadIdx.x, lane = tid & 31, warp = tid >> 5;
  // the layout of the batch's largest rank, the same in every CTA of a cluster
  double2* tile = reinterpret_cast<double2*>(init_sm);                // [ITR][ldt]
  double2* gred = tile + (size_t)ITR * init_ldt(max_m1);              // [groups][nep] partial sums
  double2* L = gred + IT;                                             // [M1][ldt]
  double2* Li = L + (size_t)max_m1 * init_ldt(max_m1);                // [M1][ldt]  L^-1
  double2* gsum = Li + (size_t)max_m1 * init_ldt(max_m1);             // [slots][M1 (M1 + 1) / 2]  G over the own parts
  __shared__ double dinv[IM + 1];
  double2* W = Wbase + d.z_off;
  T2* Z = Zbase + d.z_off;
  const int psi = d.level0 * d.Nr * d.Nf;
  const int V = min(IV, (N + ITR - 1) / ITR);   // parts; those of rank r: [V r / C, V (r + 1) / C)
  const int v_lo = V * q / C, v_hi = V * (q + 1) / C;
  auto row_of = [N, V](int v) { return (int)((long long)N * v / V); };
  const int r_lo = row_of(v_lo), r_hi = row_of(v_hi);
  const int two_rounds = sizeof(T2) == sizeof(double2) || N < 4 * M;
  const unsigned long long ts = splitmix64(seed, (unsigned long long)tj);
  const double w0 = sqrt(1.0 - M1 * eps), we = sqrt(eps);
  // column 0, and the rank padding of the row
  for (int n = r_lo + tid; n < r_hi; n += IT)
    for (int j = 0; j < ld; ++j)
      if (j == 0 || j >= M) Z[(size_t)n * ld + j] = mkc<T2>(j == 0 && n == psi ? w0 : 0.0, 0.0);
  // Gram entry of this thread: pair (gi <= gj) number tid % nep of the upper
  // triangle, over the rows r = group (mod groups) of every tile
  const int ne = M1 * (M1 + 1) / 2, nep = (ne + 31) / 32 * 32, groups = nep ? IT / nep : 0;
  const int ent = nep ? tid % nep : 0, group = nep ? tid / nep : 0;
  int gj = 0;
  while ((gj + 1) * (gj + 2) / 2 <= ent) ++gj;
  const int gi = ent - gj * (gj + 1) / 2;
  const bool mine = ent < ne && group < groups;
  for (int round = 0; round < (M1 > 0 ? 1 + two_rounds : 0); ++round) {
    for (int v = v_lo; v < v_hi; ++v) {
      double gr = 0.0, gim = 0.0;
      const int p_hi = row_of(v + 1);
      for (int t0 = row_of(v); t0 < p_hi; t0 += ITR) {
        const int rows = min(ITR, p_hi - t0);
        for (int e = tid; e < rows * M1; e += IT) {
          const int r = e / M1, j = e - r * M1, n = t0 + r;
          double2 w;
          if (round == 0) {
            const unsigned long long pidx = (unsigned long long)j * N + n;
            const double u1 = uniform_open0(ts, 2ull * pidx), u2 = uniform_open0(ts, 2ull * pidx + 1ull);
            const double rad = sqrt(-2.0 * log(u1));
            double sn, cs;
            sincospi(2.0 * u2, &sn, &cs);
            w = n == psi ? mk(0.0, 0.0) : mk(rad * cs, rad * sn);
            W[(size_t)n * ld + j + 1] = w;
          } else {
            w = W[(size_t)n * ld + j + 1];
          }
          tile[r * ldt + j] = w;
        }
        __syncthreads();
        if (mine)
          for (int r = group; r < rows; r += groups) {
            const double2 a = tile[r * ldt + gi], b = tile[r * ldt + gj];   // conj(a) b
            gr = fma(a.x, b.x, fma(a.y, b.y, gr));
            gim = fma(a.x, b.y, fma(-a.y, b.x, gim));
          }
        __syncthreads();
      }
      if (mine) gred[group * nep + ent] = mk(gr, gim);
      __syncthreads();
      for (int e = tid; e < ne; e += IT) {
        double2 s = gred[e];
        for (int g = 1; g < groups; ++g) s = mk(s.x + gred[g * nep + e].x, s.y + gred[g * nep + e].y);
        double2* out = gsum + (C == 1 ? 0 : v - v_lo) * ne + e;
        *out = C == 1 && v > 0 ? mk(out->x + s.x, out->y + s.y) : s;
      }
      __syncthreads();
    }
    cluster.sync();
    for (int e = tid; e < ne; e += IT) {   // the parts in order; lower triangle G_ji = conj(G_ij)
      double2 s = gsum[e];
      if (C > 1) {
        s = mk(0.0, 0.0);
        for (int r = 0; r < C; ++r)
          for (int k = 0; k < V * (r + 1) / C - V * r / C; ++k) {
            const double2 w = cluster.map_shared_rank(gsum, r)[k * ne + e];
            s = mk(s.x + w.x, s.y + w.y);
          }
      }
      int j = 0;
      while ((j + 1) * (j + 2) / 2 <= e) ++j;
      L[j * ldt + e - j * (j + 1) / 2] = mk(s.x, -s.y);
    }
    cluster.sync();   // every rank has read the partials: they may be overwritten
    for (int k = 0; k < M1; ++k) {   // right-looking Cholesky, warp 0 on the pivot column
      if (warp == 0) {
        const double inv = 1.0 / sqrt(L[k * ldt + k].x);
        __syncwarp();
        if (lane == 0) {
          L[k * ldt + k].x *= inv;
          dinv[k] = inv;
        }
        for (int i = k + 1 + lane; i < M1; i += 32) L[i * ldt + k] = mk(L[i * ldt + k].x * inv, L[i * ldt + k].y * inv);
      }
      __syncthreads();
      const int w = M1 - k - 1;
      for (int e = tid; e < w * w; e += IT) {
        const int i = k + 1 + e / w, j = k + 1 + e % w;
        if (j > i) continue;
        const double2 a = L[i * ldt + k], c = L[j * ldt + k];   // L_ij -= L_ik conj(L_jk)
        L[i * ldt + j] = mk(L[i * ldt + j].x - (a.x * c.x + a.y * c.y), L[i * ldt + j].y - (a.y * c.x - a.x * c.y));
      }
      __syncthreads();
    }
    for (int j = warp; j < M1; j += IT / 32) {   // column j of L^-1 by a warp, lane = row
      double2 x = mk(lane == j ? 1.0 : 0.0, 0.0);
      for (int k = j; k < M1; ++k) {
        double2 xk = mk(__shfl_sync(0xffffffffu, x.x, k), __shfl_sync(0xffffffffu, x.y, k));
        xk = mk(xk.x * dinv[k], xk.y * dinv[k]);
        if (lane == k) {
          x = xk;
        } else if (lane > k && lane < M1) {
          const double2 l = L[lane * ldt + k];
          x = mk(x.x - (l.x * xk.x - l.y * xk.y), x.y - (l.x * xk.y + l.y * xk.x));
        }
      }
      if (lane >= j && lane < M1) Li[lane * ldt + j] = x;
    }
    __syncthreads();
    // Q[n][j] = sum_{i <= j} W[n][i] conj(L^-1[j][i]): a warp takes 32 rows of a
    // tile and the columns p and M1 - 1 - p (equal work for every p)
    const bool last = round == two_rounds;
    const int np = (M1 + 1) / 2;
    for (int t0 = r_lo; t0 < r_hi; t0 += ITR) {
      const int rows = min(ITR, r_hi - t0);
      for (int e = tid; e < rows * M1; e += IT) {
        const int r = e / M1, j = e - r * M1;
        tile[r * ldt + j] = W[(size_t)(t0 + r) * ld + j + 1];
      }
      __syncthreads();
      for (int task = warp; task < (ITR / 32) * np; task += IT / 32) {
        const int r = (task / np) * 32 + lane, p = task % np;
        if (r >= rows) continue;
        for (int h = 0; h < 2; ++h) {
          const int j = h ? M1 - 1 - p : p;
          if (h && j == p) break;
          double xr = 0.0, xi = 0.0;
          for (int i = 0; i <= j; ++i) {
            const double2 a = tile[r * ldt + i], l = Li[j * ldt + i];   // a conj(l)
            xr = fma(a.x, l.x, fma(a.y, l.y, xr));
            xi = fma(a.y, l.x, fma(-a.x, l.y, xi));
          }
          const size_t o = (size_t)(t0 + r) * ld + j + 1;
          if (last) {
            Z[o] = mkc<T2>(we * xr, we * xi);
          } else {
            W[o] = mk(xr, xi);
          }
        }
      }
      __syncthreads();
    }
  }
}

// Rank growth (adaptive rank): one block per trajectory. The source state's
// columns are kept; columns M_src .. M_dst-1 are sqrt(eps) q_j with q_j the
// normalised component of a complex Gaussian vector xi_j (same generator as the
// initial state, pair index (j - M_src) N + n) orthogonal to span(Z_src) and to
// q_{M_src} .. q_{j-1}. The projection onto span(Z_src) is Z G^-1 Z^dag with
// G = Z^dag Z (Cholesky, FP64), applied twice (reorthogonalisation).
__device__ __forceinline__ double2 to_d2(double2 v) { return v; }
__device__ __forceinline__ double2 to_d2(float2 v) { return make_double2(v.x, v.y); }

template <typename T2>
__global__ void __launch_bounds__(IT) grow_kernel(const TrajDev* __restrict__ dtraj, const TrajDev* __restrict__ straj,
                                                  const T2* __restrict__ Zsrc, double2* __restrict__ Wbase,
                                                  T2* __restrict__ Zdst, unsigned long long seed, double eps,
                                                  unsigned* err) {
  __shared__ double sh[33];
  __shared__ double2 L[LR_MAX_RANK][LR_MAX_RANK + 1];
  __shared__ double2 y[LR_MAX_RANK];
  __shared__ int bad;
  const int tj = blockIdx.x;
  const TrajDev d = dtraj[tj], sr = straj[tj];
  const int N = d.N, Ms = sr.M, Md = d.M, lds = sr.ld, ldd = d.ld;
  double2* W = Wbase + d.z_off;
  const T2* Zs = Zsrc + sr.z_off;
  T2* Z = Zdst + d.z_off;
  const unsigned long long ts = splitmix64(seed, (unsigned long long)tj);
  if (threadIdx.x == 0) bad = 0;
  for (int n = threadIdx.x; n < N; n += IT) {
    for (int j = 0; j < Ms; ++j) W[(size_t)n * ldd + j] = to_d2(Zs[(size_t)n * lds + j]);
    for (int j = Ms; j < Md; ++j) {
      const unsigned long long pidx = (unsigned long long)(j - Ms) * N + n;
      const double u1 = uniform_open0(ts, 2ull * pidx), u2 = uniform_open0(ts, 2ull * pidx + 1ull);
      const double r = sqrt(-2.0 * log(u1));
      double sn, cs;
      sincospi(2.0 * u2, &sn, &cs);
      W[(size_t)n * ldd + j] = mk(r * cs, r * sn);
    }
  }
  __syncthreads();
  // inner product <W_i, W_j> = sum_n conj(W_ni) W_nj (fixed-order block sums)
  auto dot = [&](int i, int j) {
    double re = 0.0, im = 0.0;
    for (int n = threadIdx.x; n < N; n += IT) {
      const double2 a = W[(size_t)n * ldd + i], b = W[(size_t)n * ldd + j];
      re += a.x * b.x + a.y * b.y;
      im += a.x * b.y - a.y * b.x;
    }
    re = block_sum<IT>(re, sh);
    im = block_sum<IT>(im, sh);
    return mk(re, im);
  };
  // G = Z^dag Z, lower triangle: G_ij = <W_i, W_j> for i >= j
  for (int i = 0; i < Ms; ++i)
    for (int j = 0; j <= i; ++j) {
      const double2 g = dot(i, j);
      if (threadIdx.x == 0) L[i][j] = g;
    }
  __syncthreads();
  if (threadIdx.x == 0) {   // Cholesky G = L L^dag (serial, M <= 32)
    for (int k = 0; k < Ms && !bad; ++k) {
      double piv = L[k][k].x;
      for (int q = 0; q < k; ++q) piv -= L[k][q].x * L[k][q].x + L[k][q].y * L[k][q].y;
      if (!(piv > 0.0)) {
        bad = 1;
        break;
      }
      const double lkk = sqrt(piv);
      L[k][k] = mk(lkk, 0.0);
      for (int i = k + 1; i < Ms; ++i) {
        double re = L[i][k].x, im = L[i][k].y;   // G_ik - sum_q L_iq conj(L_kq)
        for (int q = 0; q < k; ++q) {
          re -= L[i][q].x * L[k][q].x + L[i][q].y * L[k][q].y;
          im -= L[i][q].y * L[k][q].x - L[i][q].x * L[k][q].y;
        }
        L[i][k] = mk(re / lkk, im / lkk);
      }
    }
  }
  __syncthreads();
  if (bad) {
    if (threadIdx.x == 0) set_error(err, DEV_NOT_PD);
    return;
  }
  for (int j = Ms; j < Md; ++j) {
    for (int pass = 0; pass < 2; ++pass) {
      // remove the span(Z) component: c = Z^dag w, G y = c, w -= Z y
      for (int i = 0; i < Ms; ++i) {
        const double2 c = dot(i, j);
        if (threadIdx.x == 0) y[i] = c;
      }
      __syncthreads();
      if (threadIdx.x == 0) {
        for (int i = 0; i < Ms; ++i) {   // L u = c
          double re = y[i].x, im = y[i].y;
          for (int q = 0; q < i; ++q) {
            re -= L[i][q].x * y[q].x - L[i][q].y * y[q].y;
            im -= L[i][q].x * y[q].y + L[i][q].y * y[q].x;
          }
          y[i] = mk(re / L[i][i].x, im / L[i][i].x);
        }
        for (int i = Ms - 1; i >= 0; --i) {   // L^dag y = u
          double re = y[i].x, im = y[i].y;
          for (int q = i + 1; q < Ms; ++q) {
            re -= L[q][i].x * y[q].x + L[q][i].y * y[q].y;
            im -= L[q][i].x * y[q].y - L[q][i].y * y[q].x;
          }
          y[i] = mk(re / L[i][i].x, im / L[i][i].x);
        }
      }
      __syncthreads();
      for (int n = threadIdx.x; n < N; n += IT) {
        double2 w = W[(size_t)n * ldd + j];
        for (int i = 0; i < Ms; ++i) {
          const double2 a = W[(size_t)n * ldd + i], c = y[i];
          w = mk(w.x - (a.x * c.x - a.y * c.y), w.y - (a.x * c.y + a.y * c.x));
        }
        W[(size_t)n * ldd + j] = w;
      }
      __syncthreads();
      // and the components along the new orthonormal columns so far
      for (int k = Ms; k < j; ++k) {
        const double2 r = dot(k, j);
        for (int n = threadIdx.x; n < N; n += IT) {
          const double2 a = W[(size_t)n * ldd + k], b = W[(size_t)n * ldd + j];
          W[(size_t)n * ldd + j] = mk(b.x - (r.x * a.x - r.y * a.y), b.y - (r.x * a.y + r.y * a.x));
        }
        __syncthreads();
      }
    }
    const double nn = dot(j, j).x;
    const double inv = 1.0 / sqrt(nn);
    for (int n = threadIdx.x; n < N; n += IT) {
      const double2 b = W[(size_t)n * ldd + j];
      W[(size_t)n * ldd + j] = mk(b.x * inv, b.y * inv);
    }
    __syncthreads();
  }
  const double we = sqrt(eps);
  for (int n = threadIdx.x; n < N; n += IT)
    for (int j = 0; j < ldd; ++j) {
      T2 v;
      if (j < Ms) {
        v = Zs[(size_t)n * lds + j];   // the kept columns, unchanged
      } else if (j < Md) {
        const double2 q = W[(size_t)n * ldd + j];
        v.x = q.x * we;
        v.y = q.y * we;
      } else {
        v.x = 0;
        v.y = 0;
      }
      Z[(size_t)n * ldd + j] = v;
    }
}

cudaError_t launch_grow(const DevPtrs& dst, const DevPtrs& src, int n_traj, int prec_fp32, uint64_t seed, double eps,
                        cudaStream_t s) {
  double2* W = reinterpret_cast<double2*>(dst.Za);
  if (prec_fp32)
    grow_kernel<float2><<<n_traj, IT, 0, s>>>(dst.traj, src.traj, reinterpret_cast<const float2*>(src.Zn), W,
                                              reinterpret_cast<float2*>(dst.Zn), seed, eps, dst.err);
  else
    grow_kernel<double2><<<n_traj, IT, 0, s>>>(dst.traj, src.traj, reinterpret_cast<const double2*>(src.Zn), W,
                                               reinterpret_cast<double2*>(dst.Zn), seed, eps, dst.err);
  return cudaGetLastError();
}

template <typename T2>
static cudaError_t launch_initial_t(const DevPtrs& p, const RunParams& rp, int max_N, int max_M, unsigned long long seed,
                                    double eps, cudaStream_t s) {
  int dev = 0, sms = 0;
  cudaError_t e = cudaGetDevice(&dev);
  if (e == cudaSuccess) e = cudaDeviceGetAttribute(&sms, cudaDevAttrMultiProcessorCount, dev);
  if (e == cudaSuccess)
    e = cudaFuncSetAttribute(initial_state_kernel<T2>, cudaFuncAttributeMaxDynamicSharedMemorySize,
                             (int)init_smem(IM, init_slots(2)));
  if (e != cudaSuccess) return e;
  // one CTA per SM in all: a team takes the SMs that the batch leaves over, at
  // least a tile of rows per CTA, within the portable cluster size
  const int C = std::max(1, std::min({IV, sms / std::max(1, rp.n_traj), (max_N + ITR - 1) / ITR}));
  cudaLaunchConfig_t cfg = {};
  cfg.gridDim = dim3(C * rp.n_traj);
  cfg.blockDim = dim3(IT);
  cfg.dynamicSmemBytes = init_smem(std::max(1, max_M - 1), init_slots(C));
  cfg.stream = s;
  cudaLaunchAttribute at[1];
  at[0].id = cudaLaunchAttributeClusterDimension;
  at[0].val.clusterDim.x = C;
  at[0].val.clusterDim.y = 1;
  at[0].val.clusterDim.z = 1;
  cfg.attrs = at;
  cfg.numAttrs = 1;
  return cudaLaunchKernelEx(&cfg, initial_state_kernel<T2>, p.traj, reinterpret_cast<double2*>(p.Za),
                            reinterpret_cast<T2*>(p.Zn), seed, eps, std::max(1, max_M - 1));
}

cudaError_t launch_initial_state(const DevPtrs& p, const RunParams& rp, int max_N, int max_M, int prec_fp32, uint64_t seed,
                                 double eps, cudaStream_t s) {
  if (prec_fp32) return launch_initial_t<float2>(p, rp, max_N, max_M, seed, eps, s);
  return launch_initial_t<double2>(p, rp, max_N, max_M, seed, eps, s);
}

// One block per candidate: trapezoid of |beta_e - beta_g|^2 over the step grid,
// SNR = sqrt(2 eta kappa S), eps_a = erfc(SNR/2)/2 + tau gamma/2.
__global__ void __launch_bounds__(ET) eps_a_kernel(DevPtrs p, RunParams rp, long n_added) {
  __shared__ double sh[33];
  const int c = blockIdx.x;
  const long step = (long)*p.dstep + n_added;
  if (step < 0 || step > rp.max_steps) {   // the integrate before it refused to run past capacity
    if (c == 0 && threadIdx.x == 0) set_error(p.err, DEV_CAPACITY);
    return;
  }
  const TrajDev d = p.traj[2 * c];
  const double2* bg = p.beta + (size_t)(2 * c) * (rp.max_steps + 1);
  const double2* be = p.beta + (size_t)(2 * c + 1) * (rp.max_steps + 1);
  double acc = 0.0;
  for (long i = threadIdx.x; i <= step; i += ET) {
    const double dx = be[i].x - bg[i].x, dy = be[i].y - bg[i].y;
    const double w = (i == 0 || i == step) ? 0.5 : 1.0;
    acc += w * (dx * dx + dy * dy);
  }
  acc = block_sum<ET>(acc, sh);
  // ionization penalty (Sec. S3.B): populations of transmon levels k >= 2 of
  // both trajectories, trapezoid over the recorded grid up to the last record
  const long last = step / rp.pop_every;
  const int Nt = d.Nt;
  double ion = 0.0;
  for (long r = threadIdx.x; r <= last; r += ET) {
    const double w = (r == 0 || r == last) ? 0.5 : 1.0;
    double sum = 0.0;
    for (int tj = 2 * c; tj <= 2 * c + 1; ++tj)
      for (int k = 2; k < Nt; ++k) sum += p.pops[((size_t)tj * rp.n_rec + r) * rp.nt_max + k];
    ion += w * sum;
  }
  ion = block_sum<ET>(ion, sh);
  if (threadIdx.x == 0) {
    const double S = step > 0 ? rp.dt * acc : 0.0;
    const double snr = sqrt(2.0 * rp.eta * d.kappa * S);
    const double tau = (double)step * rp.dt;
    const double e = 0.5 * erfc(0.5 * snr) + 0.5 * tau * d.gamma;
    p.eps_a[c] = e;
    const double T = (step > 0 && last > 0) ? ion * rp.pop_every * rp.dt / tau : 0.0;
    p.ion[c] = T;
    p.loss[c] = log10(e + T);
    if (!isfinite(e)) set_error(p.err, DEV_NONFINITE);
  }
}

// Advance the device step counter once every block of eps_a_kernel has read it
// (a kernel of its own, ordered after it in the stream); a run past capacity
// leaves the counter where it was.
__global__ void advance_step_kernel(long long* dstep, long n_added, long max_steps) {
  const long long s = *dstep + n_added;
  if (s >= 0 && s <= max_steps) *dstep = s;
}

cudaError_t launch_eps_a(const DevPtrs& p, const RunParams& rp, long n_added, cudaStream_t s) {
  eps_a_kernel<<<rp.n_cand, ET, 0, s>>>(p, rp, n_added);
  cudaError_t e = cudaGetLastError();
  if (e != cudaSuccess) return e;
  advance_step_kernel<<<1, 1, 0, s>>>(p.dstep, n_added, rp.max_steps);
  return cudaGetLastError();
}

__global__ void convert_kernel(const void* __restrict__ src, void* __restrict__ dst, long long n, int to_fp32) {
  for (long long i = (long long)blockIdx.x * blockDim.x + threadIdx.x; i < n; i += (long long)gridDim.x * blockDim.x) {
    if (to_fp32) {
      const double2 v = reinterpret_cast<const double2*>(src)[i];
      reinterpret_cast<float2*>(dst)[i] = make_float2((float)v.x, (float)v.y);
    } else {
      const float2 v = reinterpret_cast<const float2*>(src)[i];
      reinterpret_cast<double2*>(dst)[i] = make_double2(v.x, v.y);
    }
  }
}

cudaError_t launch_convert(const void* src, void* dst, long long n, int to_fp32, cudaStream_t s) {
  const int blocks = (int)((n + 255) / 256 < 1024 ? (n + 255) / 256 : 1024);
  convert_kernel<<<blocks < 1 ? 1 : blocks, 256, 0, s>>>(src, dst, n, to_fp32);
  return cudaGetLastError();
}

}  // namespace lr
