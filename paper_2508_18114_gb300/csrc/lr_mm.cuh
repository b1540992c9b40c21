// The M x M phase of an RK4 stage, shared by the fused kernels: G^-1 of the
// Gram matrix by symmetric sweeps with the entries in registers, and the
// double-word FP32 arithmetic (~2^-48 relative) in which the FP32 state runs it.
#pragma once

#include "lr_internal.cuh"

namespace lr {

// ----------------------------------------------------------------- double-word arithmetic
// An unevaluated sum of two floats hi + lo: exact FP32 products by FMA
// (TwoProduct), Knuth's two-sum, results normalised: ~2^-48 relative.
struct alignas(8) DW {
  float hi, lo;
};
__device__ __forceinline__ void dw_add_prod(DW& s, float a, float b) {   // s += a b
  const float p = a * b;
  const float e = fmaf(a, b, -p);
  const float t = s.hi + p;
  const float bp = t - s.hi;
  const float err = (s.hi - (t - bp)) + (p - bp);
  s.hi = t;
  s.lo += err + e;
}
__device__ __forceinline__ void dw_add(DW& s, const DW& o) {
  const float t = s.hi + o.hi;
  const float bp = t - s.hi;
  const float err = (s.hi - (t - bp)) + (o.hi - bp);
  s.hi = t;
  s.lo += err + o.lo;
}
__device__ __forceinline__ void dw_add_f(DW& s, float x) {   // s += x (Knuth's two-sum into hi)
  const float t = s.hi + x;
  const float bp = t - s.hi;
  s.lo += (s.hi - (t - bp)) + (x - bp);
  s.hi = t;
}
__device__ __forceinline__ double dw_value(const DW& s) { return (double)s.hi + (double)s.lo; }
__device__ __forceinline__ DW dw_norm(DW a) {   // |lo| <= ulp(hi) / 2
  DW r;
  r.hi = a.hi + a.lo;
  r.lo = a.lo - (r.hi - a.hi);
  return r;
}
struct alignas(16) DWC {
  DW re, im;
};
// A sum of a team's double-word partials in three floats: each addition keeps what lies
// below 2^-48 of the sum, which a double-word one drops (an FP64 sum of the same terms
// holds the FP64 pipe for ~1000 cycles at M = 20).
struct DWSum {
  float h = 0.f, m = 0.f, l = 0.f;
  static __device__ __forceinline__ float two_sum(float a, float b, float& e) {
    const float s = a + b, t = s - a;
    e = (a - (s - t)) + (b - t);
    return s;
  }
  __device__ __forceinline__ void add(DW v) {
    float e1, e2, e3;
    h = two_sum(h, v.hi, e1);
    m = two_sum(m, v.lo, e2);
    m = two_sum(m, e1, e3);
    l += e2 + e3;
  }
  __device__ __forceinline__ DW dw() const { return dw_norm(DW{h, m + l}); }
  __device__ __forceinline__ double value() const { return (double)h + ((double)m + (double)l); }
};

// ----------------------------------------------------------------- entry arithmetic
__device__ __forceinline__ float rcp_approx(float x) {   // 1 / x to an ulp: the start of both Newton steps
  float r;
  asm("rcp.approx.ftz.f32 %0, %1;" : "=f"(r) : "f"(x));
  return r;
}
// Complex entries C and real pivots R of the matrix that is swept, in
// double-word FP32 (FP32 state) or FP64.
struct DwArith {
  using C = DWC;
  using R = DW;
  static __device__ __forceinline__ C minus_one() { return C{{-1.f, 0.f}, {0.f, 0.f}}; }
  static __device__ __forceinline__ C zero() { return C{{0.f, 0.f}, {0.f, 0.f}}; }
  static __device__ __forceinline__ C conj(C v) { return C{v.re, {-v.im.hi, -v.im.lo}}; }
  static __device__ __forceinline__ C neg(C v) { return C{{-v.re.hi, -v.re.lo}, {-v.im.hi, -v.im.lo}}; }
  static __device__ __forceinline__ float magnitude(C v) { return v.re.hi; }
  struct Sum {   // of a team's partials
    DWSum re, im;
    __device__ __forceinline__ void add(C v) { re.add(v.re), im.add(v.im); }
    __device__ __forceinline__ C entry() const { return C{re.dw(), im.dw()}; }
    __device__ __forceinline__ double2 value() const { return make_double2(re.value(), im.value()); }
  };
  static __device__ __forceinline__ double2 value(C v) { return make_double2(dw_value(v.re), dw_value(v.im)); }
  // p e with p + e = a b to ~2^-48 (not normalised)
  static __device__ __forceinline__ DW prod(DW a, DW b) {
    DW r;
    r.hi = a.hi * b.hi;
    r.lo = fmaf(a.lo, b.hi, fmaf(a.hi, b.lo, fmaf(a.hi, b.hi, -r.hi)));
    return r;
  }
  // a - x - y: two two-sums of the leading parts, the small parts added plainly
  static __device__ __forceinline__ DW sub2(DW a, DW x, DW y) {
    const float t = a.hi - x.hi, b1 = t - a.hi, e1 = (a.hi - (t - b1)) - (x.hi + b1);
    const float u = t - y.hi, b2 = u - t, e2 = (t - (u - b2)) - (y.hi + b2);
    return dw_norm(DW{u, ((a.lo - x.lo) - y.lo) + (e1 + e2)});
  }
  // v - x conj(y) d
  static __device__ __forceinline__ C update(C v, C x, C y, R d) {
    const DW sr = dw_norm(prod(y.re, d)), si = dw_norm(prod(y.im, d));
    const DW ni = DW{-si.hi, -si.lo};
    return C{sub2(v.re, prod(x.re, sr), prod(x.im, si)), sub2(v.im, prod(x.im, sr), prod(x.re, ni))};
  }
  // 1 / p for p > 0: the FP32 quotient r and the correction r (e + e^2), e = 1 - p r
  static __device__ __forceinline__ R recip(C p) {
    const float r = rcp_approx(p.re.hi);
    const float e = fmaf(-p.re.lo, r, fmaf(-p.re.hi, r, 1.0f));
    return dw_norm(DW{r, r * fmaf(e, e, e)});
  }
  static __device__ __forceinline__ R one() { return R{1.f, 0.f}; }
  static __device__ __forceinline__ bool breakdown(C p, float d0, int) {
    return !(p.re.hi > 1e-13f * d0) || !isfinite(p.re.hi) || p.re.hi < 1e-30f;
  }
};

struct F64Arith {
  using C = double2;
  using R = double;
  static __device__ __forceinline__ C minus_one() { return mk(-1.0, 0.0); }
  static __device__ __forceinline__ C zero() { return mk(0.0, 0.0); }
  static __device__ __forceinline__ C conj(C v) { return mk(v.x, -v.y); }
  static __device__ __forceinline__ C neg(C v) { return mk(-v.x, -v.y); }
  static __device__ __forceinline__ double magnitude(C v) { return v.x; }
  struct Sum {
    double x = 0.0, y = 0.0;
    __device__ __forceinline__ void add(C v) { x += v.x, y += v.y; }
    __device__ __forceinline__ C entry() const { return mk(x, y); }
    __device__ __forceinline__ double2 value() const { return mk(x, y); }
  };
  static __device__ __forceinline__ double2 value(C v) { return v; }
  static __device__ __forceinline__ C update(C v, C x, C y, R d) {   // v - x conj(y) d
    const double sr = y.x * d, si = y.y * d;
    return mk(fma(-x.y, si, fma(-x.x, sr, v.x)), fma(x.x, si, fma(-x.y, sr, v.y)));
  }
  // Newton-Raphson r <- r (2 - p r) from the FP32 quotient: 24 -> 48 -> 96 bits
  static __device__ __forceinline__ R recip(C p) {
    double r = (double)rcp_approx((float)p.x);
    r = r * fma(-p.x, r, 2.0);
    return r * fma(-p.x, r, 2.0);
  }
  static __device__ __forceinline__ R one() { return 1.0; }
  static __device__ __forceinline__ bool breakdown(C p, double d0, int) {
    return !(p.x > 1e-13 * d0) || !isfinite(p.x) || p.x < 1e-30;
  }
};

// ----------------------------------------------------------------- the inverse
// Warps that hold entries of an M x M lower triangle, of a block of `nwarp`.
__device__ __forceinline__ int mm_warps(int M, int nwarp) { return min(nwarp, (M * (M + 1) / 2 + 31) / 32); }

template <typename A>
struct MmShared {   // column k of the matrix and 1 / a_kk, by parity of k
  typename A::C col[2][LR_MAX_RANK];
  typename A::R rec[2];
  int bad;
};

// G^-1 of a Hermitian positive definite G by M symmetric sweeps (Gauss-Jordan
// on the diagonal): sweep k sets a_ij -= a_ik a_kj / a_kk, a_ik /= a_kk, a_kj /=
// a_kk and a_kk = -1 / a_kk, and the matrix stays Hermitian, so its lower triangle
// is enough; after M of them it is -G^-1. Entry e of the triangle (tri[e] = (i,
// j), i >= j) belongs to thread e mod NT, which passes it in g and keeps it in
// registers; a sweep reads only column k, which the owners left in shared memory
// at the end of sweep k - 1: one barrier per sweep, among the warps that hold
// entries. The owner of the next pivot forms its reciprocal before the barrier.
// With column k's own entry stored as -1, v - c_i conj(c_j) / a_kk (v = 0 in row
// and column k) is every case of the sweep.
//
// Bound by the latency of a sweep (update, reciprocal, barrier; ~700 cycles in
// double-word), not by its M^2/2 updates. It replaces an L D L^dag factorisation,
// L^-1 and G^-1 = L^-dag D^-1 L^-1 (three passes with ~870 cycles per elimination
// step): 36k -> 14k cycles at M = 20. The error is that of the
// factorisation, the condition number of the scaled G times the unit roundoff: X_k =
// G^-1 T_k in FP64 against 200 bits, M = 4 .. 32, cond 1 .. 5e9, has 0.2 to 0.8
// of the forward error of Cholesky substitution.
//
// Called by the warps below mm_warps(M, NT / 32) with all their lanes; the result
// is in gi[i * ldg + j] after the block barrier that the caller adds.
template <typename A, int NT>
__device__ __forceinline__ void mm_invert(typename A::C (&g)[2], typename A::C* gi, int ldg, MmShared<A>& sh,
                                          const short2* tri, int M, int tid) {
  using C = typename A::C;
  const int ne = M * (M + 1) / 2, nthr = mm_warps(M, NT / 32) * 32;
  auto sync = [nthr]() { asm volatile("bar.sync 2, %0;" ::"r"(nthr) : "memory"); };
  int ei[2], ej[2];
  decltype(A::magnitude(g[0])) d0[2];
#pragma unroll
  for (int q = 0; q < 2; ++q) {
    const int e = tid + q * NT;
    ei[q] = e < ne ? tri[e].x : -1;
    ej[q] = e < ne ? tri[e].y : -1;
    d0[q] = A::magnitude(g[q]);
  }
  // column k of entry q's value, and the pivot's reciprocal
  auto leave = [&](int q, int k) {
    if (ej[q] == k) {
      if (ei[q] == k) {
        const bool bad = A::breakdown(g[q], d0[q], k);
        if (bad) sh.bad = 1;
        sh.rec[k & 1] = bad ? A::one() : A::recip(g[q]);
        sh.col[k & 1][k] = A::minus_one();
      } else {
        sh.col[k & 1][ei[q]] = g[q];
      }
    } else if (ei[q] == k) {
      sh.col[k & 1][ej[q]] = A::conj(g[q]);
    }
  };
#pragma unroll
  for (int q = 0; q < 2; ++q) leave(q, 0);
  sync();
  for (int k = 0; k < M; ++k) {
    const auto d = sh.rec[k & 1];
#pragma unroll
    for (int q = 0; q < 2; ++q) {
      if (ei[q] < 0) continue;
      const C v = ei[q] == k || ej[q] == k ? A::zero() : g[q];
      g[q] = A::update(v, sh.col[k & 1][ei[q]], sh.col[k & 1][ej[q]], d);
      leave(q, k + 1);
    }
    sync();
  }
#pragma unroll
  for (int q = 0; q < 2; ++q) {
    if (ei[q] < 0) continue;
    const C v = A::neg(g[q]);
    gi[ei[q] * ldg + ej[q]] = v;
    if (ei[q] != ej[q]) gi[ej[q] * ldg + ei[q]] = A::conj(v);
  }
}

// Entry (m, l) of X = G^-1 T: row m of G^-1 (gi), column l of T (t, row stride ldt).
// FP32 state: the FP32 T times the double-word G^-1 in a double-word sum, rounded
// once (G^-1 has entries up to 1 / p_M; FP32 products would lose the small columns).
__device__ __forceinline__ float2 mm_xk(const DWC* gi, const float2* t, int ldt, int M) {
  DW re{0.f, 0.f}, im{0.f, 0.f};
  for (int j = 0; j < M; ++j) {
    const DWC g = gi[j];
    const float2 v = t[j * ldt];
    dw_add_prod(re, g.re.hi, v.x);
    dw_add_prod(im, g.re.hi, v.y);
    dw_add_prod(re, -g.im.hi, v.y);
    dw_add_prod(im, g.im.hi, v.x);
    re.lo = fmaf(-g.im.lo, v.y, fmaf(g.re.lo, v.x, re.lo));
    im.lo = fmaf(g.im.lo, v.x, fmaf(g.re.lo, v.y, im.lo));
  }
  return make_float2(re.hi + re.lo, im.hi + im.lo);
}
__device__ __forceinline__ double2 mm_xk(const double2* gi, const double2* t, int ldt, int M) {
  double xr = 0.0, xi = 0.0;
  for (int j = 0; j < M; ++j) {
    const double2 g = gi[j], v = t[j * ldt];
    xr = fma(g.x, v.x, fma(-g.y, v.y, xr));
    xi = fma(g.x, v.y, fma(g.y, v.x, xi));
  }
  return mk(xr, xi);
}

// ----------------------------------------------------------------- whole-chip schedules
// Entry e of the upper triangle by columns: (i, j), i <= j (the lower one by rows: (j, i)).
__device__ __forceinline__ void tri_entry(int e, int& i, int& j) {
  j = (int)((sqrtf(8.f * e + 1.f) - 1.f) * 0.5f);
  while (j * (j + 1) / 2 > e) --j;
  while ((j + 1) * (j + 2) / 2 <= e) ++j;
  i = e - j * (j + 1) / 2;
}

constexpr int ST = 544;   // threads of the solve kernels: one entry of the 32 x 32 triangle each

// The FP64 entry arithmetic of the sweeps; a pivot counts as zero where it is lost in
// the rounding of the k updates of its diagonal entry so far (k 2^-51 of it), so that a
// rank-deficient state is told whatever the sign of that rounding and any other is taken.
struct WidePivot : F64Arith {
  static __device__ __forceinline__ double recip(double2 p) {
    return p.x > 1e-30 && p.x < 1e30 ? F64Arith::recip(p) : 1.0 / p.x;
  }
  static __device__ __forceinline__ bool breakdown(double2 p, double d0, int k) {
    return !(p.x > k * 0x1p-51 * d0) || !isfinite(p.x);
  }
};
// Entries of G and T from their FP64 sums. FP32 state: G in double-word FP32 and an FP32
// T, as in the fused kernels (a sweep of double-word FP32 takes ~2/3 of an FP64 one).
__device__ __forceinline__ void to_entry(double2 v, double2& e) { e = v; }
__device__ __forceinline__ void to_entry(double2 v, DWC& e) {
  e.re.hi = (float)v.x;
  e.re.lo = (float)(v.x - (double)e.re.hi);
  e.im.hi = (float)v.y;
  e.im.lo = (float)(v.y - (double)e.im.hi);
}
__device__ __forceinline__ void to_entry(double2 v, float2& e) { e = make_float2((float)v.x, (float)v.y); }
__device__ __forceinline__ double2 to_sum(double2 v) { return v; }
__device__ __forceinline__ double2 to_sum(float2 v) { return mk((double)v.x, (double)v.y); }
template <typename A> struct XEntry { using t = double2; };
template <> struct XEntry<DwArith> { using t = float2; };

// The block's share of X_k = G^-1 T_k: whole columns of the K M of all jumps, XC at a
// time with their T entries in shared memory (read from L2 in the dot products, a
// chain of M loads, they took as long as the sweeps).
constexpr int XC = 8;
template <typename A>
struct XColumns {
  typename XEntry<A>::t t[XC][LR_MAX_RANK + 1];
  // columns [c0, c0 + n) of T [K][M][M]
  __device__ __forceinline__ void load(const double2* T, int M, int c0, int n, int tid) {
    for (int e = tid; e < n * M; e += ST) {
      const int c = e / M, l = e - c * M, k = (c0 + c) / M, j = c0 + c - k * M;
      to_entry(T[(k * M + l) * M + j], t[c][l]);
    }
  }
};
// Called by every thread with the first columns loaded and G^-1 in Gs, both behind a
// barrier; put(k, i, j, X_ij) stores.
template <typename A, typename Put>
__device__ __forceinline__ void x_columns(XColumns<A>& xc, const typename A::C* Gs, int ldg, const double2* T, int M, int lo,
                                          int hi, int tid, Put put) {
  for (int c0 = lo; c0 < hi; c0 += XC) {
    const int n = min(XC, hi - c0);
    if (c0 > lo) {
      __syncthreads();
      xc.load(T, M, c0, n, tid);
      __syncthreads();
    }
    for (int e = tid; e < n * M; e += ST) {
      const int c = e / M, i = e - c * M, k = (c0 + c) / M;
      put(k, i, c0 + c - k * M, to_sum(mm_xk(Gs + i * ldg, xc.t[c], 1, M)));
    }
  }
}

}  // namespace lr
