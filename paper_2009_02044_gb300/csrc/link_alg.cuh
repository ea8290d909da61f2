// Arithmetic on stored links.
//
// FP64 links are stored and multiplied as full matrices (Group<NC, double>).
// FP32 links are stored and multiplied as their deviation from the identity,
// d = U - 1.  Links near the identity (weak fields, vacuum, and the slowly
// varying pure-gauge links of the nuclei, |U - 1| <~ 0.1) then carry
// rounding errors of the size u |d| instead of u, in storage and in every
// product, so the force -- a small anti-hermitian difference of O(1)
// products -- keeps about log10(1/|d|) more digits in FP32.
//
// Interface shared by both representations (M = a stored-form link):
//   ident, mul, mul_d (x y^+), d_mul (x^+ y)       products of links
//   Sum, zero_sum, sum_add                          weighted staple sums
//   proj_mul(u, S)                                  Im tr t^a (U S)
//   staple_fwd(x, y, z), staple_bwd(x, y, z)        x y^+ z^+, (x y)^+ z
//   proj_prod(x, y), proj_prod_d(x, y)              Im tr t^a (x y), (x y^+)
//                                                   of two stored-form links
//   expi(v, c)                                      exp(i c v^a t^a)
//   evolve(v, c, u)                                 exp(i c v^a t^a) u,
//                                                   re-unitarised in FP32
//   reunit, adj (U q U^+), adj_dag (U^+ q U)
// Links are members of SU(N); staple_fwd, staple_bwd, adj and adj_dag with ANY
// true take them as any matrices (SU(2): real quaternions).
//
// The FP32 forms are templates over the lane type T: float (one site per
// thread) or f2 (pair.cuh: two sites per thread in the lanes of the packed
// f32x2 instructions).  With T = float every expression is the scalar one.
#pragma once
#include "su_n.cuh"
#ifdef __CUDACC__
#include "pair.cuh"
#endif

namespace glasma {
// fma for the scalar lane types, visible next to the f2 overload of the
// same name (which would otherwise hide the global ones in this namespace)
GL_HD float fma(float a, float b, float c) { return fmaf(a, b, c); }
GL_HD double fma(double a, double b, double c) { return ::fma(a, b, c); }
// lane helpers for T = float (pair.cuh has the f2 forms)
GL_HD bool all_zero_s(float a) { return a == 0.f; }
GL_HD bool any_gt_s(float a, float b) { return a > b; }
GL_HD bool all_abs_lt_s(float a, float b) { return fabsf(a) < b; }
GL_HD float lane_div_s(float a, float b) { return a / b; }
// a / b, and 0 in a lane where b = 0 (a scalar caller has returned before)
GL_HD float lane_div0_s(float a, float b) { return a / b; }
#ifdef __CUDACC__
__device__ __forceinline__ bool all_zero_s(f2 a) { return all_zero(a); }
__device__ __forceinline__ bool any_gt_s(f2 a, float b) { return any_gt(a, b); }
__device__ __forceinline__ bool all_abs_lt_s(f2 a, float b) { return all_abs_lt(a, b); }
__device__ __forceinline__ f2 lane_div_s(f2 a, f2 b) { return lane_div(a, b); }
__device__ __forceinline__ f2 lane_div0_s(f2 a, f2 b) {
  return f2(b.v.x != 0.f ? a.v.x / b.v.x : 0.f, b.v.y != 0.f ? a.v.y / b.v.y : 0.f);
}
__device__ __forceinline__ f2 gl_sqrt(f2 x) { return lane_sqrt(x); }
__device__ __forceinline__ void gl_sincos(f2 x, f2* s, f2* c) { *s = lane_sincos_s(x, c); }
#endif
}  // namespace glasma

namespace glasma {

template <int NC, typename R> struct LinkAlg;

// ---------------------------------------------------------------------------
// Full matrices (FP64 state).
// ---------------------------------------------------------------------------
template <int NC>
struct LinkAlg<NC, double> : Group<NC, double> {
  typedef Group<NC, double> G;
  typedef typename G::M M;
  static constexpr bool kDelta = false;
  typedef M Sum;
  GL_HD static M full(const M& u) { return u; }
  GL_HD static M evolve(const double* v, double c, const M& u) { return G::evolve(v, c, u); }
  GL_HD static Sum zero_sum() { return G::zero(); }
  GL_HD static void sum_add(Sum& s, double w, const M& t) { G::scale_add(s, w, t); }
  template <bool ANY = false>
  GL_HD static M staple_fwd(const M& x, const M& y, const M& z) { return G::mul_d(G::mul_d(x, y), z); }
  template <bool ANY = false>
  GL_HD static M staple_bwd(const M& x, const M& y, const M& z) { return G::d_mul(G::mul(x, y), z); }
  GL_HD static void proj_mul_sum(const M& u, const Sum& s, double* out) { G::proj_mul(u, s, out); }
  GL_HD static void proj_prod(const M& x, const M& y, double* out) { G::proj_mul(x, y, out); }
  GL_HD static void proj_prod_d(const M& x, const M& y, double* out) { G::proj_mul(x, G::dag(y), out); }
};

// ---------------------------------------------------------------------------
// SU(3), FP32, deviation form: M holds d = U - 1 (row major).
// ---------------------------------------------------------------------------
template <typename T>
struct LinkAlgDev3 {
  typedef T R;
  typedef Group<3, T> G;
  typedef typename G::M M;
  static constexpr int NA = 8;
  static constexpr bool kDelta = true;

  GL_HD static M ident() { return G::zero(); }
  GL_HD static M full(const M& d) {
    M u = d;
    u.m[0].re += 1.f;
    u.m[4].re += 1.f;
    u.m[8].re += 1.f;
    return u;
  }
  // (1+x)(1+y) - 1 = x (1+y) + y: the products carry the small factor x,
  // so their rounding stays of the size u |x| even though 1+y is O(1).
  GL_HD static M mul(const M& x, const M& y) {
    const M y1 = full(y);
    M r;
#pragma unroll
    for (int i = 0; i < 3; ++i)
#pragma unroll
      for (int j = 0; j < 3; ++j) {
        cplx<R> acc = fma_c(x.m[3 * i], y1.m[j], y.m[3 * i + j]);
        acc = fma_c(x.m[3 * i + 1], y1.m[3 + j], acc);
        acc = fma_c(x.m[3 * i + 2], y1.m[6 + j], acc);
        r.m[3 * i + j] = acc;
      }
    return r;
  }
  // (1+x)(1+y)^+ - 1 = x (1+y)^+ + y^+
  GL_HD static M mul_d(const M& x, const M& y) {
    const M y1 = full(y);
    M r;
#pragma unroll
    for (int i = 0; i < 3; ++i)
#pragma unroll
      for (int j = 0; j < 3; ++j) {
        cplx<R> acc = fma_cj(x.m[3 * i], y1.m[3 * j], cj(y.m[3 * j + i]));
        acc = fma_cj(x.m[3 * i + 1], y1.m[3 * j + 1], acc);
        r.m[3 * i + j] = fma_cj(x.m[3 * i + 2], y1.m[3 * j + 2], acc);
      }
    return r;
  }
  // (1+x)^+(1+y) - 1 = (1+x)^+ y + x^+
  GL_HD static M d_mul(const M& x, const M& y) {
    const M x1 = full(x);
    M r;
#pragma unroll
    for (int i = 0; i < 3; ++i)
#pragma unroll
      for (int j = 0; j < 3; ++j) {
        cplx<R> acc = fma_cj(y.m[j], x1.m[i], cj(x.m[3 * j + i]));
        acc = fma_cj(y.m[3 + j], x1.m[3 + i], acc);
        r.m[3 * i + j] = fma_cj(y.m[6 + j], x1.m[6 + i], acc);
      }
    return r;
  }

  // A staple is a product of three links, so a link itself: two of its rows
  // take the same two rows (staple_bwd: columns) of the inner product, and the
  // third is the conjugate of their cross product, written for the deviations as in reunit.  176
  // multiply-adds and a third of one link's loads less than the 216 of two full
  // products, for every kernel that sums staples.  The third row repeats the
  // rounding of the first two, where it had its own; so each sum here takes its
  // products of two deviations first and the two terms of first order last, and
  // rounds twice instead of six times at their size, and staple_fwd and
  // staple_bwd derive different rows.  SU(3) 512 x 64^2: 0.446 -> 0.423 ms per step
  // (staged), 0.470 -> 0.435 (staple), T^{mu nu} 0.459 -> 0.442, improved scheme
  // 3.39 -> 3.24; rms error against FP64, with the order of proj_mul_sum below, of
  // E 1.47e-5 -> 1.35e-5 of its rms, of U 2.1e-7 -> 1.9e-7 (80 x 64^2, 40 steps, six
  // seeds); without the two orders U's was 1.3 times larger than before.
  template <int i, int j>
  GL_HD static cplx<R> dev_dot(const cplx<R>& x0, const cplx<R>& x1, const cplx<R>& x2, const cplx<R>& y0,
                               const cplx<R>& y1, const cplx<R>& y2) {
    // entry (i, j) of (1 + x)(1 + y) - 1 from row i of x and column j of y
    const cplx<R> x[3] = {x0, x1, x2}, y[3] = {y0, y1, y2};
    constexpr int l = i == j ? (i + 1) % 3 : 3 - i - j, m = i == j ? (i + 2) % 3 : j;
    cplx<R> s;
    s.re = fma(-x[l].im, y[l].im, x[l].re * y[l].re);
    s.im = fma(x[l].im, y[l].re, x[l].re * y[l].im);
    if (i == j) {
      s = fma_c(x[m], y[m], s);
      s.re = fma(-x[i].im, y[i].im, s.re) + y[i].re;
      s.re = fma(x[i].re, 1.f + y[i].re, s.re);
    } else {
      s.re = fma(-x[i].im, y[i].im, fma(-x[j].im, y[j].im, s.re));
      s.im = fma(x[i].im, y[i].re, fma(x[j].re, y[j].im, s.im));
      s.re = fma(x[j].re, 1.f + y[j].re, fma(1.f + x[i].re, y[i].re, s.re));
    }
    s.im = fma(x[j].im, 1.f + y[j].re, fma(1.f + x[i].re, y[i].im, s.im));
    return s;
  }
  template <int i> GL_HD static void dev_row(const M& x, const M& y, M& t) {  // row i of x y
    const cplx<R>*a = &x.m[3 * i], *b = y.m;
    t.m[3 * i] = dev_dot<i, 0>(a[0], a[1], a[2], b[0], b[3], b[6]);
    t.m[3 * i + 1] = dev_dot<i, 1>(a[0], a[1], a[2], b[1], b[4], b[7]);
    t.m[3 * i + 2] = dev_dot<i, 2>(a[0], a[1], a[2], b[2], b[5], b[8]);
  }
  template <int i> GL_HD static void dev_row_d(const M& x, const M& y, M& t) {  // row i of x y^+
    const cplx<R>*a = &x.m[3 * i], *b = y.m;
    t.m[3 * i] = dev_dot<i, 0>(a[0], a[1], a[2], cj(b[0]), cj(b[1]), cj(b[2]));
    t.m[3 * i + 1] = dev_dot<i, 1>(a[0], a[1], a[2], cj(b[3]), cj(b[4]), cj(b[5]));
    t.m[3 * i + 2] = dev_dot<i, 2>(a[0], a[1], a[2], cj(b[6]), cj(b[7]), cj(b[8]));
  }
  template <int i> GL_HD static void d_dev_row(const M& x, const M& y, M& t) {  // row i of x^+ y
    const cplx<R>*a = &x.m[i], *b = y.m;
    t.m[3 * i] = dev_dot<i, 0>(cj(a[0]), cj(a[3]), cj(a[6]), b[0], b[3], b[6]);
    t.m[3 * i + 1] = dev_dot<i, 1>(cj(a[0]), cj(a[3]), cj(a[6]), b[1], b[4], b[7]);
    t.m[3 * i + 2] = dev_dot<i, 2>(cj(a[0]), cj(a[3]), cj(a[6]), b[2], b[5], b[8]);
  }
  template <int j> GL_HD static void dev_col(const M& x, const M& y, M& t) {  // column j of x y
    const cplx<R>*a = x.m, *b = &y.m[j];
    t.m[j] = dev_dot<0, j>(a[0], a[1], a[2], b[0], b[3], b[6]);
    t.m[3 + j] = dev_dot<1, j>(a[3], a[4], a[5], b[0], b[3], b[6]);
    t.m[6 + j] = dev_dot<2, j>(a[6], a[7], a[8], b[0], b[3], b[6]);
  }
  // row r from the two after it, conj(row r1 x row r2)
  template <int r> GL_HD static void third_row(M& t) {
    constexpr int r1 = (r + 1) % 3, r2 = (r + 2) % 3;
    const cplx<R>*a = &t.m[3 * r1], *b = &t.m[3 * r2];
    const R a1 = 1.f + a[r1].re, b2 = 1.f + b[r2].re;
    cplx<R>&p = t.m[3 * r + r1], &q = t.m[3 * r + r2], &d = t.m[4 * r];
    p.re = fma(-a[r].re, b2, fma(a[r].im, b[r2].im, fma(-a[r2].im, b[r].im, a[r2].re * b[r].re)));
    p.im = fma(a[r].im, b2, fma(a[r].re, b[r2].im, fma(-a[r2].im, b[r].re, -a[r2].re * b[r].im)));
    q.re = fma(-a1, b[r].re, fma(a[r1].im, b[r].im, fma(-a[r].im, b[r1].im, a[r].re * b[r1].re)));
    q.im = fma(a1, b[r].im, fma(a[r1].im, b[r].re, fma(-a[r].im, b[r1].re, -a[r].re * b[r1].im)));
    d.re = fma(a[r1].re, b2, fma(-a[r1].im, b[r2].im, fma(a[r2].im, b[r1].im, -a[r2].re * b[r1].re)) + b[r2].re);
    d.im = fma(-a[r1].im, b2, fma(-a1, b[r2].im, fma(a[r2].im, b[r1].re, a[r2].re * b[r1].im)));
  }
  template <bool ANY = false>
  GL_HD static M staple_fwd(const M& x, const M& y, const M& z) {
    if (ANY) return mul_d(mul_d(x, y), z);
    M p, t;
    dev_row_d<0>(x, y, p);
    dev_row_d<1>(x, y, p);
    dev_row_d<0>(p, z, t);
    dev_row_d<1>(p, z, t);
    third_row<2>(t);
    return t;
  }
  template <bool ANY = false>
  GL_HD static M staple_bwd(const M& x, const M& y, const M& z) {
    if (ANY) return d_mul(mul(x, y), z);
    M p, t;
    dev_col<1>(x, y, p);
    dev_col<2>(x, y, p);
    d_dev_row<1>(p, z, t);
    d_dev_row<2>(p, z, t);
    third_row<0>(t);
    return t;
  }

  // Staple sums c 1 + d (d a full matrix, c the summed weights).
  struct Sum {
    R c;
    M d;
  };
  GL_HD static Sum zero_sum() { return Sum{0.f, G::zero()}; }
  GL_HD static void sum_add(Sum& s, R w, const M& t) {
    s.c += w;
    G::scale_add(s.d, w, t);
  }
  // Im tr t^a (1+u)(c + d) = Im tr t^a (d + u (c + d)): the identity part
  // projects to zero; only the anti-hermitian part of d + u (c + d) is formed.
  // d is close to c u^+, so c u nearly cancels it: that term comes first, and
  // the others round at the size of what is left.
  GL_HD static void proj_mul_sum(const M& u, const Sum& s, R* o) {
    M d1 = s.d;
    d1.m[0].re += s.c;
    d1.m[4].re += s.c;
    d1.m[8].re += s.c;
    cplx<R> p[9];
#pragma unroll
    for (int i = 0; i < 3; ++i)
#pragma unroll
      for (int j = 0; j < 3; ++j) {
        if (i == j) continue;
        const cplx<R> uj = u.m[3 * i + j], dj = d1.m[4 * j];
        cplx<R> acc{fma(uj.re, dj.re, s.d.m[3 * i + j].re), fma(uj.im, dj.re, s.d.m[3 * i + j].im)};
        acc = cplx<R>{fma(-uj.im, dj.im, acc.re), fma(uj.re, dj.im, acc.im)};
        acc = fma_c(u.m[4 * i], d1.m[3 * i + j], acc);
        p[3 * i + j] = fma_c(u.m[3 * i + 3 - i - j], d1.m[3 * (3 - i - j) + j], acc);
      }
    R dg[3];
#pragma unroll
    for (int i = 0; i < 3; ++i) {
      R acc = fma(u.m[4 * i].im, d1.m[4 * i].re, s.d.m[4 * i].im);
      acc = fma(u.m[4 * i].re, d1.m[4 * i].im, acc);
#pragma unroll
      for (int m = 1; m < 3; ++m) {
        const int k = (i + m) % 3;
        acc = fma(u.m[3 * i + k].re, d1.m[3 * k + i].im, acc);
        acc = fma(u.m[3 * i + k].im, d1.m[3 * k + i].re, acc);
      }
      dg[i] = acc;
    }
    o[0] = 0.5f * (p[1].im + p[3].im);
    o[1] = 0.5f * (p[1].re - p[3].re);
    o[2] = 0.5f * (dg[0] - dg[1]);
    o[3] = 0.5f * (p[2].im + p[6].im);
    o[4] = 0.5f * (p[2].re - p[6].re);
    o[5] = 0.5f * (p[5].im + p[7].im);
    o[6] = 0.5f * (p[5].re - p[7].re);
    o[7] = (dg[0] + dg[1] - 2.f * dg[2]) * 0.28867513459481288225f;
  }
  // Same interface for a plain product (1+u) X with X full.
  GL_HD static void proj_mul(const M& u, const M& x, R* o) {
    Sum s{0.f, x};
    proj_mul_sum(u, s, o);
  }
  // Im tr t^a (1+x)(1+y) and Im tr t^a (1+x)(1+y)^+ of two deviations:
  // the staple-sum form with weight 1 and d = y (or y^+), so every
  // rounding stays of the size u |x|, u |y|.
  GL_HD static void proj_prod(const M& x, const M& y, R* o) {
    Sum s{1.f, y};
    proj_mul_sum(x, s, o);
  }
  GL_HD static void proj_prod_d(const M& x, const M& y, R* o) {
    Sum s{1.f, G::dag(y)};
    proj_mul_sum(x, s, o);
  }

  // exp(i c v^a t^a) - 1 by Cayley-Hamilton.  Q = c v^a t^a is hermitian and
  // traceless, so Q^3 = c1 Q + c0 with c1 = tr(Q^2)/2 and c0 = det Q, and
  // every power is Q^n = al_n + be_n Q + ga_n Q^2 with
  //   al_{n+1} = c0 ga_n,  be_{n+1} = al_n + c1 ga_n,  ga_{n+1} = be_n.
  // exp(iQ) - 1 = sum_{n>=1} (i^n/n!) Q^n = f0 + f1 Q + f2 Q^2, summed to
  // n = 9: the remainder is below ||Q||^10/10! < 6e-10 ||Q|| for
  // ||Q||_F <= 1/2.  f0 collects only terms of order ||Q||^3 and up, so
  // nothing of size 1 is formed.  Larger ||Q|| is halved s times first and
  // the result doubled exactly, e_{2h} = 2 e_h + e_h^2.
  GL_HD static M expi(const R* v, R c) {
    R nq2 = 0.f;
#pragma unroll
    for (int a = 0; a < NA; ++a) nq2 += v[a] * v[a];
    R nn = 0.5f * c * c * nq2;  // ||Q||_F^2
    if (all_zero_s(nn)) return G::zero();
    int s = 0;
    R sc = c;
    while (any_gt_s(nn, 0.25f) && s < 40) {
      nn *= 0.25f;
      sc *= 0.5f;
      ++s;
    }
    R cv[NA];
#pragma unroll
    for (int a = 0; a < NA; ++a) cv[a] = sc * v[a];
    const M Q = G::herm(cv);
    // Q^2: real diagonal, upper triangle, lower = conjugate
    R d2[3];
#pragma unroll
    for (int i = 0; i < 3; ++i) {
      R acc = Q.m[4 * i].re * Q.m[4 * i].re;
#pragma unroll
      for (int k = 0; k < 3; ++k)
        if (k != i) acc = fma(Q.m[3 * i + k].re, Q.m[3 * i + k].re, fma(Q.m[3 * i + k].im, Q.m[3 * i + k].im, acc));
      d2[i] = acc;
    }
    const cplx<R> q01 = fma_c(Q.m[2], Q.m[7], fma_c(Q.m[1], Q.m[4], Q.m[0].re * Q.m[1]));
    const cplx<R> q02 = fma_c(Q.m[1], Q.m[5], fma_c(Q.m[2], Q.m[8], Q.m[0].re * Q.m[2]));
    const cplx<R> q12 = fma_c(Q.m[3], Q.m[2], fma_c(Q.m[5], Q.m[8], Q.m[4].re * Q.m[5]));
    const R c1 = 0.5f * (d2[0] + d2[1] + d2[2]);
    // det Q = q00 q11 q22 + 2 Re(Q01 Q12 Q20) - q00 |Q12|^2 - q11 |Q02|^2 - q22 |Q01|^2
    const cplx<R> t = Q.m[1] * Q.m[5];
    R c0 = Q.m[0].re * Q.m[4].re * Q.m[8].re;
    c0 = fma(2.f * t.re, Q.m[2].re, c0);
    c0 = fma(2.f * t.im, Q.m[2].im, c0);
    c0 = fma(-Q.m[0].re, Q.m[5].re * Q.m[5].re + Q.m[5].im * Q.m[5].im, c0);
    c0 = fma(-Q.m[4].re, Q.m[2].re * Q.m[2].re + Q.m[2].im * Q.m[2].im, c0);
    c0 = fma(-Q.m[8].re, Q.m[1].re * Q.m[1].re + Q.m[1].im * Q.m[1].im, c0);
    // series: n = 1 gives i Q; n >= 2 by the recurrence
    R al = 0.f, be = 1.f, ga = 0.f;
    cplx<R> f0{0.f, 0.f}, f1{0.f, 1.f}, f2{0.f, 0.f};
    const float inv_fact[10] = {1.f, 1.f, 0.5f, 1.f / 6.f, 1.f / 24.f, 1.f / 120.f, 1.f / 720.f, 1.f / 5040.f,
                                1.f / 40320.f, 1.f / 362880.f};
#pragma unroll
    for (int n = 2; n <= 9; ++n) {
      const R nal = c0 * ga, nbe = fma(c1, ga, al);
      ga = be;
      al = nal;
      be = nbe;
      const float k = inv_fact[n];
      // i^n: n mod 4 = 0: +1, 1: +i, 2: -1, 3: -i
      if ((n & 3) == 0) {
        f0.re = fma(k, al, f0.re); f1.re = fma(k, be, f1.re); f2.re = fma(k, ga, f2.re);
      } else if ((n & 3) == 1) {
        f0.im = fma(k, al, f0.im); f1.im = fma(k, be, f1.im); f2.im = fma(k, ga, f2.im);
      } else if ((n & 3) == 2) {
        f0.re = fma(-k, al, f0.re); f1.re = fma(-k, be, f1.re); f2.re = fma(-k, ga, f2.re);
      } else {
        f0.im = fma(-k, al, f0.im); f1.im = fma(-k, be, f1.im); f2.im = fma(-k, ga, f2.im);
      }
    }
    M e;
#pragma unroll
    for (int i = 0; i < 3; ++i) {
      const R qd = Q.m[4 * i].re;
      e.m[4 * i] = cplx<R>{fma(f2.re, d2[i], fma(f1.re, qd, f0.re)), fma(f2.im, d2[i], fma(f1.im, qd, f0.im))};
    }
    e.m[1] = fma_c(f2, q01, f1 * Q.m[1]);
    e.m[2] = fma_c(f2, q02, f1 * Q.m[2]);
    e.m[5] = fma_c(f2, q12, f1 * Q.m[5]);
    e.m[3] = fma_c(f2, cj(q01), f1 * Q.m[3]);
    e.m[6] = fma_c(f2, cj(q02), f1 * Q.m[6]);
    e.m[7] = fma_c(f2, cj(q12), f1 * Q.m[7]);
    for (int k = 0; k < s; ++k) {
      const M e2 = G::mul(e, e);
#pragma unroll
      for (int q = 0; q < 9; ++q) e.m[q] = (R)2 * e.m[q] + e2.m[q];
    }
    return e;
  }

  // Re-unitarisation of 1 + d: rows 0 and 1 by Gram-Schmidt, row 2 =
  // conj(row0 x row1), every step written for the deviation from e_k so
  // that no O(1) quantity is formed.
  GL_HD static R inv_sqrt_m1(R eps) {  // 1/sqrt(1+eps) - 1
    // a link one step from the group has |eps| ~ 1e-7: the binomial series
    // -eps/2 + 3 eps^2/8 - 5 eps^3/16 is exact to 35/128 eps^4 there
    if (all_abs_lt_s(eps, 1e-3f)) return eps * fma(eps, fma(eps, R(-0.3125f), R(0.375f)), R(-0.5f));
    const R r = gl_sqrt(R(1.f) + eps);
    return lane_div_s(-eps, r * (R(1.f) + r));
  }
  GL_HD static M reunit(const M& x) {
    M r;
    const cplx<R>* a = &x.m[0];
    R e0 = 2.f * a[0].re;
#pragma unroll
    for (int k = 0; k < 3; ++k) e0 += a[k].re * a[k].re + a[k].im * a[k].im;
    const R g0 = inv_sqrt_m1(e0), f0 = 1.f + g0;
    cplx<R> ap[3];
#pragma unroll
    for (int k = 0; k < 3; ++k) ap[k] = f0 * a[k];
    ap[0].re += g0;
    // row 1 = e1 + b: p = <row0', row1> = b0 + conj(a'_1) + sum conj(a'_k) b_k
    const cplx<R>* b = &x.m[3];
    cplx<R> p = b[0] + cj(ap[1]);
#pragma unroll
    for (int k = 0; k < 3; ++k) p = fma_cj(b[k], ap[k], p);
    cplx<R> bb[3];
#pragma unroll
    for (int k = 0; k < 3; ++k) bb[k] = b[k] - p * ap[k];
    bb[0] = bb[0] - p;
    R e1 = 2.f * bb[1].re;
#pragma unroll
    for (int k = 0; k < 3; ++k) e1 += bb[k].re * bb[k].re + bb[k].im * bb[k].im;
    const R g1 = inv_sqrt_m1(e1), f1 = 1.f + g1;
    cplx<R> bp[3];
#pragma unroll
    for (int k = 0; k < 3; ++k) bp[k] = f1 * bb[k];
    bp[1].re += g1;
    // row 2 - e2 = conj(e0 x b' + a' x e1 + a' x b')
    const cplx<R> c0 = ap[1] * bp[2] - ap[2] * bp[1] - ap[2];
    const cplx<R> c1 = ap[2] * bp[0] - ap[0] * bp[2] - bp[2];
    const cplx<R> c2 = ap[0] * bp[1] - ap[1] * bp[0] + bp[1] + ap[0];
#pragma unroll
    for (int k = 0; k < 3; ++k) {
      r.m[k] = ap[k];
      r.m[3 + k] = bp[k];
    }
    r.m[6] = cj(c0);
    r.m[7] = cj(c1);
    r.m[8] = cj(c2);
    return r;
  }

  // Adjoint transport of an algebra vector (not a small difference: the full
  // link is used).
  template <bool ANY = false> GL_HD static void adj(const M& u, R* q) { G::template adj<ANY>(full(u), q); }
  template <bool ANY = false> GL_HD static void adj_dag(const M& u, R* q) { G::template adj_dag<ANY>(full(u), q); }
  // the re-unitarised exp(i c v^a t^a) u, which takes two rows.  One of them sums
  // its small terms first (dev_dot), with two roundings of its size where mul has
  // six, against those of the staples' derived rows.  Rms error of E after two
  // steps of generic links 2.50e-7 -> 2.45e-7 (2.48e-7 with three rows of every
  // product), after 60 steps 7.09e-7 -> 6.42e-7 (7.12e-7); 512 x 64^2 staged 0.379 ->
  // 0.378 ms, 131 x 45 x 48 staple 0.0652 -> 0.0659.  Both rows: 2.37e-7 and
  // 5.17e-7, but 0.383 and 0.0662 ms.
  GL_HD static M evolve(const R* v, R c, const M& u) {
    const M e = expi(v, c);
    M t = mul(e, u);
    dev_row<1>(e, u, t);
    return reunit(t);
  }
};

template <>
struct LinkAlg<3, float> : LinkAlgDev3<float> {};

// ---------------------------------------------------------------------------
// SU(2), FP32, deviation form: M = (alpha - 1, beta).
// ---------------------------------------------------------------------------
template <typename T>
struct LinkAlgDev2 {
  typedef T R;
  typedef Group<2, T> G;
  typedef typename G::M M;
  static constexpr int NA = 3;
  static constexpr bool kDelta = true;

  GL_HD static M ident() { return G::zero(); }
  GL_HD static M full(const M& d) { return M{{d.a.re + 1.f, d.a.im}, d.b}; }
  GL_HD static M dag(const M& x) { return M{cj(x.a), -x.b}; }
  // alpha = a1 + a2 + a1 a2 - b1 b2*, beta = b1 + b2 + a1 b2 + b1 a2*
  GL_HD static M mul(const M& x, const M& y) {
    return M{x.a + y.a + x.a * y.a - mulc(x.b, y.b), x.b + y.b + x.a * y.b + mulc(x.b, y.a)};
  }
  GL_HD static M mul_d(const M& x, const M& y) { return mul(x, dag(y)); }
  GL_HD static M d_mul(const M& x, const M& y) { return mul(dag(x), y); }
  template <bool ANY = false>
  GL_HD static M staple_fwd(const M& x, const M& y, const M& z) { return mul_d(mul_d(x, y), z); }
  template <bool ANY = false>
  GL_HD static M staple_bwd(const M& x, const M& y, const M& z) { return d_mul(mul(x, y), z); }

  struct Sum {
    R c;
    M d;
  };
  GL_HD static Sum zero_sum() { return Sum{0.f, G::zero()}; }
  GL_HD static void sum_add(Sum& s, R w, const M& t) {
    s.c += w;
    G::scale_add(s.d, w, t);
  }
  // Im tr t^a (1+u)(c + d) = Im tr t^a (c u + d + u d)
  GL_HD static void proj_mul_sum(const M& u, const Sum& s, R* o) {
    M y{s.c * u.a + s.d.a, s.c * u.b + s.d.b};
    R p[NA], q[NA];
    G::proj(y, p);
    G::proj(G::mul(u, s.d), q);
#pragma unroll
    for (int k = 0; k < NA; ++k) o[k] = p[k] + q[k];
  }
  GL_HD static void proj_mul(const M& u, const M& x, R* o) {
    Sum s{0.f, x};
    proj_mul_sum(u, s, o);
  }
  GL_HD static void proj_prod(const M& x, const M& y, R* o) {
    Sum s{1.f, y};
    proj_mul_sum(x, s, o);
  }
  GL_HD static void proj_prod_d(const M& x, const M& y, R* o) {
    Sum s{1.f, dag(y)};
    proj_mul_sum(x, s, o);
  }
  // exp(i c v.sigma/2) - 1 = (cos th - 1 + i sin th n3, sin th (n2 + i n1)),
  // cos th - 1 = -2 sin^2(th/2); by series where th allows, as in reunit (the
  // staple step has few other instructions: 200 x 30 x 20 0.0105 -> 0.0098 ms)
  GL_HD static M expi(const R* v, R c) {
    const R n2 = v[0] * v[0] + v[1] * v[1] + v[2] * v[2];
    if (all_zero_s(n2)) return G::zero();
    const R x = R(0.25f) * c * c * n2;  // th^2: Taylor series up to 1/4 (remainders below 2.5e-11)
    if (all_abs_lt_s(x, 0.25f)) {
      const R co = x * fma(x, fma(x, fma(x, fma(x, R(-1.f / 3628800.f), R(1.f / 40320.f)), R(-1.f / 720.f)),
                                  R(1.f / 24.f)), R(-0.5f));
      const R f = R(0.5f) * c * fma(x, fma(x, fma(x, fma(x, R(1.f / 362880.f), R(-1.f / 5040.f)), R(1.f / 120.f)),
                                           R(-1.f / 6.f)), R(1.f));
      return M{{co, f * v[2]}, {f * v[1], f * v[0]}};
    }
    const R nrm = gl_sqrt(n2);
    R sh, ch;
    gl_sincos(0.25f * c * nrm, &sh, &ch);  // half of th = c |v| / 2
    // a lane whose field is zero while its partner's is not has nrm = 0
    // and v = 0: its factor is set to 0
    const R s = 2.f * sh * ch, f = lane_div0_s(s, nrm);
    return M{{-2.f * sh * sh, f * v[2]}, {f * v[1], f * v[0]}};
  }
  GL_HD static M reunit(const M& x) {
    const R eps = 2.f * x.a.re + x.a.re * x.a.re + x.a.im * x.a.im + x.b.re * x.b.re + x.b.im * x.b.im;
    R g;  // 1 / sqrt(1 + eps) - 1
    if (all_abs_lt_s(eps, 1e-3f)) {
      g = eps * fma(eps, fma(eps, R(-0.3125f), R(0.375f)), R(-0.5f));
    } else {
      const R r = gl_sqrt(R(1.f) + eps);
      g = lane_div_s(-eps, r * (R(1.f) + r));
    }
    const R f = R(1.f) + g;
    return M{{g + f * x.a.re, f * x.a.im}, f * x.b};
  }
  template <bool ANY = false> GL_HD static void adj(const M& u, R* q) { G::template adj<ANY>(full(u), q); }
  template <bool ANY = false> GL_HD static void adj_dag(const M& u, R* q) { G::template adj_dag<ANY>(full(u), q); }
  // the re-unitarised exp(i c v^a t^a) u
  GL_HD static M evolve(const R* v, R c, const M& u) { return reunit(mul(expi(v, c), u)); }
};

template <>
struct LinkAlg<2, float> : LinkAlgDev2<float> {};

}  // namespace glasma
