// SU(2) and SU(3) arithmetic for the Glasma kernels (host+device).
//
// Conventions (Sec. 2 of Ipp & Mueller: traceless hermitian generators):
//   t^a = sigma^a / 2 (SU(2)) or lambda^a / 2 (SU(3)), tr(t^a t^b) = delta/2;
//   an algebra vector v[a] stands for the hermitian matrix sum_a v^a t^a;
//   proj(X)[a] = Im tr(t^a X), the generator projection of the
//   anti-hermitian traceless part of X used by the leapfrog force
//   (Sec. 3, Eq. lattice_1).
//
// SU(2) elements (and real multiples of them, e.g. sums of plaquettes) are
// stored as the complex pair (alpha, beta) of [[alpha, beta], [-beta*, alpha*]].
// SU(3) elements are 3x3 complex matrices, row major.
#pragma once
#include <cuda_runtime.h>
#include <math.h>

#define GL_HD __host__ __device__ __forceinline__

namespace glasma {

template <typename R>
struct cplx {
  R re, im;
};

template <typename R> GL_HD cplx<R> mk(R a, R b) { return cplx<R>{a, b}; }
template <typename R> GL_HD cplx<R> operator+(cplx<R> a, cplx<R> b) { return {a.re + b.re, a.im + b.im}; }
template <typename R> GL_HD cplx<R> operator-(cplx<R> a, cplx<R> b) { return {a.re - b.re, a.im - b.im}; }
template <typename R> GL_HD cplx<R> operator-(cplx<R> a) { return {-a.re, -a.im}; }
template <typename R> GL_HD cplx<R> operator*(cplx<R> a, cplx<R> b) {
  return {a.re * b.re - a.im * b.im, a.re * b.im + a.im * b.re};
}
template <typename R> GL_HD cplx<R> operator*(R s, cplx<R> a) { return {s * a.re, s * a.im}; }
template <typename R> GL_HD cplx<R> cj(cplx<R> a) { return {a.re, -a.im}; }
// a * conj(b)
template <typename R> GL_HD cplx<R> mulc(cplx<R> a, cplx<R> b) {
  return {a.re * b.re + a.im * b.im, a.im * b.re - a.re * b.im};
}
// acc + a*conj(b), four fused multiply-adds
template <typename R> GL_HD cplx<R> fma_cj(cplx<R> a, cplx<R> b, cplx<R> acc) {
  acc.re = fma(a.re, b.re, acc.re);
  acc.re = fma(a.im, b.im, acc.re);
  acc.im = fma(a.im, b.re, acc.im);
  acc.im = fma(-a.re, b.im, acc.im);
  return acc;
}
// acc + a*b
template <typename R> GL_HD cplx<R> fma_c(cplx<R> a, cplx<R> b, cplx<R> acc) {
  acc.re = fma(a.re, b.re, acc.re);
  acc.re = fma(-a.im, b.im, acc.re);
  acc.im = fma(a.re, b.im, acc.im);
  acc.im = fma(a.im, b.re, acc.im);
  return acc;
}

template <typename R> GL_HD R gl_sqrt(R x) { return sqrt(x); }
template <> GL_HD float gl_sqrt<float>(float x) { return sqrtf(x); }
template <typename R> GL_HD void gl_sincos(R x, R* s, R* c) { sincos(x, s, c); }
template <> GL_HD void gl_sincos<float>(float x, float* s, float* c) { sincosf(x, s, c); }

template <int NC, typename R> struct Group;

// ---------------------------------------------------------------------------
// SU(2): (alpha, beta) pair.
// ---------------------------------------------------------------------------
template <typename R>
struct Group<2, R> {
  static constexpr int NA = 3;
  static constexpr int NV = 2;  // complex numbers per stored link
  struct M {
    cplx<R> a, b;
  };
  GL_HD static M ident() { return M{{R(1), R(0)}, {R(0), R(0)}}; }
  GL_HD static M mul(const M& x, const M& y) {
    // [[a1,b1],[-b1*,a1*]] [[a2,b2],[-b2*,a2*]]
    return M{x.a * y.a - mulc(x.b, y.b), x.a * y.b + mulc(x.b, y.a)};
  }
  GL_HD static M dag(const M& x) { return M{cj(x.a), -x.b}; }
  // x * y^dagger
  GL_HD static M mul_d(const M& x, const M& y) { return mul(x, dag(y)); }
  // x^dagger * y
  GL_HD static M d_mul(const M& x, const M& y) { return mul(dag(x), y); }
  GL_HD static void proj(const M& x, R* out) {
    out[0] = x.b.im;  // Im tr(sigma1/2 X)
    out[1] = x.b.re;  // Im tr(sigma2/2 X)
    out[2] = x.a.im;  // Im tr(sigma3/2 X)
  }
  GL_HD static R re_tr(const M& x) { return R(2) * x.a.re; }
  // proj(x y) without forming the unused parts of the product
  GL_HD static void proj_mul(const M& x, const M& y, R* out) { proj(mul(x, y), out); }
  GL_HD static void scale_add(M& acc, R w, const M& x) {
    acc.a = acc.a + w * x.a;
    acc.b = acc.b + w * x.b;
  }
  GL_HD static M zero() { return M{{R(0), R(0)}, {R(0), R(0)}}; }
  // exp(i c sum_a v^a sigma^a/2) - 1 = (cos(th) - 1) + i sin(th) n.sigma,
  // th = c|v|/2.  For th <= 1/2 (every link of a time step and most of the
  // initial state) cos(th) - 1 and sin(th)/th are their Taylor series in
  // th^2, to th^16/16! (remainder below 1e-21): 15 multiply-adds in place of
  // a square root, a sine, a cosine and a division, several times as many
  // operations on the narrow FP64 pipe that bounds the FP64 kernels.
  GL_HD static M expi_m1(const R* v, R c) {
    const R n2 = fma(v[0], v[0], fma(v[1], v[1], v[2] * v[2]));
    const R x = R(0.25) * c * c * n2;  // th^2
    R co, f;                           // cos(th) - 1, sin(th) / |v|
    if (x <= R(0.25)) {
      co = R(1.0 / 20922789888000.0);
      co = fma(co, -x, R(1.0 / 87178291200.0));
      co = fma(co, -x, R(1.0 / 479001600.0));
      co = fma(co, -x, R(1.0 / 3628800.0));
      co = fma(co, -x, R(1.0 / 40320.0));
      co = fma(co, -x, R(1.0 / 720.0));
      co = fma(co, -x, R(1.0 / 24.0));
      co = fma(co, -x, R(0.5));
      co = -x * co;
      f = R(1.0 / 355687428096000.0);
      f = fma(f, -x, R(1.0 / 1307674368000.0));
      f = fma(f, -x, R(1.0 / 6227020800.0));
      f = fma(f, -x, R(1.0 / 39916800.0));
      f = fma(f, -x, R(1.0 / 362880.0));
      f = fma(f, -x, R(1.0 / 5040.0));
      f = fma(f, -x, R(1.0 / 120.0));
      f = fma(f, -x, R(1.0 / 6.0));
      f = R(0.5) * c * fma(f, -x, R(1));
    } else {
      const R nrm = gl_sqrt(n2);
      R s, sh, ch;
      gl_sincos(R(0.25) * c * nrm, &sh, &ch);
      s = R(2) * sh * ch;
      co = R(-2) * sh * sh;
      f = s / nrm;
    }
    return M{{co, f * v[2]}, {f * v[1], f * v[0]}};
  }
  GL_HD static M expi(const R* v, R c) {
    M e = expi_m1(v, c);
    e.a.re += R(1);
    return e;
  }
  // exp(i c v.sigma/2) u
  GL_HD static M evolve(const R* v, R c, const M& u) {
    const M e = expi_m1(v, c);
    return M{fma_c(e.a, u.a, fma_cj(-e.b, u.b, u.a)), fma_c(e.a, u.b, fma_cj(e.b, u.a, u.b))};
  }
  // U = w + i (x, y, z).sigma with alpha = w + i z, beta = y + i x turns
  // the algebra vector: with c = (x, y, z) x q,
  // U q U^+ = |U|^2 q + 2 [(x, y, z) x c - w c], and U^+ q U has w -> -w.
  // half_turn adds the bracket to h: 15 multiply-adds.
  GL_HD static void half_turn(R w, const M& u, const R* q, R* h) {
    const R x = u.b.im, y = u.b.re, z = u.a.im;
    const R c0 = fma(y, q[2], -(z * q[1])), c1 = fma(z, q[0], -(x * q[2])), c2 = fma(x, q[1], -(y * q[0]));
    h[0] = fma(y, c2, fma(-z, c1, fma(-w, c0, h[0])));
    h[1] = fma(z, c0, fma(-x, c2, fma(-w, c1, h[1])));
    h[2] = fma(x, c1, fma(-y, c0, fma(-w, c2, h[2])));
  }
  // for |U| = 1: 18 multiply-adds, where the two matrix products take 32
  GL_HD static void rotate(R w, const M& u, R* q) {
    R h[3] = {R(0), R(0), R(0)};
    half_turn(w, u, q, h);
#pragma unroll
    for (int k = 0; k < 3; ++k) q[k] = fma(R(2), h[k], q[k]);
  }
  // A sum of algebra vectors n + 2 h, and what U q U^+ (DAG: U^+ q U) adds to
  // it for any U: 22 multiply-adds
  struct Acc {
    R n[3], h[3];
  };
  GL_HD static Acc acc(const R* q) { return Acc{{q[0], q[1], q[2]}, {R(0), R(0), R(0)}}; }
  template <bool DAG>
  GL_HD static void conj_add(const M& u, const R* q, Acc& t) {
    const R n = fma(u.a.re, u.a.re, fma(u.a.im, u.a.im, fma(u.b.re, u.b.re, u.b.im * u.b.im)));
    half_turn(DAG ? -u.a.re : u.a.re, u, q, t.h);
#pragma unroll
    for (int k = 0; k < 3; ++k) t.n[k] = fma(n, q[k], t.n[k]);
  }
  GL_HD static void from_acc(const Acc& t, R* q) {
#pragma unroll
    for (int k = 0; k < 3; ++k) q[k] = fma(R(2), t.h[k], t.n[k]);
  }
  template <bool DAG>
  GL_HD static void conj_any(const M& u, R* q) {
    Acc t{{R(0), R(0), R(0)}, {R(0), R(0), R(0)}};
    conj_add<DAG>(u, q, t);
    from_acc(t, q);
  }
  // q <- U^dagger q U and U q U^dagger for U in SU(2); ANY: for any U
  template <bool ANY = false>
  GL_HD static void adj_dag(const M& u, R* q) {
    if (ANY) conj_any<true>(u, q);
    else rotate(-u.a.re, u, q);
  }
  template <bool ANY = false>
  GL_HD static void adj(const M& u, R* q) {
    if (ANY) conj_any<false>(u, q);
    else rotate(u.a.re, u, q);
  }
  GL_HD static M reunit(const M& x) {
    R n2 = x.a.re * x.a.re + x.a.im * x.a.im + x.b.re * x.b.re + x.b.im * x.b.im;
    R f = R(1) / gl_sqrt(n2);
    return M{f * x.a, f * x.b};
  }
  GL_HD static M add(const M& x, const M& y) { return M{x.a + y.a, x.b + y.b}; }
  // squared Frobenius norm of x - y (the 2x2 matrix holds alpha, beta twice)
  GL_HD static R fro2_diff(const M& x, const M& y) {
    cplx<R> da = x.a - y.a, db = x.b - y.b;
    return R(2) * (da.re * da.re + da.im * da.im + db.re * db.re + db.im * db.im);
  }
  // full 2x2 complex matrix element (row r, column c)
  GL_HD static cplx<R> elem(const M& x, int r, int c) {
    if (r == 0) return c == 0 ? x.a : x.b;
    return c == 0 ? -cj(x.b) : cj(x.a);
  }
};

// ---------------------------------------------------------------------------
// SU(3): 3x3 complex, row major.
// ---------------------------------------------------------------------------
template <typename R>
struct Group<3, R> {
  static constexpr int NA = 8;
  static constexpr int NV = 9;
  struct M {
    cplx<R> m[9];
  };
  GL_HD static M ident() {
    M r;
#pragma unroll
    for (int k = 0; k < 9; ++k) r.m[k] = cplx<R>{R(k % 4 == 0 ? 1 : 0), R(0)};
    return r;
  }
  GL_HD static M mul(const M& x, const M& y) {
    M r;
#pragma unroll
    for (int i = 0; i < 3; ++i)
#pragma unroll
      for (int j = 0; j < 3; ++j) {
        cplx<R> acc = x.m[3 * i] * y.m[j];
        acc = fma_c(x.m[3 * i + 1], y.m[3 + j], acc);
        acc = fma_c(x.m[3 * i + 2], y.m[6 + j], acc);
        r.m[3 * i + j] = acc;
      }
    return r;
  }
  // x * y^dagger: (x y^+)_ij = sum_k x_ik conj(y_jk)
  GL_HD static M mul_d(const M& x, const M& y) {
    M r;
#pragma unroll
    for (int i = 0; i < 3; ++i)
#pragma unroll
      for (int j = 0; j < 3; ++j) {
        cplx<R> acc = mulc(x.m[3 * i], y.m[3 * j]);
        acc = fma_cj(x.m[3 * i + 1], y.m[3 * j + 1], acc);
        r.m[3 * i + j] = fma_cj(x.m[3 * i + 2], y.m[3 * j + 2], acc);
      }
    return r;
  }
  // x^dagger * y: sum_k conj(x_ki) y_kj
  GL_HD static M d_mul(const M& x, const M& y) {
    M r;
#pragma unroll
    for (int i = 0; i < 3; ++i)
#pragma unroll
      for (int j = 0; j < 3; ++j) {
        cplx<R> acc = mulc(y.m[j], x.m[i]);
        acc = fma_cj(y.m[3 + j], x.m[3 + i], acc);
        r.m[3 * i + j] = fma_cj(y.m[6 + j], x.m[6 + i], acc);
      }
    return r;
  }
  GL_HD static M dag(const M& x) {
    M r;
#pragma unroll
    for (int i = 0; i < 3; ++i)
#pragma unroll
      for (int j = 0; j < 3; ++j) r.m[3 * i + j] = cj(x.m[3 * j + i]);
    return r;
  }
  GL_HD static M add(const M& x, const M& y) {
    M r;
#pragma unroll
    for (int k = 0; k < 9; ++k) r.m[k] = x.m[k] + y.m[k];
    return r;
  }
  GL_HD static R fro2_diff(const M& x, const M& y) {
    R acc = R(0);
#pragma unroll
    for (int k = 0; k < 9; ++k) {
      cplx<R> d = x.m[k] - y.m[k];
      acc += d.re * d.re + d.im * d.im;
    }
    return acc;
  }
  // Im tr(lambda^a/2 X), Gell-Mann basis
  GL_HD static void proj(const M& x, R* o) {
    const cplx<R>* m = x.m;
    o[0] = R(0.5) * (m[1].im + m[3].im);
    o[1] = R(0.5) * (m[1].re - m[3].re);
    o[2] = R(0.5) * (m[0].im - m[4].im);
    o[3] = R(0.5) * (m[2].im + m[6].im);
    o[4] = R(0.5) * (m[2].re - m[6].re);
    o[5] = R(0.5) * (m[5].im + m[7].im);
    o[6] = R(0.5) * (m[5].re - m[7].re);
    o[7] = (m[0].im + m[4].im - R(2) * m[8].im) * R(0.28867513459481288225);  // 1/(2 sqrt 3)
  }
  GL_HD static R re_tr(const M& x) { return x.m[0].re + x.m[4].re + x.m[8].re; }
  GL_HD static M zero() {
    M r;
#pragma unroll
    for (int k = 0; k < 9; ++k) r.m[k] = cplx<R>{R(0), R(0)};
    return r;
  }
  GL_HD static void scale_add(M& acc, R w, const M& x) {
#pragma unroll
    for (int k = 0; k < 9; ++k) acc.m[k] = acc.m[k] + w * x.m[k];
  }
  // (x y)_ij
  GL_HD static cplx<R> prod_elem(const M& x, const M& y, int i, int j) {
    cplx<R> acc = x.m[3 * i] * y.m[j];
    acc = fma_c(x.m[3 * i + 1], y.m[3 + j], acc);
    return fma_c(x.m[3 * i + 2], y.m[6 + j], acc);
  }
  GL_HD static R prod_diag_im(const M& x, const M& y, int i) {
    R acc = x.m[3 * i].re * y.m[i].im + x.m[3 * i].im * y.m[i].re;
    acc = fma(x.m[3 * i + 1].re, y.m[3 + i].im, acc);
    acc = fma(x.m[3 * i + 1].im, y.m[3 + i].re, acc);
    acc = fma(x.m[3 * i + 2].re, y.m[6 + i].im, acc);
    acc = fma(x.m[3 * i + 2].im, y.m[6 + i].re, acc);
    return acc;
  }
  // proj(x y) from the six off-diagonal and three diagonal imaginary parts
  GL_HD static void proj_mul(const M& x, const M& y, R* o) {
    const cplx<R> p01 = prod_elem(x, y, 0, 1), p10 = prod_elem(x, y, 1, 0);
    const cplx<R> p02 = prod_elem(x, y, 0, 2), p20 = prod_elem(x, y, 2, 0);
    const cplx<R> p12 = prod_elem(x, y, 1, 2), p21 = prod_elem(x, y, 2, 1);
    const R d0 = prod_diag_im(x, y, 0), d1 = prod_diag_im(x, y, 1), d2 = prod_diag_im(x, y, 2);
    o[0] = R(0.5) * (p01.im + p10.im);
    o[1] = R(0.5) * (p01.re - p10.re);
    o[2] = R(0.5) * (d0 - d1);
    o[3] = R(0.5) * (p02.im + p20.im);
    o[4] = R(0.5) * (p02.re - p20.re);
    o[5] = R(0.5) * (p12.im + p21.im);
    o[6] = R(0.5) * (p12.re - p21.re);
    o[7] = (d0 + d1 - R(2) * d2) * R(0.28867513459481288225);
  }
  // hermitian H = sum_a v^a lambda^a / 2
  GL_HD static M herm(const R* v) {
    const R r3 = R(0.57735026918962576451);  // 1/sqrt 3
    M h;
    h.m[0] = cplx<R>{R(0.5) * (v[2] + r3 * v[7]), R(0)};
    h.m[4] = cplx<R>{R(0.5) * (-v[2] + r3 * v[7]), R(0)};
    h.m[8] = cplx<R>{-r3 * v[7], R(0)};
    h.m[1] = cplx<R>{R(0.5) * v[0], R(-0.5) * v[1]};
    h.m[3] = cj(h.m[1]);
    h.m[2] = cplx<R>{R(0.5) * v[3], R(-0.5) * v[4]};
    h.m[6] = cj(h.m[2]);
    h.m[5] = cplx<R>{R(0.5) * v[5], R(-0.5) * v[6]};
    h.m[7] = cj(h.m[5]);
    return h;
  }
  // components 2 Re tr(t^a H) = Re tr(lambda^a H) of a hermitian H
  GL_HD static void from_herm(const M& h, R* v) {
    const R r3 = R(0.57735026918962576451);
    v[0] = h.m[1].re + h.m[3].re;
    v[1] = h.m[3].im - h.m[1].im;
    v[2] = h.m[0].re - h.m[4].re;
    v[3] = h.m[2].re + h.m[6].re;
    v[4] = h.m[6].im - h.m[2].im;
    v[5] = h.m[5].re + h.m[7].re;
    v[6] = h.m[7].im - h.m[5].im;
    v[7] = r3 * (h.m[0].re + h.m[4].re - R(2) * h.m[8].re);
  }
  // The upper triangle of a sum of hermitian matrices 2 q^a t^a, whose entries
  // off the diagonal are the components themselves, and what V q V^+ (V = U, or
  // V = U^+ for DAG) adds to it: rows 0 and 1 of M = V H, H = 2 q^a t^a with a
  // real diagonal (10 multiply-adds per entry), the triangle of M V^+ and its
  // last diagonal entry as a quadratic form of V's third row (28): 136
  // multiply-adds, where two full products take 216.  SU: V in SU(3), so that the
  // trace stays that of H, 0 (t2 is left out): 108.  (The Gauss residual is held
  // to its formula on any links: those of an FP32 state are unitary to their
  // rounding only, and a residual is what differences leave.)
  struct Acc {
    cplx<R> t01, t02, t12;
    R t0, t1, t2;
  };
  GL_HD static Acc acc(const R* q) {
    const R r3 = R(0.57735026918962576451);  // 1/sqrt 3
    return Acc{{q[0], -q[1]}, {q[3], -q[4]}, {q[5], -q[6]}, fma(r3, q[7], q[2]), fma(r3, q[7], -q[2]),
               R(-2) * (r3 * q[7])};
  }
  template <bool DAG, bool SU = false>
  GL_HD static void conj_add(const M& u, const R* q, Acc& t) {
    const Acc H = acc(q);
    const R hd[3] = {H.t0, H.t1, H.t2};
    const cplx<R> h[3] = {H.t01, H.t02, H.t12};
    cplx<R> v[9], m[6];
#pragma unroll
    for (int i = 0; i < 3; ++i)
#pragma unroll
      for (int j = 0; j < 3; ++j) v[3 * i + j] = DAG ? cj(u.m[3 * j + i]) : u.m[3 * i + j];
#pragma unroll
    for (int i = 0; i < 2; ++i)
#pragma unroll
      for (int j = 0; j < 3; ++j) {
        const cplx<R> d = v[3 * i + j];
        cplx<R> s{hd[j] * d.re, hd[j] * d.im};
#pragma unroll
        for (int k = 0; k < 3; ++k) {  // H_kj = conj(H_jk)
          if (k < j) s = fma_c(v[3 * i + k], h[k + j - 1], s);
          if (k > j) s = fma_cj(v[3 * i + k], h[k + j - 1], s);
        }
        m[3 * i + j] = s;
      }
#pragma unroll
    for (int k = 0; k < 3; ++k) {
      t.t01 = fma_cj(m[k], v[3 + k], t.t01);
      t.t02 = fma_cj(m[k], v[6 + k], t.t02);
      t.t12 = fma_cj(m[3 + k], v[6 + k], t.t12);
      t.t0 = fma(m[k].re, v[k].re, fma(m[k].im, v[k].im, t.t0));
      t.t1 = fma(m[3 + k].re, v[3 + k].re, fma(m[3 + k].im, v[3 + k].im, t.t1));
    }
    if (SU) return;
    R s = R(0);
#pragma unroll
    for (int k = 0; k < 3; ++k) {
      const cplx<R> p = mulc(v[k == 2 ? 7 : 6], v[k == 0 ? 7 : 8]);  // of the pairs 01, 02, 12
      s = fma(h[k].re, p.re, fma(-h[k].im, p.im, s));
      t.t2 = fma(hd[k], fma(v[6 + k].re, v[6 + k].re, v[6 + k].im * v[6 + k].im), t.t2);
    }
    t.t2 = fma(R(2), s, t.t2);
  }
  template <bool SU = false>
  GL_HD static void from_acc(const Acc& t, R* q) {
    q[0] = t.t01.re;
    q[1] = -t.t01.im;
    q[2] = R(0.5) * (t.t0 - t.t1);
    q[3] = t.t02.re;
    q[4] = -t.t02.im;
    q[5] = t.t12.re;
    q[6] = -t.t12.im;
    // (t0 + t1 - 2 t2) / (2 sqrt 3); SU: t2 = -t0 - t1
    if (SU) q[7] = R(0.86602540378443864676) * (t.t0 + t.t1);
    else q[7] = R(0.28867513459481288225) * fma(R(-2), t.t2, t.t0 + t.t1);
  }
  template <bool DAG, bool SU>
  GL_HD static void conj_alg(const M& u, R* q) {
    const cplx<R> z{R(0), R(0)};
    Acc t{z, z, z, R(0), R(0), R(0)};
    conj_add<DAG, SU>(u, q, t);
    from_acc<SU>(t, q);
  }
  // q <- U^dagger q U and U q U^dagger for U in SU(3); ANY: for any U
  template <bool ANY = false>
  GL_HD static void adj_dag(const M& u, R* q) { conj_alg<true, !ANY>(u, q); }
  template <bool ANY = false>
  GL_HD static void adj(const M& u, R* q) { conj_alg<false, !ANY>(u, q); }

  // exp(i c v^a t^a) - 1 by Cayley-Hamilton for ||Q||_F <= 1/2, Q = c v^a t^a:
  // Q^3 = c1 Q + c0 with c1 = tr(Q^2)/2 and c0 = det Q, so every power is
  // Q^n = al_n + be_n Q + ga_n Q^2 with al_{n+1} = c0 ga_n, be_{n+1} = al_n +
  // c1 ga_n, ga_{n+1} = be_n, and the series sum_{n>=1} (i^n/n!) Q^n = f0 + f1 Q
  // + f2 Q^2 is summed to n = N: its remainder is below ||Q||^(N+1)/(N+1)!.
  template <int N>
  GL_HD static M expi_series_m1(const M& Q) {
    R d2[3];
#pragma unroll
    for (int i = 0; i < 3; ++i) {
      R acc = Q.m[4 * i].re * Q.m[4 * i].re;
#pragma unroll
      for (int k = 0; k < 3; ++k)
        if (k != i) acc = fma(Q.m[3 * i + k].re, Q.m[3 * i + k].re, fma(Q.m[3 * i + k].im, Q.m[3 * i + k].im, acc));
      d2[i] = acc;
    }
    // the upper triangle of Q^2: Q_ik Q_kj, with the traceless diagonal
    const cplx<R> q01 = fma_c(Q.m[2], Q.m[7], (-Q.m[8].re) * Q.m[1]);
    const cplx<R> q02 = fma_c(Q.m[1], Q.m[5], (-Q.m[4].re) * Q.m[2]);
    const cplx<R> q12 = fma_c(Q.m[3], Q.m[2], (-Q.m[0].re) * Q.m[5]);
    const R c1 = R(0.5) * (d2[0] + d2[1] + d2[2]);
    // det Q = q00 q11 q22 + 2 Re(Q01 Q12 Q20) - q00 |Q12|^2 - q11 |Q02|^2 - q22 |Q01|^2
    const cplx<R> t = Q.m[1] * Q.m[5];
    R c0 = Q.m[0].re * Q.m[4].re * Q.m[8].re;
    c0 = fma(R(2) * t.re, Q.m[2].re, c0);
    c0 = fma(R(2) * t.im, Q.m[2].im, c0);
    c0 = fma(-Q.m[0].re, fma(Q.m[5].re, Q.m[5].re, Q.m[5].im * Q.m[5].im), c0);
    c0 = fma(-Q.m[4].re, fma(Q.m[2].re, Q.m[2].re, Q.m[2].im * Q.m[2].im), c0);
    c0 = fma(-Q.m[8].re, fma(Q.m[1].re, Q.m[1].re, Q.m[1].im * Q.m[1].im), c0);
    R al = R(0), be = R(1), ga = R(0), k = R(1);
    cplx<R> f0{R(0), R(0)}, f1{R(0), R(1)}, f2{R(0), R(0)};
#pragma unroll
    for (int n = 2; n <= N; ++n) {
      const R nal = c0 * ga, nbe = fma(c1, ga, al);
      ga = be;
      al = nal;
      be = nbe;
      k = k / R(n);
      const R sk = (n & 2) ? -k : k;  // i^n: n mod 4 = 0: +1, 1: +i, 2: -1, 3: -i
      if ((n & 1) == 0) {
        f0.re = fma(sk, al, f0.re);
        f1.re = fma(sk, be, f1.re);
        f2.re = fma(sk, ga, f2.re);
      } else {
        f0.im = fma(sk, al, f0.im);
        f1.im = fma(sk, be, f1.im);
        f2.im = fma(sk, ga, f2.im);
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
    return e;
  }

  // exp(i c v^a t^a) - 1.  ||Q||_F <= 1/16 (a time step's links, dt E ~ 0.05)
  // takes 9 terms (remainder below 4.1e-18 ||Q||), ||Q||_F <= 1/2 takes 15
  // (below 2e-18 ||Q||), about 170 and 200 multiply-adds; larger arguments
  // take the eigenvalue form below, whose inverse cosine, square roots,
  // divisions and four sine and cosine pairs are some 600 operations of the
  // FP64 pipe.
  GL_HD static M expi_m1(const R* v, R c) {
    R cv[8];
    R nn = R(0);
#pragma unroll
    for (int a = 0; a < 8; ++a) {
      cv[a] = c * v[a];
      nn = fma(cv[a], cv[a], nn);
    }
    nn *= R(0.5);  // ||Q||_F^2
    if (nn <= R(1.0 / 256.0)) return expi_series_m1<9>(herm(cv));
    if (nn <= R(0.25)) return expi_series_m1<15>(herm(cv));
    M e;
    expi_eigen(cv, &e);
    e.m[0].re -= R(1);
    e.m[4].re -= R(1);
    e.m[8].re -= R(1);
    return e;
  }
  GL_HD static M expi(const R* v, R c) {
    R nn = R(0);
#pragma unroll
    for (int a = 0; a < 8; ++a) nn = fma(c * v[a], c * v[a], nn);
    M e;
    if (R(0.5) * nn <= R(0.25)) {
      e = expi_m1(v, c);
      e.m[0].re += R(1);
      e.m[4].re += R(1);
      e.m[8].re += R(1);
      return e;
    }
    R cv[8];
#pragma unroll
    for (int a = 0; a < 8; ++a) cv[a] = c * v[a];
    expi_eigen(cv, &e);
    return e;
  }
  // exp(i c v^a t^a) u
  GL_HD static M evolve(const R* v, R c, const M& u) {
    const M e = expi_m1(v, c);
    M r;
#pragma unroll
    for (int i = 0; i < 3; ++i)
#pragma unroll
      for (int j = 0; j < 3; ++j) {
        cplx<R> acc = fma_c(e.m[3 * i], u.m[j], u.m[3 * i + j]);
        acc = fma_c(e.m[3 * i + 1], u.m[3 + j], acc);
        r.m[3 * i + j] = fma_c(e.m[3 * i + 2], u.m[6 + j], acc);
      }
    return r;
  }

  // exp(i c H) for H = sum v^a t^a by the Cayley-Hamilton form
  //   exp(iQ) = f0 + f1 Q + f2 Q^2,  Q = c H,
  // with f_j from the eigenvalue parametrisation of Morningstar & Peardon,
  // Phys. Rev. D 69 (2004) 054501, Sec. III: c0 = det Q, c1 = tr(Q^2)/2,
  // theta = acos(c0 / c0max), u = sqrt(c1/3) cos(theta/3),
  // w = sqrt(c1) sin(theta/3); negative c0 by f_j(-c0) = (-1)^j conj f_j(c0).
  // cv = c v.  Not inlined: no link of a time step comes here, and its
  // registers stay out of the step kernels.
  static __host__ __device__ __noinline__ void expi_eigen(const R* cv, M* out) {
    M Q = herm(cv);
    M Q2 = mul(Q, Q);
    R c1 = R(0.5) * (Q2.m[0].re + Q2.m[4].re + Q2.m[8].re);
    // det of the hermitian Q (real)
    cplx<R> d = Q.m[0] * (Q.m[4] * Q.m[8] - Q.m[5] * Q.m[7]) -
                Q.m[1] * (Q.m[3] * Q.m[8] - Q.m[5] * Q.m[6]) +
                Q.m[2] * (Q.m[3] * Q.m[7] - Q.m[4] * Q.m[6]);
    R c0 = d.re;
    bool neg = c0 < R(0);
    if (neg) c0 = -c0;
    R s13 = gl_sqrt(c1 / R(3));
    R c0max = R(2) * s13 * s13 * s13;
    R ratio = c0 / c0max;
    if (ratio > R(1)) ratio = R(1);
    R theta = acos(ratio);
    R st, ct;
    gl_sincos(theta / R(3), &st, &ct);
    R u = s13 * ct;
    R w = gl_sqrt(c1) * st;
    R u2 = u * u, w2 = w * w;
    R xi0;
    if (fabs(w) < R(0.05)) {
      xi0 = R(1) - w2 / R(6) * (R(1) - w2 / R(20) * (R(1) - w2 / R(42)));
    } else {
      R sw, cw_;
      gl_sincos(w, &sw, &cw_);
      xi0 = sw / w;
    }
    R cw, sw_unused;
    gl_sincos(w, &sw_unused, &cw);
    R s2u, c2u, su, cu;
    gl_sincos(R(2) * u, &s2u, &c2u);
    gl_sincos(u, &su, &cu);
    cplx<R> e2iu{c2u, s2u};
    cplx<R> emiu{cu, -su};
    cplx<R> h0 = (u2 - w2) * e2iu +
                 emiu * cplx<R>{R(8) * u2 * cw, R(2) * u * (R(3) * u2 + w2) * xi0};
    cplx<R> h1 = (R(2) * u) * e2iu - emiu * cplx<R>{R(2) * u * cw, -(R(3) * u2 - w2) * xi0};
    cplx<R> h2 = e2iu - emiu * cplx<R>{cw, R(3) * u * xi0};
    R den = R(1) / (R(9) * u2 - w2);
    cplx<R> f0 = den * h0, f1 = den * h1, f2 = den * h2;
    if (neg) {
      f0 = cj(f0);
      f1 = -cj(f1);
      f2 = cj(f2);
    }
    M r;
#pragma unroll
    for (int k = 0; k < 9; ++k) {
      cplx<R> acc = f1 * Q.m[k];
      acc = acc + f2 * Q2.m[k];
      if (k % 4 == 0) acc = acc + f0;
      r.m[k] = acc;
    }
    *out = r;
  }

  // Rows 0, 1 Gram-Schmidt normalised, row 2 = conj(row0 x row1).
  GL_HD static M reunit(const M& x) {
    M r;
    R n0 = R(0);
#pragma unroll
    for (int k = 0; k < 3; ++k) n0 += x.m[k].re * x.m[k].re + x.m[k].im * x.m[k].im;
    R f0 = R(1) / gl_sqrt(n0);
#pragma unroll
    for (int k = 0; k < 3; ++k) r.m[k] = f0 * x.m[k];
    // project row 1 off row 0: p = <row0, row1> = sum conj(r0k) x1k
    cplx<R> p{R(0), R(0)};
#pragma unroll
    for (int k = 0; k < 3; ++k) p = p + mulc(x.m[3 + k], r.m[k]);
    R n1 = R(0);
#pragma unroll
    for (int k = 0; k < 3; ++k) {
      r.m[3 + k] = x.m[3 + k] - p * r.m[k];
      n1 += r.m[3 + k].re * r.m[3 + k].re + r.m[3 + k].im * r.m[3 + k].im;
    }
    R f1 = R(1) / gl_sqrt(n1);
#pragma unroll
    for (int k = 0; k < 3; ++k) r.m[3 + k] = f1 * r.m[3 + k];
    r.m[6] = cj(r.m[1] * r.m[5] - r.m[2] * r.m[4]);
    r.m[7] = cj(r.m[2] * r.m[3] - r.m[0] * r.m[5]);
    r.m[8] = cj(r.m[0] * r.m[4] - r.m[1] * r.m[3]);
    return r;
  }
  GL_HD static cplx<R> elem(const M& x, int r, int c) { return x.m[3 * r + c]; }
};

}  // namespace glasma
