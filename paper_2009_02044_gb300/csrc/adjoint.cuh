// Reverse-mode building blocks of the SU(2) adjoint, FP64.
//
// An SU(2) link [[alpha, beta], [-beta*, alpha*]] is the quaternion
// q = (w, x, y, z) with alpha = w + i z, beta = y + i x, i.e.
// U = w 1 + i (x sigma1 + y sigma2 + z sigma3).  Products, daggers and the
// generator projection Im tr(t^a M) = (x, y, z) are polynomials in these
// four reals, so every step of the forward map is a smooth function of the
// link components; the adjoint differentiates those formulas (extended off
// the group by the same expressions).  Because the forward map keeps links
// on the group, the extension does not change the gradient with respect to
// the initial charges.
//
// Adjoint convention: for a real quantity v, vbar = dO/dv; a quaternion's
// adjoint is the 4-vector of partial derivatives of O with respect to its
// components.
//
// Through the time steps a link's adjoint is kept in its tangent space: the
// three derivatives g = dO/d eta of O under U -> (1 + i eta.sigma) U.  A step
// keeps links on the group, so the fourth (radial) component never matters, and
// every step of the map turns into rotations and cross products of 3-vectors:
// about 510 multiply-adds per site for the plaquettes and 75 per link on the
// FP64 pipe that bounds the reverse pass, against 2350 and 180 for reverse-mode
// products of quaternions.  q_mul(q_pure(g), U) is the quaternion adjoint with
// zero radial part, which the initial state's reverse works on.
#pragma once
#include "glasma_internal.cuh"

namespace glasma {
namespace adj {

struct Q4 {
  double w, x, y, z;
};

GL_HD Q4 q_zero() { return Q4{0.0, 0.0, 0.0, 0.0}; }
GL_HD Q4 q_pure(const double* v) { return Q4{0.0, v[0], v[1], v[2]}; }
GL_HD Q4 q_dag(const Q4& a) { return Q4{a.w, -a.x, -a.y, -a.z}; }
GL_HD void q_acc(Q4& acc, const Q4& a) {
  acc.w += a.w;
  acc.x += a.x;
  acc.y += a.y;
  acc.z += a.z;
}

// (w + i a.s)(v + i b.s) = (w v - a.b) + i (w b + v a - a x b).s
GL_HD Q4 q_mul(const Q4& a, const Q4& b) {
  return Q4{a.w * b.w - (a.x * b.x + a.y * b.y + a.z * b.z),
            a.w * b.x + b.w * a.x - (a.y * b.z - a.z * b.y),
            a.w * b.y + b.w * a.y - (a.z * b.x - a.x * b.z),
            a.w * b.z + b.w * a.z - (a.x * b.y - a.y * b.x)};
}

// reverse of C = A B: abar += dC/dA^T cbar, bbar += dC/dB^T cbar
GL_HD void q_mul_rev(const Q4& a, const Q4& b, const Q4& cb, Q4& ab, Q4& bb) {
  ab.w += b.w * cb.w + b.x * cb.x + b.y * cb.y + b.z * cb.z;
  ab.x += -cb.w * b.x + b.w * cb.x - (b.y * cb.z - b.z * cb.y);
  ab.y += -cb.w * b.y + b.w * cb.y - (b.z * cb.x - b.x * cb.z);
  ab.z += -cb.w * b.z + b.w * cb.z - (b.x * cb.y - b.y * cb.x);
  bb.w += a.w * cb.w + a.x * cb.x + a.y * cb.y + a.z * cb.z;
  bb.x += -cb.w * a.x + a.w * cb.x + (a.y * cb.z - a.z * cb.y);
  bb.y += -cb.w * a.y + a.w * cb.y + (a.z * cb.x - a.x * cb.z);
  bb.z += -cb.w * a.z + a.w * cb.z + (a.x * cb.y - a.y * cb.x);
}

// reverse of D = A^dagger
GL_HD void q_dag_rev(const Q4& db, Q4& ab) {
  ab.w += db.w;
  ab.x -= db.x;
  ab.y -= db.y;
  ab.z -= db.z;
}

GL_HD Q4 q_from(const Group<2, double>::M& m) { return Q4{m.a.re, m.b.im, m.b.re, m.a.im}; }

// link d at site s of an FP64 SU(2) link array ((alpha, beta) as double2)
GL_HD Q4 q_load(const double2* U, int d, int64_t V, int64_t s) {
  const double2 a = U[link_index(2, d, 0, V, s)];
  const double2 b = U[link_index(2, d, 1, V, s)];
  return Q4{a.x, b.y, b.x, a.y};
}

// quaternion adjoints of links: [d][4][V]
GL_HD Q4 qb_load(const double* B, int d, int64_t V, int64_t s) {
  return Q4{B[(int64_t)(d * 4 + 0) * V + s], B[(int64_t)(d * 4 + 1) * V + s], B[(int64_t)(d * 4 + 2) * V + s],
            B[(int64_t)(d * 4 + 3) * V + s]};
}
GL_HD void qb_store(double* B, int d, int64_t V, int64_t s, const Q4& q) {
  B[(int64_t)(d * 4 + 0) * V + s] = q.w;
  B[(int64_t)(d * 4 + 1) * V + s] = q.x;
  B[(int64_t)(d * 4 + 2) * V + s] = q.y;
  B[(int64_t)(d * 4 + 3) * V + s] = q.z;
}

// X = exp(i th.sigma/2) = (cos(r/2), sin(r/2) th / r), r = |th|; thbar +=
// dX/dth^T Xbar:
//   dX0/dth = -(sin(r/2) / (2 r)) th,
//   dXv/dth = g I + (g'(r) / r) th th^T,  g(r) = sin(r/2) / r;
// near r = 0 the Taylor series of the three coefficients is used.
GL_HD void q_expi_rev(const double* th, const Q4& xb, double* thb) {
  const double r2 = th[0] * th[0] + th[1] * th[1] + th[2] * th[2];
  double a0, g, gp;  // sin(r/2)/(2r), g, g'/r
  if (r2 < 1e-6) {
    a0 = 0.25 - r2 / 96.0;
    g = 0.5 - r2 / 48.0;
    gp = -1.0 / 24.0 + r2 / 960.0;
  } else {
    const double r = sqrt(r2);
    const double s = sin(0.5 * r), c = cos(0.5 * r);
    a0 = s / (2.0 * r);
    g = s / r;
    gp = (0.5 * r * c - s) / (r2 * r);
  }
  const double tv = th[0] * xb.x + th[1] * xb.y + th[2] * xb.z;
  thb[0] += -a0 * th[0] * xb.w + g * xb.x + gp * tv * th[0];
  thb[1] += -a0 * th[1] * xb.w + g * xb.y + gp * tv * th[1];
  thb[2] += -a0 * th[2] * xb.w + g * xb.z + gp * tv * th[2];
}

// Reverse of h = kappa(w0, r) wv with kappa = 2 atan2(r, w0) / r (the
// principal SU(2) logarithm, exp(i h.sigma/2) = W):
//   dh/dw0 = -2 wv / (w0^2 + r^2),
//   dh/dwv = kappa I + (dkappa/dr / r) wv wv^T,
//   dkappa/dr / r = 2 [w0 r / (w0^2 + r^2) - atan2(r, w0)] / r^3
// (series -4 / (3 w0^3) + O(r^2) near r = 0).
GL_HD void q_log_rev(const Q4& W, const double* hb, Q4& wb) {
  const double r2 = W.x * W.x + W.y * W.y + W.z * W.z;
  const double n2 = W.w * W.w + r2;
  double kap, kr;
  if (r2 < 1e-12 * W.w * W.w) {
    kap = 2.0 / W.w;
    kr = -4.0 / (3.0 * W.w * W.w * W.w);
  } else {
    const double r = sqrt(r2);
    const double at = atan2(r, W.w);
    kap = 2.0 * at / r;
    kr = 2.0 * (W.w * r / n2 - at) / (r2 * r);
  }
  const double wh = W.x * hb[0] + W.y * hb[1] + W.z * hb[2];
  wb.w += -2.0 * wh / n2;
  wb.x += kap * hb[0] + kr * wh * W.x;
  wb.y += kap * hb[1] + kr * wh * W.y;
  wb.z += kap * hb[2] + kr * wh * W.z;
}

// Reverse of q' = Vec(A (0, q) B) for fixed-shape transports
// (A, B) = (U^dagger, U) or (U, U^dagger): given qbar' returns qbar and
// accumulates the adjoint of U.
GL_HD void transport_rev(const Q4& U, bool dagger_first, const double* q, const double* qpb, double* qb, Q4& ub) {
  const Q4 A = dagger_first ? q_dag(U) : U;
  const Q4 B = dagger_first ? U : q_dag(U);
  const Q4 P = q_pure(q);
  const Q4 p1 = q_mul(A, P);
  const Q4 mb = Q4{0.0, qpb[0], qpb[1], qpb[2]};
  Q4 p1b = q_zero(), bb = q_zero(), ab = q_zero(), pb = q_zero();
  q_mul_rev(p1, B, mb, p1b, bb);
  q_mul_rev(A, P, p1b, ab, pb);
  if (dagger_first) {
    q_dag_rev(ab, ub);
    q_acc(ub, bb);
  } else {
    q_acc(ub, ab);
    q_dag_rev(bb, ub);
  }
  qb[0] = pb.x;
  qb[1] = pb.y;
  qb[2] = pb.z;
}

// ---------------------------------------------------------------------------
// Per-element bodies of the adjoint kernels (host and device, so that the
// same code can be run on the CPU).
// ---------------------------------------------------------------------------

// planes (i, j), i < j: (x, y), (x, z), (y, z)
__host__ __device__ __forceinline__ int plane_i(int pl) { return pl == 2 ? 1 : 0; }
__host__ __device__ __forceinline__ int plane_j(int pl) { return pl == 0 ? 1 : 2; }

GL_HD void cross(const double* a, const double* b, double* c) {
  c[0] = fma(a[1], b[2], -(a[2] * b[1]));
  c[1] = fma(a[2], b[0], -(a[0] * b[2]));
  c[2] = fma(a[0], b[1], -(a[1] * b[0]));
}
// v <- Vec(U (0, v) U^+), v <- Vec(U^+ (0, v) U)
GL_HD void rotate(const Q4& u, double* v) {
  typedef Group<2, double> G;
  G::rotate(u.w, G::M{{0.0, u.z}, {u.y, u.x}}, v);
}
GL_HD void rotate_back(const Q4& u, double* v) { rotate(Q4{-u.w, u.x, u.y, u.z}, v); }

// Per base site x and plane (i, j), i < j, with a = U_i(x), b = U_j(x+i),
// c = U_i(x+j), d = U_j(x) and P = a b c^+ d^+ = p0 + i p.sigma, the
// plaquette's share of
//   phi = fs * sum_links Ebar . F   (F of Sec. 3 Eq. lattice_1)
//       + wsl(iz) * |a b - d c|_F^2 / (a_i a_j)^2   (its energy term).
// The loops at the four corners are P (link a), P^+ (link d), a^+ P a (link b)
// and (d^+ P d)^+ (link c), so with s = -fs [w_j Ebar_i(x) - w_i Ebar_j(x)],
// t4 = Ad_a(-fs w_i Ebar_j(x+i)), t2 = Ad_d(-fs w_j Ebar_i(x+j)) the force part
// is (s + t4 - t2).p, and the energy part is 4 f (1 - p0).  Varying a link
// multiplies P from one side: e.p changes by L(e).eta = (p0 e - p x e).eta from
// the left and by R(e).eta = (p0 e + p x e).eta from the right, which gives
//   g_a = L(s - t2) + R(t4) + 4 f p     g_b = Ad_a^+ [L(s + t4 - t2) + 4 f p]
//   g_d = L(t2) - R(s + t4) - 4 f p     g_c = -Ad_d^+ [R(s + t4 - t2) + 4 f p].
// Writes them to G[((plane*4 + role)*3 + component)*V + s] (zero for absent
// plaquettes).
GL_HD void plaq_rev_at(const double2* U, const double* Eb, double fs, const double* wsl, double* G, const Geom& g,
                       double wt, double wz, double ia2t, double ia2z, int64_t s, int pl) {
  const SiteNbr n = site_nbr(g, s);
  const int i = plane_i(pl), j = plane_j(pl);
  double r[4][3] = {{0, 0, 0}, {0, 0, 0}, {0, 0, 0}, {0, 0, 0}};
  if ((j != 2) || (n.iz <= g.nz - 2)) {
    const Q4 a = q_load(U, i, g.V, s), d = q_load(U, j, g.V, s);
    const Q4 P = q_mul(q_mul(a, q_load(U, j, g.V, n.p[i])), q_dag(q_mul(d, q_load(U, i, g.V, n.p[j]))));
    const double p[3] = {P.x, P.y, P.z};
    const double wi = i == 2 ? wz : wt, wj = j == 2 ? wz : wt;
    double e[3], t4[3], t2[3], pe[3], p4[3], p2[3];
#pragma unroll
    for (int k = 0; k < 3; ++k) {
      e[k] = -fs * (wj * Eb[(int64_t)(i * 3 + k) * g.V + s] - wi * Eb[(int64_t)(j * 3 + k) * g.V + s]);
      t4[k] = -fs * wi * Eb[(int64_t)(j * 3 + k) * g.V + n.p[i]];
      t2[k] = -fs * wj * Eb[(int64_t)(i * 3 + k) * g.V + n.p[j]];
    }
    rotate(a, t4);
    rotate(d, t2);
    cross(p, e, pe);
    cross(p, t4, p4);
    cross(p, t2, p2);
    const double ws = wsl ? wsl[n.iz] : 0.0;
    const double f = 4.0 * ws * (i == 2 || j == 2 ? ia2t * ia2z : ia2t * ia2t);
#pragma unroll
    for (int k = 0; k < 3; ++k) {
      const double fp = f * p[k], se = e[k] - t2[k], ce = pe[k] - p2[k];
      r[0][k] = fma(P.w, se + t4[k], fp) - (ce - p4[k]);
      r[1][k] = fma(P.w, se + t4[k], fp) - (ce + p4[k]);
      r[2][k] = -(fma(P.w, se + t4[k], fp) + (ce + p4[k]));
      r[3][k] = -(fma(P.w, se + t4[k], fp) + (pe[k] + p4[k] + p2[k]));
    }
    rotate_back(a, r[1]);
    rotate_back(d, r[2]);
  }
#pragma unroll
  for (int q = 0; q < 4; ++q)
#pragma unroll
    for (int k = 0; k < 3; ++k) G[(int64_t)((pl * 4 + q) * 3 + k) * g.V + s] = r[q][k];
}

GL_HD void g_add(const double* G, int pl, int role, int64_t V, int64_t s, double* acc) {
  const double* gp = G + (int64_t)((pl * 4 + role) * 3) * V + s;
  acc[0] += gp[0];
  acc[1] += gp[V];
  acc[2] += gp[2 * V];
}

// acc += the parts of the four plaquettes that hold link (x, d): as a (base
// x) and c (base x - j) when d is the plane's first direction, as d (base x)
// and b (base x - i) when it is the second.
GL_HD void gather_at(const double* G, const Geom& g, int d, const SiteNbr& n, double* acc) {
  for (int pl = 0; pl < 3; ++pl) {
    const int i = plane_i(pl), j = plane_j(pl);
    if (d == i) {
      g_add(G, pl, 0, g.V, n.s, acc);
      if (j != 2 || n.iz >= 1) g_add(G, pl, 2, g.V, n.m[j], acc);
    } else if (d == j) {
      g_add(G, pl, 3, g.V, n.s, acc);
      g_add(G, pl, 1, g.V, n.m[i], acc);
    }
  }
}

// g[(d*3 + k)*V + s]: tangent adjoints of the links
GL_HD void tan_load(const double* T, int d, int64_t V, int64_t s, double* v) {
#pragma unroll
  for (int k = 0; k < 3; ++k) v[k] = T[(int64_t)(d * 3 + k) * V + s];
}
GL_HD void tan_store(double* T, int d, int64_t V, int64_t s, const double* v) {
#pragma unroll
  for (int k = 0; k < 3; ++k) T[(int64_t)(d * 3 + k) * V + s] = v[k];
}

// The tangent adjoints T plus the plaquettes' parts G as quaternion adjoints
// of the links (radial part zero).
GL_HD void tangent_to_quat_at(const double2* U, const double* T, const double* G, double* Ub, const Geom& g, int d,
                              int64_t s) {
  const SiteNbr n = site_nbr(g, s);
  double v[3] = {0.0, 0.0, 0.0};
  if (d != 2 || n.iz != g.nz - 1) {
    tan_load(T, d, g.V, s, v);
    gather_at(G, g, d, n, v);
  }
  qb_store(Ub, d, g.V, s, q_mul(q_pure(v), q_load(U, d, g.V, s)));
}

struct LinkRevArgs {
  const double2* U;   // U_n
  const double* En;   // E_{n+1/2}
  const double* G;    // plaquettes' parts of the adjoint of U_{n+1}
  double* T;          // in: the rest of it; out: adjoint of U_n before the force part
  double* Eb;         // adjoint of E_{n+1/2} (in and out)
  const double* QA;   // charges at step n (before the hop)
  const double* QB;
  double* QAb;        // in: adjoint after the hop; out: before
  double* QBb;
  int hop, zA0, WA, zB0, WB;
  Geom g;
  double dt, az2;
};

// For X = exp(i th.sigma/2), r = |th|, x = r^2: A = sin(r) / (2 r),
// B = (1 - cos r) / (2 x), C = (1 - sin(r) / r) / (2 x), by their series for
// r <= 1 (remainders below 1e-18).
GL_HD void expi_coeffs(double x, double& A, double& B, double& C) {
  if (x <= 1.0) {
    double a = 0.0, b = 0.0;
    // 1 / (2 (2k+1)!) and 1 / (2 (2k+2)!): A from k = 0, C from k = 1
    const double fa[10] = {0.5, 1.0 / 12.0, 1.0 / 240.0, 1.0 / 10080.0, 1.0 / 725760.0, 1.0 / 79833600.0,
                           1.0 / 12454041600.0, 1.0 / 2615348736000.0, 1.0 / 711374856192000.0,
                           1.0 / 243290200817664000.0};
    const double fb[9] = {0.25, 1.0 / 48.0, 1.0 / 1440.0, 1.0 / 80640.0, 1.0 / 7257600.0, 1.0 / 958003200.0,
                          1.0 / 174356582400.0, 1.0 / 41845579776000.0, 1.0 / 12804747411456000.0};
#pragma unroll
    for (int k = 9; k >= 1; --k) a = fma(-x, a, fa[k]);
#pragma unroll
    for (int k = 8; k >= 0; --k) b = fma(-x, b, fb[k]);
    C = a;
    A = fma(-x, a, 0.5);
    B = b;
  } else {
    const double r = sqrt(x), sh = sin(0.5 * r);
    A = sin(r) / (2.0 * r);
    B = sh * sh / x;
    C = (0.5 - A) / x;
  }
}

// Reverse of U_{n+1} = X U_n, X = exp(i th.sigma/2), th = dt E_{n+1/2}: a
// change of U_n turns with X, and of E enters through the derivative of the
// exponential, delta X = i xi.sigma X with xi = A dth + B dth x th +
// C (th.dth) th.  On hop steps the charge transport and the current on the z
// links:
//   B: Q'_B = Vec(U^+ (0, Q_B) U) at the slot of x, E_z(x) -= a_z^2 Q_B;
//   A: Q'_A = Vec(U (0, Q_A) U^+) at the slot of x + z, E_z(x) += a_z^2 Q'_A.
GL_HD void link_rev_at(const LinkRevArgs& a, int d, int64_t s) {
  const Geom& g = a.g;
  const SiteNbr n = site_nbr(g, s);
  const int iz = n.iz;
  if (d == 2 && iz == g.nz - 1) {  // absent link: no field, no adjoint
    for (int k = 0; k < 3; ++k) a.Eb[(int64_t)(6 + k) * g.V + s] = 0.0;
    return;
  }
  double th[3], t[3], tx[3], u[3], eb[3];
#pragma unroll
  for (int k = 0; k < 3; ++k) th[k] = a.dt * a.En[(int64_t)(d * 3 + k) * g.V + s];
  tan_load(a.T, d, g.V, s, t);
  gather_at(a.G, g, d, n, t);
  const double x = fma(th[0], th[0], fma(th[1], th[1], th[2] * th[2]));
  const double tt = fma(th[0], t[0], fma(th[1], t[1], th[2] * t[2]));
  double A, B, C;
  expi_coeffs(x, A, B, C);
  cross(th, t, tx);
#pragma unroll
  for (int k = 0; k < 3; ++k) {
    u[k] = fma(2.0, fma(A, tx[k], B * fma(tt, th[k], -(x * t[k]))), t[k]);
    eb[k] = fma(a.dt, fma(A, t[k], fma(B, tx[k], C * tt * th[k])), a.Eb[(int64_t)(d * 3 + k) * g.V + s]);
    a.Eb[(int64_t)(d * 3 + k) * g.V + s] = eb[k];
  }
  if (d == 2 && a.hop) {
    const int64_t tr = s - (int64_t)iz * g.nxy;
    const int kb = iz - a.zB0, ka = iz + 1 - a.zA0;
    const bool inb = kb >= 0 && kb < a.WB, ina = ka >= 0 && ka < a.WA;
    if (inb || ina) {
      const Q4 q4 = q_load(a.U, 2, g.V, s);
      double q[3], qb[3], c[3];
      if (inb) {
        for (int k = 0; k < 3; ++k) {
          q[k] = a.QB[((int64_t)k * a.WB + kb) * g.nxy + tr];
          qb[k] = a.QBb[((int64_t)k * a.WB + kb) * g.nxy + tr];
        }
        rotate(q4, qb);
        cross(q, qb, c);
        for (int k = 0; k < 3; ++k) {
          u[k] = fma(2.0, c[k], u[k]);
          a.QBb[((int64_t)k * a.WB + kb) * g.nxy + tr] = qb[k] - a.az2 * eb[k];
        }
      }
      if (ina) {
        for (int k = 0; k < 3; ++k) {
          q[k] = a.QA[((int64_t)k * a.WA + ka) * g.nxy + tr];
          qb[k] = a.QAb[((int64_t)k * a.WA + ka) * g.nxy + tr] + a.az2 * eb[k];
        }
        rotate(q4, q);
        cross(q, qb, c);
        rotate_back(q4, qb);
        for (int k = 0; k < 3; ++k) {
          u[k] = fma(-2.0, c[k], u[k]);
          a.QAb[((int64_t)k * a.WA + ka) * g.nxy + tr] = qb[k];
        }
      }
    }
  }
  tan_store(a.T, d, g.V, s, u);
}

// The current part of the observable's own E update (no transported-charge
// adjoint): E'_z(x) += a_z^2 (Q'_A - Q_B) with adjoint Ebp_z(x); T holds the
// tangent adjoints of the links.
GL_HD void hop_current_rev_at(const double2* U, const double* Ebp, const double* QA, const double* QB, double* QAb,
                              double* QBb, double* T, int zA0, int WA, int zB0, int WB, const Geom& g, double az2,
                              int64_t s) {
  const int iz = (int)(s / g.nxy);
  const int64_t t = s - (int64_t)iz * g.nxy;
  double eb[3];
  for (int k = 0; k < 3; ++k) eb[k] = Ebp[(int64_t)(6 + k) * g.V + s];
  const int kb = iz - zB0;
  if (kb >= 0 && kb < WB)
    for (int k = 0; k < 3; ++k) QBb[((int64_t)k * WB + kb) * g.nxy + t] -= az2 * eb[k];
  const int ka = iz + 1 - zA0;
  if (ka >= 0 && ka < WA) {
    const Q4 u = q_load(U, 2, g.V, s);
    double q[3], qb[3], c[3], v[3];
    for (int k = 0; k < 3; ++k) {
      q[k] = QA[((int64_t)k * WA + ka) * g.nxy + t];
      qb[k] = az2 * eb[k];
    }
    rotate(u, q);
    cross(q, qb, c);
    rotate_back(u, qb);
    tan_load(T, 2, g.V, s, v);
    for (int k = 0; k < 3; ++k) v[k] = fma(-2.0, c[k], v[k]);
    tan_store(T, 2, g.V, s, v);
    for (int k = 0; k < 3; ++k) QAb[((int64_t)k * WA + ka) * g.nxy + t] += qb[k];
  }
}

// Direct energy terms of the observable: eps holds (1/4) sum_i (E_i^2 +
// E'_i^2) / a_i^2 per site, E' = E(n+1/2) from the non-committing update:
//   Ebp = w(iz) E' / (2 a_i^2) (adjoint of E'), Eb = w(iz) E / (2 a_i^2) + Ebp
// with w(iz) the slice weight a_z / (nx ny) inside the window.
GL_HD void obs_rev_at(const double* E, const double* Ep, const double* wsl, double* Eb, double* Ebp, const Geom& g,
                      double ia2t, double ia2z, int64_t idx) {
  {
    const int comp = (int)(idx / g.V);
    const int64_t s = idx - (int64_t)comp * g.V;
    const int d = comp / 3;
    const double w = wsl[s / g.nxy] * 0.5 * (d == 2 ? ia2z : ia2t);
    const double bp = w * Ep[idx];
    Ebp[idx] = bp;
    Eb[idx] = w * E[idx] + bp;
  }
}

// Adjoint of the charge density rho(x) = sum_i [E_i(x) - T_i(x)] / a_i^2,
// T_i(x) = Vec(U_i^+(x-i) (0, E_i(x-i)) U_i(x-i)), through the split
// Q_A = rho (z > z_c), Q_B = rho (z < z_c) read from the windows; only the
// transverse links and fields depend on the charges (U_z = 1, E_z = 0).
GL_HD void rho_bar(const double* QAb, const double* QBb, int zA0, int WA, int zB0, int WB,
                                        const Geom& g, int iz, int64_t t, double* out) {
  for (int k = 0; k < 3; ++k) out[k] = 0.0;
  const int ka = iz - zA0, kb = iz - zB0;
  if (ka >= 0 && ka < WA)
    for (int k = 0; k < 3; ++k) out[k] += QAb[((int64_t)k * WA + ka) * g.nxy + t];
  if (kb >= 0 && kb < WB)
    for (int k = 0; k < 3; ++k) out[k] += QBb[((int64_t)k * WB + kb) * g.nxy + t];
}

GL_HD void div_rev_at(const double2* U, const double* E, const double* QAb, const double* QBb, int zA0, int WA,
                      int zB0, int WB, double* Eb, double* Ub, const Geom& g, double ia2t, int64_t s) {
  {
    const SiteNbr n = site_nbr(g, s);
    const int64_t t = s - (int64_t)n.iz * g.nxy;
    double r0[3];
    rho_bar(QAb, QBb, zA0, WA, zB0, WB, g, n.iz, t, r0);
    for (int d = 0; d < 2; ++d) {
      const int64_t sp = n.p[d];
      double r1[3], q[3], qpb[3], qb[3];
      rho_bar(QAb, QBb, zA0, WA, zB0, WB, g, n.iz, sp - (int64_t)n.iz * g.nxy, r1);
      for (int k = 0; k < 3; ++k) {
        q[k] = E[(int64_t)(d * 3 + k) * g.V + s];
        qpb[k] = -ia2t * r1[k];
      }
      Q4 ub = qb_load(Ub, d, g.V, s);
      transport_rev(q_load(U, d, g.V, s), true, q, qpb, qb, ub);
      qb_store(Ub, d, g.V, s, ub);
      for (int k = 0; k < 3; ++k) Eb[(int64_t)(d * 3 + k) * g.V + s] += ia2t * r0[k] + qb[k];
    }
  }
}

// Links of the initial state rebuilt exactly as the forward builds them.
GL_HD Group<2, double>::M vdag_of(const double* phi, int N, int64_t nxy, int64_t t, double lam) {
  typedef Group<2, double> G;
  if (lam == 0.0) return G::ident();
  double v[3];
  for (int a = 0; a < 3; ++a) v[a] = phi[((int64_t)N * 3 + a) * nxy + t];
  return G::expi(v, lam);
}

GL_HD Group<2, double>::M link_of(const double* phi, double la, double lb, int64_t nxy,
                                                        int64_t t0, int64_t t1) {
  typedef Group<2, double> G;
  const G::M ua = G::d_mul(vdag_of(phi, 0, nxy, t0, la), vdag_of(phi, 0, nxy, t1, la));
  const G::M ub = G::d_mul(vdag_of(phi, 1, nxy, t0, lb), vdag_of(phi, 1, nxy, t1, lb));
  return G::mul(ua, ub);
}

// E_i = log(U0 Um^+) / dt on transverse links (zero where the two links are
// bitwise equal, as in the forward): Ub (adjoint of U0) += ..., Umb = ...
GL_HD void log_rev_at(const double* phi, const double* lam, const double* Eb, double* Ub, double* Umb, const Geom& g,
                      double dt, int64_t idx) {
  typedef Group<2, double> G;
  {
    const int d = (int)(idx / g.V);
    const int64_t s = idx - (int64_t)d * g.V;
    const SiteNbr n = site_nbr(g, s);
    const int64_t t0 = s % g.nxy, t1 = n.p[d] % g.nxy;
    const G::M u0 = link_of(phi, lam[0 * g.nz + n.iz], lam[1 * g.nz + n.iz], g.nxy, t0, t1);
    const G::M um = link_of(phi, lam[2 * g.nz + n.iz], lam[3 * g.nz + n.iz], g.nxy, t0, t1);
    Q4 mb = q_zero();
    const bool same = u0.a.re == um.a.re && u0.a.im == um.a.im && u0.b.re == um.b.re && u0.b.im == um.b.im;
    if (!same) {
      const Q4 a = q_from(u0), b = q_dag(q_from(um));
      const Q4 W = q_mul(a, b);
      double hb[3];
      for (int k = 0; k < 3; ++k) hb[k] = Eb[(int64_t)(d * 3 + k) * g.V + s] / dt;
      Q4 wb = q_zero(), a_b = qb_load(Ub, d, g.V, s), bdb = q_zero();
      q_log_rev(W, hb, wb);
      q_mul_rev(a, b, wb, a_b, bdb);
      qb_store(Ub, d, g.V, s, a_b);
      q_dag_rev(bdb, mb);
    }
    qb_store(Umb, d, g.V, s, mb);
  }
}

// For site x and nucleus N: the adjoint of V_N^+(x) at both times from the
// links (x, i) (as V_N(x) = (V_N^+(x))^+) and (x - i, i) (as V_N^+(x)),
// i = x, y, then through V^+ = exp(i Lambda phi.sigma/2):
//   phib_z[(N*3 + a)*V + s] = sum_t Lambda_N(z, t) thbar^a.
GL_HD void links_rev_at(const double* phi, const double* lam, const double* Ub, const double* Umb, double* phib_z,
                        const Geom& g, int64_t s) {
  {
    const SiteNbr n = site_nbr(g, s);
    const int64_t tx = s % g.nxy;
    double acc[2][3] = {{0.0, 0.0, 0.0}, {0.0, 0.0, 0.0}};
    for (int tm = 0; tm < 2; ++tm) {
      const double la = lam[(tm * 2 + 0) * g.nz + n.iz], lb = lam[(tm * 2 + 1) * g.nz + n.iz];
      const double* B = tm == 0 ? Ub : Umb;
      const double lamN[2] = {la, lb};
      Q4 vb[2] = {q_zero(), q_zero()};
      for (int i = 0; i < 2; ++i) {
        for (int side = 0; side < 2; ++side) {  // 0: link (x, i); 1: link (x - i, i)
          const int64_t y = side == 0 ? s : n.m[i];
          const int64_t ty = y % g.nxy;
          const SiteNbr ny_ = site_nbr(g, y);
          const int64_t tyi = ny_.p[i] % g.nxy;
          Q4 v0[2], v1[2];
          for (int N = 0; N < 2; ++N) {
            v0[N] = q_from(vdag_of(phi, N, g.nxy, ty, lamN[N]));
            v1[N] = q_from(vdag_of(phi, N, g.nxy, tyi, lamN[N]));
          }
          const Q4 ua = q_mul(q_dag(v0[0]), v1[0]);
          const Q4 ubq = q_mul(q_dag(v0[1]), v1[1]);
          const Q4 lb_ = qb_load(B, i, g.V, y);
          Q4 uab = q_zero(), ubb = q_zero();
          q_mul_rev(ua, ubq, lb_, uab, ubb);
          const Q4 fb[2] = {uab, ubb};
          for (int N = 0; N < 2; ++N) {
            Q4 v0db = q_zero(), v1b = q_zero();
            q_mul_rev(q_dag(v0[N]), v1[N], fb[N], v0db, v1b);
            if (side == 0)
              q_dag_rev(v0db, vb[N]);
            else
              q_acc(vb[N], v1b);
          }
        }
      }
      for (int N = 0; N < 2; ++N) {
        if (lamN[N] == 0.0) continue;
        double th[3], thb[3] = {0.0, 0.0, 0.0};
        for (int a = 0; a < 3; ++a) th[a] = lamN[N] * phi[((int64_t)N * 3 + a) * g.nxy + tx];
        q_expi_rev(th, vb[N], thb);
        for (int a = 0; a < 3; ++a) acc[N][a] += lamN[N] * thb[a];
      }
    }
    for (int N = 0; N < 2; ++N)
      for (int a = 0; a < 3; ++a) phib_z[(int64_t)(N * 3 + a) * g.V + s] = acc[N][a];
  }
}

GL_HD void zsum_at(const double* phib_z, double* phib, const Geom& g, int64_t idx) {
  {
    const int64_t f = idx / g.nxy, t = idx - f * g.nxy;
    double acc = 0.0;
    for (int iz = 0; iz < g.nz; ++iz) acc += phib_z[f * g.V + (int64_t)iz * g.nxy + t];
    phib[idx] = acc;
  }
}


}  // namespace adj
}  // namespace glasma
