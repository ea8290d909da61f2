// MV initial state on the device (Sec. 2 MV model; Sec. 3 Eqs. single_sheet,
// 3d_colorfield_1, 3d_colorfield_2; Sec. 4 Gaussian profile), all in FP64:
//   rho_N^a(x_T)   Philox4x32-10 + Box-Muller, or copied from the host
//   phi_N          (-Delta_T + m^2)^{-1} rho_N by separable DFTs
//   Lambda_N(z,t)  cumulative truncated Gaussian profile (erf)
//   U_i(x; t)      V_A(x) V_A^dag(x+i) V_B(x) V_B^dag(x+i), U_z = 1,
//                  V_N^dag = exp(i Lambda_N phi_N), at t0 and t0 - dt
//   E_i            -i log(U(t0) U^dag(t0 - dt)) / dt, 0 where equal
//   rho(x)         discrete Gauss divergence of the stored state
//   Q_A, Q_B       rho on either side of the box centre, cut to windows
#include <vector>

#include "glasma_internal.cuh"
#include "init_math.cuh"

namespace glasma {

// rho[(s*2 + N)*na + a][y][x] for S sheets; counter (x, y, a, N + 2 s)
__global__ void k_philox_rho(double* rho, int na, int nx, int ny, int S, unsigned long long seed, double g2mu) {
  const int64_t total = (int64_t)2 * S * na * nx * ny;
  for (int64_t i = (int64_t)blockIdx.x * blockDim.x + threadIdx.x; i < total; i += (int64_t)gridDim.x * blockDim.x) {
    const int x = (int)(i % nx);
    int64_t r = i / nx;
    const int y = (int)(r % ny);
    r /= ny;
    const int a = (int)(r % na);
    const int N = (int)(r / na);  // N + 2 s
    uint32_t c[4] = {(uint32_t)x, (uint32_t)y, (uint32_t)a, (uint32_t)N};
    philox4x32_10(c, (uint32_t)(seed & 0xFFFFFFFFull), (uint32_t)(seed >> 32));
    const double u1 = u53(c[0], c[1]), u2 = u53(c[2], c[3]);
    rho[i] = g2mu * (sqrt(-2.0 * log(u1)) * cospi(2.0 * u2));
  }
}

// The transverse Poisson solve phi = ifft(fft(rho) / (k^2 + m^2)) of F real
// [ny][nx] fields by separable DFTs.  The fields are real and the kernel even,
// so only the columns kx = 0..nx/2 are transformed, the first pass takes real
// input and the last gives real output: (1 + 2 + 2 + 1) n multiply-adds per
// site where four full complex passes take 16 n.  The factors exp(2 pi i j / n)
// come from a table: evaluating sincospi in the inner loop cost 30 times as
// much (0.45 ms per pass of the SU(3) 64^2 fields, 1.29 ms of the SU(2) 128^2
// ones).
__global__ void k_twiddle(double2* tw, int nx, int ny) {
  for (int i = blockIdx.x * blockDim.x + threadIdx.x; i < nx + ny; i += gridDim.x * blockDim.x) {
    const int n = i < nx ? nx : ny, j = i < nx ? i : i - nx;
    double s, c;
    sincospi(2.0 * (double)j / (double)n, &s, &c);
    tw[i] = make_double2(c, s);
  }
}

// out[f][y][kx] = sum_x in[f][y][x] exp(-2 pi i kx x / nx), kx < nh
__global__ void k_dft_x(const double* in, double2* out, const double2* tw, int64_t rows, int nx, int nh) {
  for (int64_t i = (int64_t)blockIdx.x * blockDim.x + threadIdx.x; i < rows * nh; i += (int64_t)gridDim.x * blockDim.x) {
    const int k = (int)(i % nh);
    const double* row = in + (i / nh) * nx;
    double re = 0.0, im = 0.0;
    for (int m = 0, km = 0; m < nx; ++m) {
      const double v = row[m];
      const double2 w = tw[km];
      re = fma(v, w.x, re);
      im = fma(-v, w.y, im);
      km += k;
      if (km >= nx) km -= nx;
    }
    out[i] = make_double2(re, im);
  }
}

// out[f][k][kx] = sum_y in[f][y][kx] exp(sign 2 pi i k y / ny), times the
// Poisson kernel 1 / (k^2 + m^2), k^2 = 4/a^2 [sin^2(pi kx/nx) + sin^2(pi ky/ny)]
// in the forward pass (sign = -1)
__global__ void k_dft_y(const double2* in, double2* out, const double2* tw, int F, int ny, int nx, int nh, int sign,
                        double a_t, double m2, double uv2) {
  const int64_t total = (int64_t)F * ny * nh;
  for (int64_t i = (int64_t)blockIdx.x * blockDim.x + threadIdx.x; i < total; i += (int64_t)gridDim.x * blockDim.x) {
    const int kx = (int)(i % nh);
    const int64_t r = i / nh;
    const int k = (int)(r % ny);
    const double2* col = in + (r / ny) * ny * nh + kx;
    double re = 0.0, im = 0.0;
    for (int m = 0, km = 0; m < ny; ++m) {
      const double2 v = col[(int64_t)m * nh], w = tw[km];
      const double s = sign * w.y;
      re = fma(v.x, w.x, fma(-v.y, s, re));
      im = fma(v.x, s, fma(v.y, w.x, im));
      km += k;
      if (km >= ny) km -= ny;
    }
    if (sign < 0) {
      const double sx = sinpi((double)kx / nx), sy = sinpi((double)k / ny);
      const double k2 = 4.0 / (a_t * a_t) * (sy * sy) + 4.0 / (a_t * a_t) * (sx * sx);
      double kern = 1.0 / (k2 + m2);
      if (uv2 > 0.0 && k2 > uv2) kern = 0.0;
      re *= kern;
      im *= kern;
    }
    out[i] = make_double2(re, im);
  }
}

// out[f][y][x] = scale Re sum_kx in[f][y][kx] exp(2 pi i kx x / nx) over all
// nx columns, those above nx/2 the conjugates of the kept ones
__global__ void k_dft_x_real(const double2* in, double* out, const double2* tw, int64_t rows, int nx, int nh,
                             double scale) {
  for (int64_t i = (int64_t)blockIdx.x * blockDim.x + threadIdx.x; i < rows * nx; i += (int64_t)gridDim.x * blockDim.x) {
    const int x = (int)(i % nx);
    const double2* row = in + (i / nx) * nh;
    double acc = 0.0;
    for (int k = 1, kx = x; 2 * k < nx; ++k) {
      const double2 v = row[k], w = tw[kx];
      acc = fma(v.x, w.x, fma(-v.y, w.y, acc));
      kx += x;
      if (kx >= nx) kx -= nx;
    }
    acc = fma(2.0, acc, row[0].x);
    if (nx % 2 == 0) acc += (x & 1) ? -row[nx / 2].x : row[nx / 2].x;
    out[i] = acc * scale;
  }
}

// lam[(t*2 + N)*nz + iz], t = 0: t0, 1: t0 - dt; N = 0: A, 1: B
// (iz is local: the slice's global index is iz + zoff)
__global__ void k_profile(double* lam, int nz, int zoff, double a_z, double sigma, double zA0, double zB0,
                          double dt) {
  const double erf4 = erf(2.0 * 1.4142135623730950488);  // erf(4 / sqrt 2)
  for (int i = blockIdx.x * blockDim.x + threadIdx.x; i < 4 * nz; i += gridDim.x * blockDim.x) {
    const int iz = i % nz, tn = i / nz, N = tn % 2, t = tn / 2;
    const double z = (iz + zoff) * a_z;
    const double zn = N == 0 ? zA0 + (t ? dt : 0.0) : zB0 - (t ? dt : 0.0);
    const double u = (z - zn) / sigma;
    const double uc = fmin(fmax(u, -4.0), 4.0);
    const double ef = erf(uc / 1.4142135623730950488);
    double L;
    if (N == 1) {  // B, moving +z: 1 behind (low z), 0 ahead
      L = (erf4 - ef) / (2.0 * erf4);
      if (u >= 4.0) L = 0.0;
      if (u <= -4.0) L = 1.0;
    } else {  // A, moving -z: 1 behind (high z), 0 ahead
      L = (ef + erf4) / (2.0 * erf4);
      if (u <= -4.0) L = 0.0;
      if (u >= 4.0) L = 1.0;
    }
    lam[i] = L;
  }
}

// V_N^dagger at transverse site t for the cumulative profile value lam.
// One sheet: exp(i lam phi_N).  S sheets (phi[(s*2 + N)*na + a][t]): the
// path-ordered exp(i L_{S-1} phi_{S-1,N}) ... exp(i L_0 phi_{0,N}) with
// L_s = clip(S lam - s, 0, 1), sheet 0 (the leading slab) acting first.
template <int NC>
GL_HD typename Group<NC, double>::M wilson_dag(const double* phi, int N, int64_t nxy, int64_t t, double lam, int S) {
  typedef Group<NC, double> G;
  double v[G::NA];
  typename G::M m = G::ident();
  bool first = true;
  for (int s = 0; s < S; ++s) {
    double ls = lam;
    if (S > 1) {
      ls = (double)S * lam - (double)s;
      ls = ls < 0.0 ? 0.0 : (ls > 1.0 ? 1.0 : ls);
    }
    if (ls == 0.0) continue;
    for (int a = 0; a < G::NA; ++a) v[a] = phi[((int64_t)(s * 2 + N) * G::NA + a) * nxy + t];
    const typename G::M f = G::expi(v, ls);
    m = first ? f : G::mul(f, m);
    first = false;
  }
  return m;
}

template <int NC>
GL_HD bool group_log(const typename Group<NC, double>::M& W, double* h);
template <>
GL_HD bool group_log<2>(const Group<2, double>::M& W, double* h) { return log_su2(W, h); }
template <>
GL_HD bool group_log<3>(const Group<3, double>::M& W, double* h) { return log_su3(W, h); }

template <int NC>
GL_HD bool same(const typename Group<NC, double>::M& a, const typename Group<NC, double>::M& b) {
  const double* pa = (const double*)&a;
  const double* pb = (const double*)&b;
  for (int k = 0; k < (int)(sizeof(a) / sizeof(double)); ++k)
    if (pa[k] != pb[k]) return false;
  return true;
}

// Behind a nucleus (Lambda = 1) the Wilson line and with it the links depend
// on the transverse site alone: full[N][t] = V_N^dag(x_T), then the links
// V_N(x) V_N^dag(x+i) in their stored form, "direction" 2 N + i of a lattice of
// one slice, formed once and copied to all slices.
template <int NC>
__global__ void k_wilson_full(const double* phi, typename Group<NC, double>::M* full, int64_t nxy, int S) {
  for (int64_t i = (int64_t)blockIdx.x * blockDim.x + threadIdx.x; i < 2 * nxy; i += (int64_t)gridDim.x * blockDim.x) {
    const int N = (int)(i / nxy);
    full[i] = wilson_dag<NC>(phi, N, nxy, i - (int64_t)N * nxy, 1.0, S);
  }
}

template <int NC, typename R>
__global__ void k_tail_links(const typename Group<NC, double>::M* full, typename V2T<R>::T* tail, Geom g) {
  const int64_t nxy = g.nxy;
  for (int64_t i = (int64_t)blockIdx.x * blockDim.x + threadIdx.x; i < 4 * nxy; i += (int64_t)gridDim.x * blockDim.x) {
    const int N = (int)(i / (2 * nxy)), d = (int)(i / nxy) & 1;
    const uint32_t t = (uint32_t)(i % nxy);
    const SiteNbr n = site_nbr_tz(g, t, 0);
    LinkIO<NC, R>::template store<double>(tail, 2 * N + d, nxy, t,
                                          Group<NC, double>::d_mul(full[N * nxy + t], full[N * nxy + n.p[d]]));
  }
}

// Links at t0 (and at t0 - dt where asked for) and E of one slice and one tile
// of kTileX x kTileY transverse sites.  The two profiles are disjoint (the
// centres lie more than 4 sigma from the box centre), so at most one nucleus
// has Lambda > 0 on a slice.  A slice ahead of both has unit links; a slice
// whose Lambda is 1 at both times copies the tail links; both have E = 0, and
// no FP64 work (the conversions and the division by dt of every site took 3 ms
// of an SU(2) 1024 x 128^2 event).  On the slices in between the Wilson lines of
// the tile and of its +x and +y neighbours at both times are formed once each in
// shared memory (2.4 exponentials per site instead of the 6 that a thread by
// itself takes): FP64-pipe bound there, bound by the stores elsewhere.  The whole
// initial state, with the DFTs, the series logarithm and the split divergence:
// SU(3) 512 x 64^2, sigma_L = 4, 7.5 -> 1.6 ms, SU(2) 1024 x 128^2 13.5 -> 1.7 ms.
// U1, the buffer the first step writes, only needs the absent z links of the
// last slice (all of it on a slab, whose halo slices are not stepped).
constexpr int kTileX = 16, kTileY = 8;

template <int NC, typename R>
__global__ void __launch_bounds__(kTileX * kTileY) k_init_links(
    const double* phi, const double* lam, const typename Group<NC, double>::M* full,
    const typename V2T<R>::T* tail, typename V2T<R>::T* U0, typename V2T<R>::T* U1,
    typename V2T<R>::T* Uprev, R* E, Geom g, double dt, int* flag, int S, int whole) {
  typedef Group<NC, double> G;
  typedef typename G::M M;
  typedef LinkIO<NC, R> IO;
  constexpr int NA = G::NA, PX = kTileX + 1, PN = PX * (kTileY + 1);
  __shared__ __align__(16) unsigned char raw[2 * PN * sizeof(M)];
  M* v = (M*)raw;  // [time][tile site]
  const int iz = blockIdx.y;
  const int ntx = (g.nx + kTileX - 1) / kTileX;
  const int x0 = ((int)blockIdx.x % ntx) * kTileX, y0 = ((int)blockIdx.x / ntx) * kTileY;
  const int lx = threadIdx.x % kTileX, ly = threadIdx.x / kTileX;
  const int ix = x0 + lx, iy = y0 + ly;
  const bool inside = ix < g.nx && iy < g.ny;
  const int64_t t = (int64_t)iy * g.nx + ix, s = (int64_t)iz * g.nxy + t;
  const bool copy1 = !whole || iz == g.nz - 1;
  const int N = lam[0 * g.nz + iz] != 0.0 || lam[2 * g.nz + iz] != 0.0 ? 0 : 1;
  const double l0 = lam[N * g.nz + iz], l1 = lam[(2 + N) * g.nz + iz];
  const bool moving = l0 != l1 || (l0 != 0.0 && l0 != 1.0);
  if (moving) {
    for (int q = threadIdx.x; q < 2 * PN; q += kTileX * kTileY) {
      const int tm = q / PN, p = q - tm * PN;
      const int64_t tt = (int64_t)((y0 + p / PX) % g.ny) * g.nx + (x0 + p % PX) % g.nx;
      const double l = tm ? l1 : l0;
      v[q] = l == 1.0 ? full[N * g.nxy + tt] : wilson_dag<NC>(phi, N, g.nxy, tt, l, S);
    }
    __syncthreads();
  }
  if (!inside) return;
  typedef LinkAlg<NC, R> L;  // links in their stored form
#pragma unroll 1
  for (int i = 0; i < 2; ++i) {
    if (moving) {
      const int p = ly * PX + lx, pn = p + (i == 0 ? 1 : PX);
      const M u0 = G::d_mul(v[p], v[pn]), u1 = G::d_mul(v[PN + p], v[PN + pn]);
      double h[NA];
#pragma unroll
      for (int a = 0; a < NA; ++a) h[a] = 0.0;
      if (!same<NC>(u0, u1) && !group_log<NC>(G::mul_d(u0, u1), h)) atomicOr(flag, 1);
#pragma unroll
      for (int a = 0; a < NA; ++a) E[(int64_t)(i * NA + a) * g.V + s] = (R)(h[a] / dt);
      IO::template store<double>(U0, i, g.V, s, u0);
      if (copy1) IO::template store<double>(U1, i, g.V, s, u0);
      if (Uprev) IO::template store<double>(Uprev, i, g.V, s, u1);
    } else {
      typename L::M u = L::ident();
      if (l0 != 0.0) u = IO::template load<R>(tail, 2 * N + i, g.nxy, t);
#pragma unroll
      for (int a = 0; a < NA; ++a) E[(int64_t)(i * NA + a) * g.V + s] = (R)0;
      IO::template store<R>(U0, i, g.V, s, u);
      if (copy1) IO::template store<R>(U1, i, g.V, s, u);
      if (Uprev) IO::template store<R>(Uprev, i, g.V, s, u);
    }
  }
#pragma unroll
  for (int a = 0; a < NA; ++a) E[(int64_t)(2 * NA + a) * g.V + s] = (R)0;
  const typename L::M one = L::ident();
  IO::template store<R>(U0, 2, g.V, s, one);
  if (copy1) IO::template store<R>(U1, 2, g.V, s, one);
  if (Uprev) IO::template store<R>(Uprev, 2, g.V, s, one);
}

// rho(x) = sum_i [E_i(x) - U_i^dag(x-i) E_i(x-i) U_i(x-i)] / a_i^2 of the
// stored state, in FP64, and max |rho| of every slice (slice_max begins as
// zeros; the bits of non-negative doubles order as the doubles do).  Only the
// slices inside the nuclei have fields, so kDivSplit blocks share a slice: with
// one block each, those slices' FP64 work lay on 130 of 152 SMs, 8 warps each
// (SU(3) 512 x 64^2: 1.38 ms).
constexpr int kDivSplit = 8;

template <int NC, typename R>
__global__ void __launch_bounds__(256) k_divergence(const typename V2T<R>::T* U, const R* E, Geom g, double ia2t,
                                                    double* rho3, double* slice_max) {
  typedef Group<NC, double> G;
  constexpr int NA = G::NA;
  __shared__ double sh[256];
  const int iz = blockIdx.x;
  double mx = 0.0;
  for (uint32_t t = blockIdx.y * blockDim.x + threadIdx.x; t < g.nxy; t += gridDim.y * blockDim.x) {
    const int64_t s = (int64_t)iz * g.nxy + t;
    const SiteNbr n = site_nbr_tz(g, t, iz);
    double dv[NA];
    for (int c = 0; c < NA; ++c) dv[c] = 0.0;
    for (int i = 0; i < 2; ++i) {  // E_z = 0
      R e[NA], em[NA];
      bool here = false, below = false;
      for (int c = 0; c < NA; ++c) {
        e[c] = E[(int64_t)(i * NA + c) * g.V + s];
        em[c] = E[(int64_t)(i * NA + c) * g.V + n.m[i]];
        here = here || e[c] != R(0);
        below = below || em[c] != R(0);
      }
      // E vanishes off the nuclei: no FP64 work there
      if (here)
        for (int c = 0; c < NA; ++c) dv[c] += ia2t * widen<double>(e[c]);
      if (!below) continue;
      double q[NA];
      for (int c = 0; c < NA; ++c) q[c] = widen<double>(em[c]);
      typename G::M um = LinkIO<NC, R>::template load<double>(U, i, g.V, n.m[i]);
      // the links of an FP32 state are unitary to their rounding only
      G::template adj_dag<sizeof(R) == 4>(um, q);
      for (int c = 0; c < NA; ++c) dv[c] -= ia2t * q[c];
    }
    for (int c = 0; c < NA; ++c) {
      rho3[(int64_t)c * g.V + s] = dv[c];
      mx = fmax(mx, fabs(dv[c]));
    }
  }
  sh[threadIdx.x] = mx;
  __syncthreads();
  for (int w = 128; w > 0; w >>= 1) {
    if ((int)threadIdx.x < w) sh[threadIdx.x] = fmax(sh[threadIdx.x], sh[threadIdx.x + w]);
    __syncthreads();
  }
  if (threadIdx.x == 0)
    atomicMax((unsigned long long*)&slice_max[iz], (unsigned long long)__double_as_longlong(sh[0]));
}

template <typename R>
__global__ void k_fill_window(const double* rho3, R* Q, int na, int z0, int W, Geom g) {
  const int64_t total = (int64_t)na * W * g.nxy;
  for (int64_t i = (int64_t)blockIdx.x * blockDim.x + threadIdx.x; i < total; i += (int64_t)gridDim.x * blockDim.x) {
    const int64_t t = i % g.nxy;
    const int64_t r = i / g.nxy;
    const int w = (int)(r % W);
    const int c = (int)(r / W);
    Q[i] = (R)rho3[(int64_t)c * g.V + (int64_t)(z0 + w) * g.nxy + t];
  }
}

static unsigned grid_for(int64_t n, int bs = 256) {
  int64_t nb = (n + bs - 1) / bs;
  if (nb > 152 * 32) nb = 152 * 32;
  if (nb < 1) nb = 1;
  return (unsigned)nb;
}

template <int NC, typename R>
static int init_t(glasma_ctx* c, const double* rho_host) {
  const glasma_params& p = c->p;
  const int na = c->na;
  const int64_t nxy = c->g.nxy, V = c->g.V;
  const int S = p.n_sheets > 1 ? p.n_sheets : 1;
  const int F = 2 * S * na;
  int st;
  // scratch: rho/phi (real), two complex work arrays and the DFT factors,
  // lambda table, Wilson lines and links behind the nuclei, rho3, slice max
  double* rho = (double*)ctx_alloc(c, sizeof(double) * F * nxy);
  double2* w0 = (double2*)ctx_alloc(c, sizeof(double2) * poisson_elems(p, F));
  double2* w1 = (double2*)ctx_alloc(c, sizeof(double2) * poisson_elems(p, F));
  double* lam = (double*)ctx_alloc(c, sizeof(double) * 4 * p.nz);
  double* rho3 = (double*)ctx_alloc(c, sizeof(double) * na * V);
  double* smax = (double*)ctx_alloc(c, sizeof(double) * p.nz);
  typedef typename Group<NC, double>::M MD;
  MD* full = (MD*)ctx_alloc(c, sizeof(MD) * 2 * nxy);
  typedef typename V2T<R>::T V2;
  V2* tail = (V2*)ctx_alloc(c, sizeof(V2) * 4 * (size_t)(link_elems(NC, nxy) / 3));
  if (!rho || !w0 || !w1 || !lam || !rho3 || !smax || !full || !tail) return set_error(GLASMA_ERR_OOM, "init scratch allocation failed");
  if (rho_host) {
    st = cuda_check(cudaMemcpyAsync(rho, rho_host, sizeof(double) * F * nxy, cudaMemcpyHostToDevice, c->stream),
                    "rho upload");
    if (st) return st;
  } else {
    k_philox_rho<<<grid_for(F * nxy), 256, 0, c->stream>>>(rho, na, p.nx, p.ny, S, p.seed,
                                                            S > 1 ? p.g2mu / sqrt((double)S) : p.g2mu);
  }
  st = device_poisson(p, rho, rho, F, w0, w1, c->stream);  // rho <- phi
  if (st) return st;
  // nucleus centres at t0 (box centre +- d) in global z (a slab's local
  // slice 0 is global slice zoff)
  const double zc = c->nz_glob * p.a_z / 2.0;
  const double d = p.z_offset > 0 ? p.z_offset : (ceil(4.0 * p.sigma_l / p.a_z) + 2.0) * p.a_z;
  k_profile<<<grid_for(4 * p.nz), 256, 0, c->stream>>>(lam, p.nz, c->zoff, p.a_z, p.sigma_l, zc + d, zc - d, p.dt);
  cudaMemsetAsync(c->dflag, 0, sizeof(int) * 8, c->stream);
  cudaMemsetAsync(smax, 0, sizeof(double) * p.nz, c->stream);
  k_wilson_full<NC><<<grid_for(2 * nxy, 64), 64, 0, c->stream>>>(rho, full, nxy, S);
  k_tail_links<NC, R><<<grid_for(4 * nxy, 64), 64, 0, c->stream>>>(full, tail, c->g);
  const unsigned tiles = (unsigned)(((p.nx + kTileX - 1) / kTileX) * ((p.ny + kTileY - 1) / kTileY));
  k_init_links<NC, R><<<dim3(tiles, (unsigned)p.nz), kTileX * kTileY, 0, c->stream>>>(
      rho, lam, full, tail, (typename V2T<R>::T*)c->U[0], (typename V2T<R>::T*)c->U[1],
      (typename V2T<R>::T*)c->Uprev, (R*)c->E, c->g, p.dt, c->dflag, S, c->slab ? 0 : 1);
  const int64_t per_slice = (nxy + 255) / 256;
  k_divergence<NC, R><<<dim3(p.nz, (unsigned)(per_slice < kDivSplit ? per_slice : kDivSplit)), 256, 0, c->stream>>>(
      (const typename V2T<R>::T*)c->U[0], (const R*)c->E, c->g, 1.0 / (p.a_t * p.a_t), rho3,
      smax);
  st = cuda_check(cudaGetLastError(), "init kernels");
  if (st) return st;
  std::vector<double> hmax(p.nz);
  int hflag = 0;
  st = cuda_check(cudaMemcpyAsync(hmax.data(), smax, sizeof(double) * p.nz, cudaMemcpyDeviceToHost, c->stream),
                  "slice max readback");
  if (st) return st;
  st = cuda_check(cudaMemcpyAsync(&hflag, c->dflag, sizeof(int), cudaMemcpyDeviceToHost, c->stream), "flag");
  if (st) return st;
  st = cuda_check(cudaStreamSynchronize(c->stream), "init sync");
  if (st) return st;
  if (hflag) return set_error(GLASMA_ERR_INVALID_ARG, "init: link change per step too large for the group log");
  // windows: A on slices above the centre, B below; none at the centre
  // (only the owned slices: a slab's halo slices carry no charge of their
  // own, and the divergence of its lower halo lacks the slice below)
  int alo = -1, ahi = -1, blo = -1, bhi = -1;
  for (int iz = c->lo; iz < c->hi; ++iz) {
    if (!(hmax[iz] == hmax[iz])) return set_error(GLASMA_ERR_NONFINITE, "init: non-finite charge density");
    if (hmax[iz] == 0.0) continue;
    const double z = (iz + c->zoff) * p.a_z;
    if (z > zc) {
      if (alo < 0) alo = iz;
      ahi = iz;
    } else if (z < zc) {
      if (blo < 0) blo = iz;
      bhi = iz;
    } else {
      return set_error(GLASMA_ERR_INTERNAL, "init: charge at the box centre");
    }
  }
  c->zA0 = alo < 0 ? 0 : alo;
  c->WA = alo < 0 ? 0 : ahi - alo + 1;
  c->zB0 = blo < 0 ? 0 : blo;
  c->WB = blo < 0 ? 0 : bhi - blo + 1;
  c->QA_cap = (size_t)(c->WA > 0 ? c->WA : 1);
  c->QB_cap = (size_t)(c->WB > 0 ? c->WB : 1);
  c->QA = ctx_alloc(c, c->rs * na * c->QA_cap * nxy);
  c->QB = ctx_alloc(c, c->rs * na * c->QB_cap * nxy);
  if (!c->QA || !c->QB) return set_error(GLASMA_ERR_OOM, "charge window allocation failed");
  if (c->WA > 0)
    k_fill_window<R><<<grid_for((int64_t)na * c->WA * nxy), 256, 0, c->stream>>>(rho3, (R*)c->QA, na, c->zA0,
                                                                                   c->WA, c->g);
  if (c->WB > 0)
    k_fill_window<R><<<grid_for((int64_t)na * c->WB * nxy), 256, 0, c->stream>>>(rho3, (R*)c->QB, na, c->zB0,
                                                                                   c->WB, c->g);
  st = cuda_check(cudaGetLastError(), "window fill");
  if (st) return st;
  if (c->Uit) {  // second iterate buffer of the implicit scheme: identity last-slice z links
    st = cuda_check(cudaMemcpyAsync(c->Uit, c->U[0], link_bytes(c), cudaMemcpyDeviceToDevice,
                                    c->stream),
                    "iterate buffer init");
    if (st) return st;
    c->uprev_valid = true;
  }
  st = cuda_check(cudaStreamSynchronize(c->stream), "init sync 2");
  ctx_free(c, tail);
  ctx_free(c, full);
  ctx_free(c, rho);
  ctx_free(c, w0);
  ctx_free(c, w1);
  ctx_free(c, lam);
  ctx_free(c, rho3);
  ctx_free(c, smax);
  return st;
}

// Device helpers shared with the adjoint: the MV draw, the transverse
// Poisson solve of F real [ny][nx] fields (in and out may alias; w0, w1 hold
// poisson_elems complex values each) and the profile table lam[(t*2 + N)*nz + iz].
int device_philox_rho(const glasma_params& p, int na, double* rho, cudaStream_t s) {
  const int64_t n = (int64_t)2 * na * p.nx * p.ny;
  k_philox_rho<<<grid_for(n), 256, 0, s>>>(rho, na, p.nx, p.ny, 1, p.seed, p.g2mu);
  return cuda_check(cudaGetLastError(), "philox rho");
}

int64_t poisson_elems(const glasma_params& p, int F) {
  return (int64_t)F * p.ny * (p.nx / 2 + 1) + p.nx + p.ny;
}

int device_poisson(const glasma_params& p, const double* in, double* out, int F, double2* w0, double2* w1,
                   cudaStream_t s) {
  const int nx = p.nx, ny = p.ny, nh = nx / 2 + 1;
  const int64_t rows = (int64_t)F * ny, nk = rows * nh, n = rows * nx;
  double2* tw = w1 + nk;  // the factors of x, then of y
  const double m2 = p.m_ir * p.m_ir, uv2 = p.uv_cutoff > 0 ? p.uv_cutoff * p.uv_cutoff : 0.0;
  k_twiddle<<<grid_for(nx + ny, 128), 128, 0, s>>>(tw, nx, ny);
  k_dft_x<<<grid_for(nk, 64), 64, 0, s>>>(in, w0, tw, rows, nx, nh);
  k_dft_y<<<grid_for(nk, 64), 64, 0, s>>>(w0, w1, tw + nx, F, ny, nx, nh, -1, p.a_t, m2, uv2);
  k_dft_y<<<grid_for(nk, 64), 64, 0, s>>>(w1, w0, tw + nx, F, ny, nx, nh, +1, p.a_t, m2, uv2);
  k_dft_x_real<<<grid_for(n, 64), 64, 0, s>>>(w0, out, tw, rows, nx, nh, 1.0 / ((double)nx * ny));
  return cuda_check(cudaGetLastError(), "poisson");
}

int device_profile(const glasma_params& p, double* lam, cudaStream_t s) {
  const double zc = p.nz * p.a_z / 2.0;
  const double d = p.z_offset > 0 ? p.z_offset : (ceil(4.0 * p.sigma_l / p.a_z) + 2.0) * p.a_z;
  k_profile<<<grid_for(4 * p.nz), 256, 0, s>>>(lam, p.nz, 0, p.a_z, p.sigma_l, zc + d, zc - d, p.dt);
  return cuda_check(cudaGetLastError(), "profile");
}

int run_init(glasma_ctx* c, const double* rho_host) {
  if (c->p.nc == 2) return c->rs == 8 ? init_t<2, double>(c, rho_host) : init_t<2, float>(c, rho_host);
  return c->rs == 8 ? init_t<3, double>(c, rho_host) : init_t<3, float>(c, rho_host);
}

}  // namespace glasma
