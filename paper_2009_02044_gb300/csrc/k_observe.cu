// Observables with FP64 accumulation: the discrete Gauss law residual
// (Sec. 3, Eq. gauss) and the per-slice energy-momentum tensor (Sec. 4).
// Reductions are deterministic: fixed grid, fixed-order tree in shared
// memory, fixed-order final pass over the block partials.
#include "dev_su2.cuh"
#include "divergence.cuh"
#include "glasma_internal.cuh"
#include "plaq_parts.cuh"

namespace glasma {

constexpr int kRedThreads = 256;
constexpr int kSu2Threads = 128;  // k_tmunu_su2

// In-block tree reduction of NV doubles per thread; op 0 = sum, 1 = max.
template <int NV, int T>
__device__ void block_reduce(double (*sh)[T], double* v, const int* op) {
  const int t = threadIdx.x;
#pragma unroll
  for (int k = 0; k < NV; ++k) sh[k][t] = v[k];
  __syncthreads();
  for (int w = T / 2; w > 0; w >>= 1) {
    if (t < w) {
#pragma unroll
      for (int k = 0; k < NV; ++k)
        sh[k][t] = op[k] ? fmax(sh[k][t], sh[k][t + w]) : sh[k][t] + sh[k][t + w];
    }
    __syncthreads();
  }
#pragma unroll
  for (int k = 0; k < NV; ++k) v[k] = sh[k][0];
}

// ---------------------------------------------------------------------------
// Gauss residual
// ---------------------------------------------------------------------------
template <typename R>
struct GaussArgs {
  const typename V2T<R>::T* U;
  const R* E;
  const R* QA;
  const R* QB;
  Geom g;
  double ia2[3];  // 1 / a_i^2
  int zA0, WA, zB0, WB;
  int64_t s0, s1;  // sites of the owned slices
  double* part;    // [gridDim][4]
};

// The FP64 pipe bounds it (SU(3): some 475 of its operations per site; 160 x 64^2
// FP32 0.651 ms, 0.700 with the general transport but its sums formed link by
// link and the maximum by FP64 comparisons).  More registers than this leave
// too few warps for the loads (0.674 at 250).
template <int NC, typename R>
__global__ void __launch_bounds__(kRedThreads, NC == 2 ? 3 : 2) k_gauss(GaussArgs<R> a) {
  typedef Group<NC, double> G;
  constexpr int NA = G::NA;
  __shared__ double sh[4][kRedThreads];
  unsigned long long gmax = 0;  // bits of the largest |G|
  double gsum2 = 0, rmax = 0, bad = 0;
  for (int64_t s = a.s0 + (int64_t)blockIdx.x * blockDim.x + threadIdx.x; s < a.s1;
       s += (int64_t)gridDim.x * blockDim.x) {
    const SiteNbr n = site_nbr(a.g, s);
    double gv[NA];
    divergence_at<NC, R>(a.U, a.E, a.g, n, a.ia2, gv);
    const int ka = n.iz - a.zA0, kb = n.iz - a.zB0;
    const bool ina = ka >= 0 && ka < a.WA, inb = kb >= 0 && kb < a.WB;
    if (ina || inb) {
      const int64_t t = s % a.g.nxy;
#pragma unroll
      for (int c = 0; c < NA; ++c) {
        double rho = 0.0;
        if (ina) rho += widen<double>(a.QA[((int64_t)c * a.WA + ka) * a.g.nxy + t]);
        if (inb) rho += widen<double>(a.QB[((int64_t)c * a.WB + kb) * a.g.nxy + t]);
        gv[c] -= rho;
        rmax = fmax(rmax, fabs(rho));
      }
    }
#pragma unroll
    for (int c = 0; c < NA; ++c) {
      // the bits of non-negative doubles order as they do: no FP64 comparison
      const unsigned long long b = (unsigned long long)__double_as_longlong(fabs(gv[c]));
      const unsigned long long inf = 0x7ff0000000000000ULL;
      if (b >= inf) bad += 1.0;
      if (b <= inf && b > gmax) gmax = b;
      gsum2 += gv[c] * gv[c];
    }
  }
  double v[4] = {__longlong_as_double((long long)gmax), gsum2, rmax, bad};
  const int op[4] = {1, 0, 1, 0};
  block_reduce<4>(sh, v, op);
  if (threadIdx.x == 0)
#pragma unroll
    for (int k = 0; k < 4; ++k) a.part[blockIdx.x * 4 + k] = v[k];
}

// One block folds nb partials of width NV in a fixed order; bit k of MAXMASK
// selects max (else sum) for component k.
template <int NV, int MAXMASK>
__global__ void __launch_bounds__(kRedThreads) k_fold(const double* part, int nb, double* out) {
  __shared__ double sh[NV][kRedThreads];
  int op[NV];
#pragma unroll
  for (int k = 0; k < NV; ++k) op[k] = (MAXMASK >> k) & 1;
  double v[NV];
#pragma unroll
  for (int k = 0; k < NV; ++k) v[k] = 0.0;
  for (int b = threadIdx.x; b < nb; b += kRedThreads)
#pragma unroll
    for (int k = 0; k < NV; ++k) v[k] = op[k] ? fmax(v[k], part[b * NV + k]) : v[k] + part[b * NV + k];
  block_reduce<NV>(sh, v, op);
  if (threadIdx.x == 0)
#pragma unroll
    for (int k = 0; k < NV; ++k) out[k] = v[k];
}

static int reduction_grid(glasma_ctx* c) {
  int sms = 152;
  cudaDeviceGetAttribute(&sms, cudaDevAttrMultiProcessorCount, c->device);
  int64_t need = ((int64_t)(c->hi - c->lo) * c->g.nxy + kRedThreads - 1) / kRedThreads;
  int64_t nb = (int64_t)sms * 4;
  return (int)(need < nb ? need : nb);
}

template <int NC, typename R>
static int gauss_t(glasma_ctx* c, double* out3) {
  GaussArgs<R> a;
  a.U = (const typename V2T<R>::T*)c->U[c->cur];
  a.E = (const R*)c->E;
  a.QA = (const R*)c->QA;
  a.QB = (const R*)c->QB;
  a.g = c->g;
  a.ia2[0] = a.ia2[1] = 1.0 / (c->p.a_t * c->p.a_t);
  a.ia2[2] = 1.0 / (c->p.a_z * c->p.a_z);
  a.zA0 = c->zA0;
  a.WA = c->WA;
  a.zB0 = c->zB0;
  a.WB = c->WB;
  a.s0 = (int64_t)c->lo * c->g.nxy;
  a.s1 = (int64_t)c->hi * c->g.nxy;
  const int nb = reduction_grid(c);
  // partials, then the op table and the 4 results, in the context's scratch
  if ((size_t)nb * 4 + 8 > c->red_cap) return set_error(GLASMA_ERR_INTERNAL, "reduction scratch too small");
  a.part = c->red;
  double* res = c->red + (size_t)nb * 4;
  k_gauss<NC, R><<<nb, kRedThreads, 0, c->stream>>>(a);
  int st = cuda_check(cudaGetLastError(), "k_gauss launch");
  if (st) return st;
  k_fold<4, 0x5><<<1, kRedThreads, 0, c->stream>>>(c->red, nb, res);
  st = cuda_check(cudaGetLastError(), "k_fold launch");
  if (st) return st;
  double h[4];
  st = cuda_check(cudaMemcpyAsync(h, res, sizeof(h), cudaMemcpyDeviceToHost, c->stream), "gauss readback");
  if (st) return st;
  st = cuda_check(cudaStreamSynchronize(c->stream), "gauss sync");
  if (st) return st;
  out3[0] = h[0];
  out3[1] = sqrt(h[1] / ((double)(a.s1 - a.s0) * (c->na)));
  out3[2] = h[2];
  if (h[3] != 0.0) return set_error(GLASMA_ERR_NONFINITE, "Gauss residual met a non-finite value");
  return GLASMA_OK;
}

int launch_gauss(glasma_ctx* c, double* out3) {
  if (c->p.nc == 2) return c->rs == 8 ? gauss_t<2, double>(c, out3) : gauss_t<2, float>(c, out3);
  return c->rs == 8 ? gauss_t<3, double>(c, out3) : gauss_t<3, float>(c, out3);
}

// ---------------------------------------------------------------------------
// Are the links on the group?  An FP64 evolution leaves it by some 1e-16 per
// step, an FP32 link by the rounding of its entries (1e-7).
// ---------------------------------------------------------------------------
template <int NC, typename R>
__global__ void __launch_bounds__(kRedThreads) k_links_off(const typename V2T<R>::T* U, int64_t V, double tol, int* off) {
  typedef Group<NC, double> G;
  double dev = 0.0;
  for (int64_t s = (int64_t)blockIdx.x * blockDim.x + threadIdx.x; s < V; s += (int64_t)gridDim.x * blockDim.x) {
    const typename G::M u = LinkIO<NC, R>::template load<double>(U, (int)blockIdx.y, V, s);
    double d;
    if constexpr (NC == 2) {
      d = fabs(fma(u.a.re, u.a.re, fma(u.a.im, u.a.im, fma(u.b.re, u.b.re, fma(u.b.im, u.b.im, -1.0)))));
    } else {
      // rows 0 and 1 orthonormal, row 2 their cross product's conjugate
      cplx<double> p = mulc(u.m[0], u.m[3]);
      p = fma_cj(u.m[1], u.m[4], p);
      p = fma_cj(u.m[2], u.m[5], p);
      d = fabs(p.re) + fabs(p.im);
#pragma unroll
      for (int r = 0; r < 2; ++r) {
        double n = -1.0;
#pragma unroll
        for (int k = 0; k < 3; ++k) n = fma(u.m[3 * r + k].re, u.m[3 * r + k].re, fma(u.m[3 * r + k].im, u.m[3 * r + k].im, n));
        d += fabs(n);
      }
#pragma unroll
      for (int k = 0; k < 3; ++k) {
        const int a = (k + 1) % 3, b = (k + 2) % 3;
        const cplx<double> x = u.m[a] * u.m[3 + b] - u.m[b] * u.m[3 + a] - cj(u.m[6 + k]);
        d += fabs(x.re) + fabs(x.im);
      }
    }
    if (!(d <= dev)) dev = d;  // a NaN stays
    if (!(dev <= tol)) break;
  }
  if (!(dev <= tol)) atomicOr(off, 1);
}

template <int NC, typename R>
static int links_off_t(glasma_ctx* c, const void* U, bool* off) {
  int* flag = c->dflag + 2;
  int st = cuda_check(cudaMemsetAsync(flag, 0, sizeof(int), c->stream), "link check");
  if (st) return st;
  k_links_off<NC, R><<<dim3(4 * c->sms, 3), kRedThreads, 0, c->stream>>>((const typename V2T<R>::T*)U, c->g.V,
                                                                        sizeof(R) == 8 ? 1e-10 : 4e-6, flag);
  st = cuda_check(cudaGetLastError(), "k_links_off launch");
  int h = 0;
  if (!st) st = cuda_check(cudaMemcpyAsync(&h, flag, sizeof(int), cudaMemcpyDeviceToHost, c->stream), "link check");
  if (!st) st = cuda_check(cudaStreamSynchronize(c->stream), "link check");
  *off = h != 0;
  return st;
}

int links_off_group(glasma_ctx* c, const void* U, bool* off) {
  if (c->p.nc == 2) return c->rs == 8 ? links_off_t<2, double>(c, U, off) : links_off_t<2, float>(c, U, off);
  return c->rs == 8 ? links_off_t<3, double>(c, U, off) : links_off_t<3, float>(c, U, off);
}

// ---------------------------------------------------------------------------
// T^{mu nu} per z slice
// ---------------------------------------------------------------------------
template <typename R>
struct TmnArgs {
  const typename V2T<R>::T* U;
  const R* E;
  const R* QA;
  const R* QB;
  Geom g;
  R dt;
  R w[3];
  R az2;
  // products of reciprocals of the spacings, formed on the host (an FP64
  // division is a long sequence on GB300's narrow FP64 pipe):
  double binv[2];   // 1 / (a_i a_j)^2 of the plane xy and of xz and yz
  double hinv2[2];  // 1 / (2 a_i^2) of x and y, and of z
  double slc;       // Poynting weight 1 / (a_t^2 a_z)
  int hop;
  int zA0, WA, zB0, WB;
  int split;     // blocks per z slice
  uint32_t per;  // consecutive sites of a block, a multiple of its threads
  double* part;  // [nz][split][5] block sums of eps, p_L, p_T, S_L, non-finite count
};

// ||x - y||_F^2 of two links in the state's representation (for FP32 the
// deviations from 1, whose difference is that of the links), in the state's
// precision: a difference of two FP32 entries rounds to within u of itself,
// and the sum of squares has no cancellation, so the FP32 value carries the
// FP32 products' own relative accuracy; it enters the FP64 sums once per
// site.
template <int NC, typename R> struct Fro2;
template <typename R>
struct Fro2<3, R> {
  GL_HD static R diff(const typename Group<3, R>::M& x, const typename Group<3, R>::M& y) {
    R acc = R(0);
#pragma unroll
    for (int k = 0; k < 9; ++k) {
      const R dr = x.m[k].re - y.m[k].re, di = x.m[k].im - y.m[k].im;
      acc += dr * dr + di * di;
    }
    return acc;
  }
};
template <typename R>
struct Fro2<2, R> {
  GL_HD static R diff(const typename Group<2, R>::M& x, const typename Group<2, R>::M& y) {
    const R a = x.a.re - y.a.re, b = x.a.im - y.a.im;
    const R c = x.b.re - y.b.re, d = x.b.im - y.b.im;
    return R(2) * (a * a + b * b + c * c + d * d);
  }
};

// FP64 sum of a thread's per-site values.  Those of an FP32 state are widened on
// the integer pipe (add) or by the conversion instruction of the FP64 pipe
// (add_cvt), whichever has time to spare: SU(3) 512 x 64^2 0.419 ms per sample by
// add alone; SU(2) 1024 x 128^2 0.660 by add alone, 0.665 by conversions alone,
// 0.631 with both (two floats, whose sum is good to 2^-48 and overflows where a
// double does not, 0.424 and 0.614).
template <typename R>
struct SiteSum {
  double s = 0.0;
  __device__ __forceinline__ void add(R x) { s += widen<double>(x); }
  __device__ __forceinline__ void add_cvt(R x) { s += (double)x; }
  __device__ __forceinline__ double get() const { return s; }
};

// The block's sums of E_x^2 + E_y^2, E_z^2, b_xy, b_xz + b_yz (without the
// spacings) and E B as its row of partial sums.
template <typename R, int T>
__device__ __forceinline__ void tmunu_write(const TmnArgs<R>& a, double (*sh)[T], const SiteSum<R>& et,
                                            const SiteSum<R>& ez, const SiteSum<R>& bl, const SiteSum<R>& bt,
                                            const SiteSum<R>& sl, int iz) {
  double v[5] = {et.get(), ez.get(), bl.get(), bt.get(), sl.get()};
  const int op[5] = {0, 0, 0, 0, 0};
  block_reduce<5>(sh, v, op);
  if (threadIdx.x == 0) {
    // eps, p_L, p_T, S_L and whether a value was not finite (the directions x
    // and y have the same spacing)
    const double e_t = 0.5 * v[0] * a.hinv2[0], e_z = 0.5 * v[1] * a.hinv2[1];
    const double b_l = v[2] * a.binv[0], b_t = v[3] * a.binv[1];
    const double p_t = e_z + b_l;
    double* out = a.part + ((int64_t)iz * a.split + blockIdx.y) * 5;
    out[0] = e_t + e_z + b_l + b_t;
    out[1] = e_t + b_t - p_t;
    out[2] = p_t;
    out[3] = v[4] * a.slc;
    out[4] = isfinite(out[0]) && isfinite(out[3]) ? 0.0 : 1.0;
  }
}

// Blocks per SM.  SU(3) FP32: 2 at 128 registers (16 warps; load latency is
// what is left).
template <int NC, typename R> struct TmnOcc { static constexpr int blocks = 1; };
template <> struct TmnOcc<3, float> { static constexpr int blocks = 2; };

// Per-site arithmetic in the state's precision R (FP32 plaquette products in
// the deviation form; the per-site sums of squares and of E B products in R,
// all of positive terms except the Poynting sum), every accumulation over sites
// in FP64.  Block (iz, p) takes `per` consecutive
// sites of slice iz, 256 at a time (neighbouring rows meet in L1); k_tmunu_fold
// adds the split block sums of a slice in a fixed order.
// The plaquettes based at a site serve three ends at once: their energy, the
// field B, and the forward half of the force on both their links; only the
// backward staples are formed for the force alone.  That is 23 link products
// per site where forward staples by themselves made 35.  Per sample: SU(3)
// 512 x 64^2 FP32 0.797 -> 0.449 ms (0.42 with staples of two rows and FP64 sums),
// FP64 15.2 -> 10.8 ms.
// ANY: for links off the group.
template <int NC, typename R, bool ANY>
__global__ void __launch_bounds__(kRedThreads, TmnOcc<NC, R>::blocks) k_tmunu(TmnArgs<R> a) {
  follow();
  typedef LinkAlg<NC, R> G;
  typedef LinkIO<NC, R> IO;
  typedef typename G::M M;
  constexpr int NA = G::NA;
  __shared__ double sh[5][kRedThreads];
  const Geom& g = a.g;
  const int iz = blockIdx.x;
  // sums of E_x^2 + E_y^2, E_z^2, b_xy, b_xz + b_yz (without the spacings), E B
  SiteSum<R> et, ez, bl, bt, sl;
  for (uint32_t t = blockIdx.y * a.per + threadIdx.x, end = min((blockIdx.y + 1) * a.per, (uint32_t)g.nxy); t < end;
       t += kRedThreads) {
    const SiteNbr n = site_nbr_tz(g, t, iz);
    const int64_t s = n.s;
    // plaquettes based here: b_ij = ||U_i(x) U_j(x+i) - U_j(x) U_i(x+j)||_F^2
    // / (a_i a_j)^2 (= 2 (N - Re tr U_ij) for unitary links, without its
    // cancellation) and Im tr t^a U_ij = Im tr t^a A B^dagger:
    // B_y = +2 Im tr t U_xz / (a_x a_z), B_x = -2 Im tr t U_yz / (a_y a_z)
    R pxy[NA], pxz[NA], pyz[NA];
    {
      const M A = G::mul(IO::template load<R>(a.U, 0, g.V, s), IO::template load<R>(a.U, 1, g.V, n.p[0]));
      const M B = G::mul(IO::template load<R>(a.U, 1, g.V, s), IO::template load<R>(a.U, 0, g.V, n.p[1]));
      bl.add(Fro2<NC, R>::diff(A, B));
      G::proj_prod_d(A, B, pxy);
    }
    if (iz <= g.nz - 2) {
      {
        const M A = G::mul(IO::template load<R>(a.U, 0, g.V, s), IO::template load<R>(a.U, 2, g.V, n.p[0]));
        const M B = G::mul(IO::template load<R>(a.U, 2, g.V, s), IO::template load<R>(a.U, 0, g.V, n.p[2]));
        bt.add(Fro2<NC, R>::diff(A, B));
        G::proj_prod_d(A, B, pxz);
      }
      {
        const M A = G::mul(IO::template load<R>(a.U, 1, g.V, s), IO::template load<R>(a.U, 2, g.V, n.p[1]));
        const M B = G::mul(IO::template load<R>(a.U, 2, g.V, s), IO::template load<R>(a.U, 1, g.V, n.p[2]));
        bt.add(Fro2<NC, R>::diff(A, B));
        G::proj_prod_d(A, B, pyz);
      }
    } else {
#pragma unroll
      for (int c = 0; c < NA; ++c) pxz[c] = pyz[c] = R(0);
    }
    const int ilast = (iz == g.nz - 1) ? 2 : 3;
#pragma unroll 1
    for (int i = 0; i < ilast; ++i) {
      // F_i = -sum_j w_j (the plaquettes based here, U_ji = U_ij^dagger) - the
      // backward staples (link_force_staple)
      R F[NA];
#pragma unroll
      for (int c = 0; c < NA; ++c)
        F[c] = i == 0 ? -a.w[1] * pxy[c] - a.w[2] * pxz[c]
                      : i == 1 ? a.w[0] * pxy[c] - a.w[2] * pyz[c] : a.w[0] * pxz[c] + a.w[1] * pyz[c];
      typename G::Sum S = G::zero_sum();
#pragma unroll 1
      for (int j = 0; j < 3; ++j) {
        if (j == i || (j == 2 && iz == 0)) continue;
        const int64_t mj = nbr_m(n, j);
        G::sum_add(S, a.w[j], G::template staple_bwd<ANY>(IO::template load<R>(a.U, i, g.V, mj),
                                            IO::template load<R>(a.U, j, g.V, nbr_p(n, i) + mj - s),
                                            IO::template load<R>(a.U, j, g.V, mj)));
      }
      R q[NA];
      G::proj_mul_sum(IO::template load<R>(a.U, i, g.V, s), S, q);
      R eo[NA], en[NA];
#pragma unroll
      for (int c = 0; c < NA; ++c) {
        eo[c] = a.E[(int64_t)(i * NA + c) * g.V + s];
        en[c] = eo[c] + a.dt * (F[c] - q[c]);
      }
      if (i == 2 && a.hop) {
        const int kb = iz - a.zB0;
        if (kb >= 0 && kb < a.WB)
#pragma unroll
          for (int c = 0; c < NA; ++c) en[c] -= a.az2 * a.QB[((int64_t)c * a.WB + kb) * g.nxy + t];
        const int ka = iz + 1 - a.zA0;
        if (ka >= 0 && ka < a.WA) {
#pragma unroll
          for (int c = 0; c < NA; ++c) q[c] = a.QA[((int64_t)c * a.WA + ka) * g.nxy + t];
          G::template adj<ANY>(IO::template load<R>(a.U, 2, g.V, s), q);
#pragma unroll
          for (int c = 0; c < NA; ++c) en[c] += a.az2 * q[c];
        }
      }
      R acc = R(0), dot = R(0);
#pragma unroll
      for (int c = 0; c < NA; ++c) {
        acc += eo[c] * eo[c] + en[c] * en[c];
        // S_L = sum_a (Ebar_x B_y - Ebar_y B_x), Ebar the time mean of E / a
        dot += (eo[c] + en[c]) * (i == 0 ? pxz[c] : pyz[c]);
      }
      if (i == 2) {
        ez.add(acc);
      } else {
        et.add(acc);
        sl.add(dot);
      }
    }
  }
  tmunu_write(a, sh, et, ez, bl, bt, sl, iz);
}

// The same for FP32 SU(2) in the quaternion form of k_step_su2.cu: the six
// backward staples are values vec AB, vec BA of the plaquettes at x - e_x, x -
// e_y and x - e_z (46 multiply-adds each, where the general form takes two
// products and a projection), and the fields are loaded before anything else.
// Load latency and the waves of blocks bound it: 8 blocks of 128 threads per SM
// at 64 registers (120 B of spills) take, on SU(2) 1024 x 128^2, 768 x 64^2 and
// 131 x 45 x 48, 0.63, 0.139 and 0.021 ms (general form 0.94, 0.227 and 0.027);
// 6 blocks at 80 registers 0.69, 0.159 and 0.021, blocks of 256 at 64 registers
// 0.63, 0.176 and 0.026.
__global__ void __launch_bounds__(kSu2Threads, 8) k_tmunu_su2(TmnArgs<float> a) {
  follow();
  __shared__ double sh[5][kSu2Threads];
  const Geom& g = a.g;
  const int iz = blockIdx.x;
  const bool up = iz < g.nz - 1, down = iz > 0;
  const uint32_t nx = (uint32_t)g.nx, ny = (uint32_t)g.ny;
  const float4* Ux = reinterpret_cast<const float4*>(a.U) + (int64_t)iz * g.nxy;
  const float4 *Uy = Ux + g.V, *Uz = Uy + g.V;
  const float wt = a.w[0], wz = a.w[2];
  SiteSum<float> et, ez, bl, bt, sl;
  auto dist2 = [](Dev4 A, Dev4 B) {  // ||A - B||_F^2
    const float w = A.w - B.w, x = A.x - B.x, y = A.y - B.y, z = A.z - B.z;
    return 2.f * fma(w, w, fma(x, x, fma(y, y, z * z)));
  };
  for (uint32_t t = blockIdx.y * a.per + threadIdx.x, end = min((blockIdx.y + 1) * a.per, (uint32_t)g.nxy); t < end;
       t += kSu2Threads) {
    const uint32_t iy = t / nx, ix = t - iy * nx;
    const uint32_t xp = ix + 1 == nx ? 0 : ix + 1, xm = ix == 0 ? nx - 1 : ix - 1;
    const uint32_t yp = (iy + 1 == ny ? 0 : iy + 1) * nx, ym = (iy == 0 ? ny - 1 : iy - 1) * nx, y0 = iy * nx;
    const uint32_t txp = y0 + xp, txm = y0 + xm, typ = yp + ix, tym = ym + ix, txmyp = yp + xm, txpym = ym + xp;
    const int64_t s = (int64_t)iz * g.nxy + t;
    Vec3 E[3];
#pragma unroll
    for (int i = 0; i < 3; ++i) {
      const float* e = a.E + (int64_t)(3 * i) * g.V + s;
      E[i] = Vec3{e[0], e[g.V], e[2 * g.V]};
    }
    const Dev4 ux = dev_load(Ux + t), uy = dev_load(Uy + t);
    Dev4 uz{0.f, 0.f, 0.f, 0.f};
    Vec3 F[3] = {{0.f, 0.f, 0.f}, {0.f, 0.f, 0.f}, {0.f, 0.f, 0.f}}, pxz{0.f, 0.f, 0.f}, pyz = pxz;
    {
      const Dev4 A = dev_mulq(ux, dev_load(Uy + txp)), B = dev_mulq(uy, dev_load(Ux + typ));
      bl.add_cvt(dist2(A, B));
      const Vec3 p = vec_ab(A, dev_dag(B));
      add3(F[0], -wt, p);
      add3(F[1], wt, p);
    }
    if (up) {
      uz = dev_load(Uz + t);
      Dev4 A = dev_mulq(ux, dev_load(Uz + txp)), B = dev_mulq(uz, dev_load(Ux + g.nxy + t));
      bt.add_cvt(dist2(A, B));
      pxz = vec_ab(A, dev_dag(B));
      A = dev_mulq(uy, dev_load(Uz + typ));
      B = dev_mulq(uz, dev_load(Uy + g.nxy + t));
      bt.add_cvt(dist2(A, B));
      pyz = vec_ab(A, dev_dag(B));
      add3(F[0], -wz, pxz);
      add3(F[1], -wz, pyz);
      add3(F[2], wt, pxz);
      add3(F[2], wt, pyz);
    }
    {
      const Dev4 vx = dev_load(Ux + txm);
      add3(F[1], -wt, vec_ab(dev_mulq(uy, dev_dag(dev_load(Ux + txmyp))), dev_mulq(dev_dag(dev_load(Uy + txm)), vx)));
      if (up)
        add3(F[2], -wt,
             vec_ab(dev_mulq(uz, dev_dag(dev_load(Ux + g.nxy + txm))), dev_mulq(dev_dag(dev_load(Uz + txm)), vx)));
    }
    {
      const Dev4 vy = dev_load(Uy + tym);
      add3(F[0], wt, vec_ab(dev_mulq(dev_dag(vy), dev_load(Ux + tym)), dev_mulq(dev_load(Uy + txpym), dev_dag(ux))));
      if (up)
        add3(F[2], -wt,
             vec_ab(dev_mulq(uz, dev_dag(dev_load(Uy + g.nxy + tym))), dev_mulq(dev_dag(dev_load(Uz + tym)), vy)));
    }
    if (down) {  // vec BA of the planes xz and yz of the slice below
      const Dev4 vz = dev_dag(dev_load(Uz - g.nxy + t));
      add3(F[0], wz, vec_ab(dev_mulq(vz, dev_load(Ux - g.nxy + t)), dev_mulq(dev_load(Uz - g.nxy + txp), dev_dag(ux))));
      add3(F[1], wz, vec_ab(dev_mulq(vz, dev_load(Uy - g.nxy + t)), dev_mulq(dev_load(Uz - g.nxy + typ), dev_dag(uy))));
    }
    Vec3 dj{0.f, 0.f, 0.f};
    if (a.hop && up) {
      const int kb = iz - a.zB0, ka = iz + 1 - a.zA0;
      if (kb >= 0 && kb < a.WB) {
        const float* q = a.QB + (int64_t)kb * g.nxy + t;
        const int64_t S = (int64_t)a.WB * g.nxy;
        add3(dj, -a.az2, Vec3{q[0], q[S], q[2 * S]});
      }
      if (ka >= 0 && ka < a.WA) {
        const float* q = a.QA + (int64_t)ka * g.nxy + t;
        const int64_t S = (int64_t)a.WA * g.nxy;
        add3(dj, a.az2, turn3(uz, Vec3{q[0], q[S], q[2 * S]}));
      }
    }
#pragma unroll
    for (int i = 0; i < 3; ++i) {
      Vec3 n = E[i];
      add3(n, a.dt, F[i]);
      if (i == 2) n = Vec3{n.x + dj.x, n.y + dj.y, n.z + dj.z};
      const float sq = fma(E[i].x, E[i].x, fma(E[i].y, E[i].y, E[i].z * E[i].z)) +
                       fma(n.x, n.x, fma(n.y, n.y, n.z * n.z));
      if (i == 2) {
        if (up) ez.add_cvt(sq);  // no z link on the last slice
      } else {
        const Vec3 p = i == 0 ? pxz : pyz;
        et.add(sq);
        sl.add(fma(E[i].x + n.x, p.x, fma(E[i].y + n.y, p.y, (E[i].z + n.z) * p.z)));
      }
    }
  }
  tmunu_write(a, sh, et, ez, bl, bt, sl, iz);
}

// FP64 where the context has the step's scratch: the plaquettes and the forces
// come from the step's first pass (k_step_plaq64.cu), which forms each
// plaquette once where k_tmunu forms 23 link products per site, and this pass
// adds E_{n+1/2} and the sums.  The FP64 pipe bounds both: SU(3) 160 x 24^2 0.607 ->
// 0.347 ms, 90 x 7 x 11 0.109 -> 0.055, 512 x 64^2 10.8 -> 7.7; SU(2) 128 x 16^2
// 0.049 -> 0.035, 512 x 64^2 2.33 -> 1.50.
template <int NC>
__global__ void __launch_bounds__(kRedThreads) k_tmunu_parts(TmnArgs<double> a, const double* vecs, int ring, int z0) {
  follow();
  typedef Group<NC, double> G;
  constexpr int NA = G::NA;
  __shared__ double sh[5][kRedThreads];
  const Geom& g = a.g;
  const int iz = z0 + (int)blockIdx.x;
  const bool up = iz < g.nz - 1;
  const int64_t S = (int64_t)ring * g.nxy, here = (int64_t)(iz % ring) * g.nxy;
  SiteSum<double> et, ez, bl, bt, sl;
  for (uint32_t t = blockIdx.y * a.per + threadIdx.x, end = min((blockIdx.y + 1) * a.per, (uint32_t)g.nxy); t < end;
       t += kRedThreads) {
    const SiteNbr n = site_nbr_tz(g, t, iz);
    const double* norm = vecs + (int64_t)kPartVecs * NA * S + here + t;
    bl.add(norm[0]);
    if (up) bt.add(norm[S] + norm[2 * S]);
#pragma unroll 1
    for (int i = 0; i < (up ? 3 : 2); ++i) {
      double F[NA], eo[NA], en[NA];
      part_force<NA>(vecs, g, ring, n, t, iz, i, a.w, F);
#pragma unroll
      for (int c = 0; c < NA; ++c) {
        eo[c] = a.E[(int64_t)(i * NA + c) * g.V + n.s];
        en[c] = fma(a.dt, F[c], eo[c]);
      }
      if (i == 2 && a.hop) {
        const int kb = iz - a.zB0, ka = iz + 1 - a.zA0;
        if (kb >= 0 && kb < a.WB)
#pragma unroll
          for (int c = 0; c < NA; ++c) en[c] -= a.az2 * a.QB[((int64_t)c * a.WB + kb) * g.nxy + t];
        if (ka >= 0 && ka < a.WA) {
          double q[NA];
#pragma unroll
          for (int c = 0; c < NA; ++c) q[c] = a.QA[((int64_t)c * a.WA + ka) * g.nxy + t];
          G::adj(LinkIO<NC, double>::template load<double>(a.U, 2, g.V, n.s), q);
#pragma unroll
          for (int c = 0; c < NA; ++c) en[c] += a.az2 * q[c];
        }
      }
      double acc = 0.0, dot = 0.0;
#pragma unroll
      for (int c = 0; c < NA; ++c) acc = fma(eo[c], eo[c], fma(en[c], en[c], acc));
      if (i == 2) {
        ez.add(acc);
        continue;
      }
      et.add(acc);
      if (up) {  // S_L: (E_x, the plane xz) and (E_y, the plane yz), as in k_tmunu
        const double* p = vecs + (int64_t)(kP0 + 1 + i) * NA * S + here + t;
#pragma unroll
        for (int c = 0; c < NA; ++c) dot = fma(eo[c] + en[c], p[c * S], dot);
        sl.add(dot);
      }
    }
  }
  tmunu_write(a, sh, et, ez, bl, bt, sl, iz);
}

// tab[iz] = (sum over the split blocks of slice iz, in block order) / nxy;
// a slice that met a non-finite value gets a NaN energy density.
__global__ void k_tmunu_fold(const double* part, int split, int nz, double inv, double* tab) {
  follow();
  const int iz = blockIdx.x * blockDim.x + threadIdx.x;
  if (iz >= nz) return;
  double v[5] = {0, 0, 0, 0, 0};
  for (int p = 0; p < split; ++p)
#pragma unroll
    for (int k = 0; k < 5; ++k) v[k] += part[((int64_t)iz * split + p) * 5 + k];
#pragma unroll
  for (int k = 0; k < 4; ++k) tab[iz * 4 + k] = v[k] * inv;
  if (v[4] != 0.0) tab[iz * 4 + 0] = __longlong_as_double(0x7ff8000000000000LL);  // NaN marks it
}

template <int NC, typename R>
static int launch_tmunu_kernel(glasma_ctx* c, const TmnArgs<R>& a) {
  const dim3 grid((unsigned)c->g.nz, (unsigned)a.split);
  if (c->links_off)
    return launch_following("k_tmunu launch", k_tmunu<NC, R, true>, grid, kRedThreads, 0, c->stream, a);
  if constexpr (sizeof(R) == 4 && NC == 2) {
    return launch_following("k_tmunu_su2 launch", k_tmunu_su2, grid, kSu2Threads, 0, c->stream, a);
  } else {
    if constexpr (sizeof(R) == 8) {
      if (c->part) {
        const int ring = c->ring;
        for (int z0 = 0; z0 < c->g.nz; z0 += ring - 1) {
          const int z1 = min(z0 + ring - 1, c->g.nz);
          int st = launch_parts_norms(c, z0, z1);
          if (!st)
            st = launch_following("k_tmunu_parts launch", k_tmunu_parts<NC>, dim3((unsigned)(z1 - z0), grid.y),
                                  kRedThreads, 0, c->stream, a, (const double*)c->part, ring, z0);
          if (st) return st;
        }
        return GLASMA_OK;
      }
    }
    return launch_following("k_tmunu launch", k_tmunu<NC, R, false>, grid, kRedThreads, 0, c->stream, a);
  }
}

template <int NC, typename R>
static int tmunu_t(glasma_ctx* c, bool hop, double* host_tab, double* dev_tab) {
  TmnArgs<R> a;
  a.U = (const typename V2T<R>::T*)c->U[c->cur];
  a.E = (const R*)c->E;
  a.QA = (const R*)c->QA;
  a.QB = (const R*)c->QB;
  a.g = c->g;
  a.dt = (R)c->p.dt;
  a.w[0] = (R)(2.0 / (c->p.a_t * c->p.a_t));
  a.w[1] = a.w[0];
  a.w[2] = (R)(2.0 / (c->p.a_z * c->p.a_z));
  a.az2 = (R)(c->p.a_z * c->p.a_z);
  const double at = c->p.a_t, az = c->p.a_z;
  a.binv[0] = 1.0 / (at * at * at * at);
  a.binv[1] = 1.0 / (at * az * at * az);
  a.hinv2[0] = 0.5 / (at * at);
  a.hinv2[1] = 0.5 / (az * az);
  a.slc = 1.0 / (at * at * az);
  a.hop = hop ? 1 : 0;
  a.zA0 = c->zA0;
  a.WA = c->WA;
  a.zB0 = c->zB0;
  a.WB = c->WB;
  // kTmunuSplit blocks per slice (fewer if the plane has fewer sites than
  // threads): the split, and with it the order of each slice's sums, depends
  // on the transverse plane alone, not on the number of slices or the device,
  // so a z slab's rows equal the whole lattice's bit for bit
  const int threads = NC == 2 && sizeof(R) == 4 && !c->links_off ? kSu2Threads : kRedThreads;
  const int64_t per_slice = (c->g.nxy + threads - 1) / threads;
  int64_t split = kTmunuSplit;
  if (split > per_slice) split = per_slice;
  if (split < 1) split = 1;
  const int64_t chunks = (per_slice + split - 1) / split;  // of a block; the last may have fewer
  split = (per_slice + chunks - 1) / chunks;
  a.per = (uint32_t)(chunks * threads);
  a.split = (int)split;
  a.part = c->tpart;
  double* tab = dev_tab ? dev_tab : c->tab;
  int st = launch_tmunu_kernel<NC, R>(c, a);
  if (st) return st;
  st = launch_following("k_tmunu_fold launch", k_tmunu_fold, (c->g.nz + 127) / 128, 128, 0, c->stream, c->tpart,
                        (int)split, c->g.nz, 1.0 / (double)c->g.nxy, tab);
  if (st || !host_tab) return st;
  st = cuda_check(cudaMemcpyAsync(host_tab, c->tab, sizeof(double) * 4 * c->g.nz, cudaMemcpyDeviceToHost,
                                  c->stream),
                  "tmunu readback");
  if (st) return st;
  return cuda_check(cudaStreamSynchronize(c->stream), "tmunu sync");
}

int launch_tmunu(glasma_ctx* c, bool hop, double* host_tab, double* dev_tab) {
  if (c->p.nc == 2)
    return c->rs == 8 ? tmunu_t<2, double>(c, hop, host_tab, dev_tab) : tmunu_t<2, float>(c, hop, host_tab, dev_tab);
  return c->rs == 8 ? tmunu_t<3, double>(c, hop, host_tab, dev_tab) : tmunu_t<3, float>(c, hop, host_tab, dev_tab);
}

}  // namespace glasma
