// FP64 leapfrog step with the CPIC hop, plaquette-centric form in two passes
// (Sec. 3, Eqs. lattice_1, plaquette, lattice_2, continuity).
//
// GB300 does two FP64 multiply-adds per SM and clock, so the FP64 step is
// bound by their number, and device memory has time to spare (SU(3): some 2300
// multiply-adds against 1.9 KB per site, 4.5 us against 0.3 us per 1000 sites).
// Hence every plaquette is formed once, by a thread of its own, and what it
// contributes to its four links goes through a scratch array:
//   k_step_plaq_parts  one thread per (site, plane): A = U_b(x+a) U_a^dag(x+b),
//                      B = U_b^dag(x) U_a(x); the projections of the loop at
//                      its corners, pAB (corner x+a, link b), pBA (corner x+b,
//                      link a) and p0 = U_a pAB U_a^dag (corner x);
//   k_step_plaq_links  one thread per link: F_a(x) = sum over the other
//                      directions of -+ w p0 and +- w pAB or pBA of the
//                      plaquette below, then update_link.
// Two products, two projections and one transport of an algebra vector are
// 510 multiply-adds per SU(3) plaquette (594 with p0 from a third product; 534,
// and 0.449 and 10.1 ms per step in the list below, with all rows of A and B by
// their sums) and 68 per SU(2) plaquette, whose pAB and pBA differ in a cross
// product's sign only.  Against a block that marches through z with a halo row and a
// warm-up slice in shared memory, no work is done twice, and threads of both
// passes are numbered straight through the sites, so a small lattice spreads
// over all SMs and a plane of any size fills its warps.
// Measured against the marching form, ms per step: SU(2) 128 x 16^2 0.191 ->
// 0.031, 512 x 64^2 2.45 -> 1.6; SU(3) 160 x 24^2 1.47 -> 0.431, 512 x 64^2 12.3 ->
// 9.5 (with the series exponentials of su_n.cuh, which came with it).
//
// The scratch holds a ring of slices (nine vectors per site).  A lattice whose
// vectors pass kPartsBytes is stepped in chunks of slices; chunk k's parts
// pass overwrites neither the parts its links pass reads from the slice below
// nor any other, as the ring has one slice more than a chunk.  Every value is
// formed by the same instructions whatever the chunk, so results do not
// depend on it.
#include "plaq_parts.cuh"
#include "step_link.cuh"

namespace glasma {

// the scratch aims at this size (it then stays in the L2 cache between the
// two passes) and holds two slices at least
constexpr size_t kPartsBytes = (size_t)64 << 20;
constexpr int kPartsThreads = 64;  // 128 left a sixth of the SMs' FP64 pipes idle on 128 x 16^2

struct PartsArgs {
  const double2* U;
  double* part;
  Geom g;
  int zfirst, z0;  // slices zfirst..: one before z0 where a slab's halo has to be added
  int ring;        // slices of the scratch
  uint32_t sites;  // sites of the launch
};

template <int NC>
struct PlaqCorners;

template <>
struct PlaqCorners<3> {
  typedef Group<3, double> G;
  typedef G::M M;
  // A product of links is a link: conj(row 0 x row 1) is its third row.
  __device__ __forceinline__ static void third_row(M& t) {
#pragma unroll
    for (int k = 0; k < 3; ++k) {
      const int k1 = (k + 1) % 3, k2 = (k + 2) % 3;
      const cplx<double> a1 = t.m[k1], a2 = t.m[k2], b1 = t.m[3 + k1], b2 = t.m[3 + k2];
      const cplx<double> c = fma_c(cplx<double>{-a2.re, -a2.im}, b1, a1 * b2);
      t.m[6 + k] = cj(c);
    }
  }
  __device__ __forceinline__ static M mul_d(const M& x, const M& y) {
    M t;
#pragma unroll
    for (int i = 0; i < 2; ++i)
#pragma unroll
      for (int j = 0; j < 3; ++j) {
        cplx<double> acc = mulc(x.m[3 * i], y.m[3 * j]);
        acc = fma_cj(x.m[3 * i + 1], y.m[3 * j + 1], acc);
        t.m[3 * i + j] = fma_cj(x.m[3 * i + 2], y.m[3 * j + 2], acc);
      }
    third_row(t);
    return t;
  }
  __device__ __forceinline__ static M d_mul(const M& x, const M& y) {
    M t;
#pragma unroll
    for (int i = 0; i < 2; ++i)
#pragma unroll
      for (int j = 0; j < 3; ++j) {
        cplx<double> acc = mulc(y.m[j], x.m[i]);
        acc = fma_cj(y.m[3 + j], x.m[3 + i], acc);
        t.m[3 * i + j] = fma_cj(y.m[6 + j], x.m[6 + i], acc);
      }
    third_row(t);
    return t;
  }
  __device__ __forceinline__ static void both(const G::M& A, const G::M& B, double* ab, double* ba) {
    G::proj_mul(A, B, ab);
    G::proj_mul(B, A, ba);
  }
};

template <>
struct PlaqCorners<2> {
  typedef Group<2, double> G;
  typedef G::M M;
  __device__ __forceinline__ static M mul_d(const M& x, const M& y) { return G::mul_d(x, y); }
  __device__ __forceinline__ static M d_mul(const M& x, const M& y) { return G::d_mul(x, y); }
  // A = p + i a.sigma, B = q + i b.sigma: AB and BA have the vector parts
  // p b + q a -+ a x b
  __device__ __forceinline__ static void both(const G::M& A, const G::M& B, double* ab, double* ba) {
    const double p = A.a.re, q = B.a.re;
    const double a[3] = {A.b.im, A.b.re, A.a.im}, b[3] = {B.b.im, B.b.re, B.a.im};
#pragma unroll
    for (int k = 0; k < 3; ++k) {
      const int k1 = (k + 1) % 3, k2 = (k + 2) % 3;
      const double s = fma(p, b[k], q * a[k]), c = fma(a[k1], b[k2], -(a[k2] * b[k1]));
      ab[k] = s - c;
      ba[k] = s + c;
    }
  }
};

// Plane pl of site idx of the launch.  NORM: also ||A - B^dag||_F^2 =
// 2 (N - Re tr of the loop), for T^{mu nu}.
template <int NC, bool NORM>
__device__ __forceinline__ void parts_of(const PartsArgs& a, uint32_t idx, int pl) {
  typedef Group<NC, double> G;
  typedef LinkIO<NC, double> IO;
  typedef typename G::M M;
  constexpr int NA = G::NA;
  if (idx >= a.sites) return;
  const Geom& g = a.g;
  const uint32_t nxy = (uint32_t)g.nxy, dz = idx / nxy, t = idx - dz * nxy;
  const int z = a.zfirst + (int)dz;
  const bool below = z < a.z0;  // only what reaches the slice above is wanted
  if (pl == 0 ? below : z >= g.nz - 1) return;
  const int da = pl == 2 ? 1 : 0, db = pl == 0 ? 1 : 2;
  const SiteNbr n = site_nbr_tz(g, t, z);
  const int64_t S = (int64_t)a.ring * nxy;
  double* out = a.part + (int64_t)(z % a.ring) * nxy + t;
  const M ua = IO::template load<double>(a.U, da, g.V, n.s);
  const M A = PlaqCorners<NC>::mul_d(IO::template load<double>(a.U, db, g.V, nbr_p(n, da)),
                                     IO::template load<double>(a.U, da, g.V, nbr_p(n, db)));
  const M B = PlaqCorners<NC>::d_mul(IO::template load<double>(a.U, db, g.V, n.s), ua);
  if (NORM) out[(kPartVecs * NA + pl) * S] = G::fro2_diff(A, G::dag(B));
  double ab[NA], ba[NA];
  PlaqCorners<NC>::both(A, B, ab, ba);
#pragma unroll
  for (int c = 0; c < NA; ++c) out[((kPBA + pl) * NA + c) * S] = ba[c];
  if (below) return;
#pragma unroll
  for (int c = 0; c < NA; ++c) out[((kPAB + pl) * NA + c) * S] = ab[c];
  G::adj(ua, ab);
#pragma unroll
  for (int c = 0; c < NA; ++c) out[((kP0 + pl) * NA + c) * S] = ab[c];
}

template <int NC, bool NORM>
__global__ void __launch_bounds__(kPartsThreads, 4) k_step_plaq_parts(PartsArgs a) {
  follow_last();
  parts_of<NC, NORM>(a, blockIdx.x * kPartsThreads + threadIdx.x, (int)blockIdx.y);
}

struct PartLinksArgs {
  StepArgs<double> s;
  const double* part;
  int z0;
  int ring;
  uint32_t sites;
};

// Link i of site idx of the launch.
template <int NC>
__device__ __forceinline__ void links_of_parts(const PartLinksArgs& pa, uint32_t idx, int i) {
  constexpr int NA = Group<NC, double>::NA;
  if (idx >= pa.sites) return;
  const StepArgs<double>& a = pa.s;
  const Geom& g = a.g;
  const uint32_t nxy = (uint32_t)g.nxy, dz = idx / nxy, t = idx - dz * nxy;
  const int z = pa.z0 + (int)dz;
  if (i == 2 && z == g.nz - 1) return;  // no z link on the last slice
  const SiteNbr n = site_nbr_tz(g, t, z);
  double F[NA];
  part_force<NA>(pa.part, g, pa.ring, n, t, z, i, a.w, F);
  update_link<NC, double>(a, i, t, z, n.s, F);
}

template <int NC>
__global__ void __launch_bounds__(kPartsThreads, 4) k_step_plaq_links(PartLinksArgs pa) {
  follow_last();
  links_of_parts<NC>(pa, blockIdx.x * kPartsThreads + threadIdx.x, (int)blockIdx.y);
}

// The two passes of several events of one geometry, whole lattices in their
// scratch, blockIdx.z the event: events that do not fill the GPU cost a launch
// each otherwise (us per step, 64 events, SU(2) 40 x 4^2 618 -> 44, SU(3) 3250 -> 310;
// the graph's staple form 124 and 786).
struct PartsEvent {
  void* U[2];  // this step's links and the next step's
  double *part, *E, *QA, *QB;
  int zA0, WA, zB0, WB, hop;
};
struct PartsGroup {
  PartLinksArgs l;
  PartsEvent ev[kMaxBatch];
};

template <int NC>
__global__ void __launch_bounds__(kPartsThreads, 4) k_step_plaq_parts_group(const __grid_constant__ PartsGroup b) {
  follow_last();
  const PartsEvent& e = b.ev[blockIdx.z];
  PartsArgs a;
  a.U = (const double2*)e.U[0];
  a.part = e.part;
  a.g = b.l.s.g;
  a.zfirst = a.z0 = 0;
  a.ring = b.l.ring;
  a.sites = b.l.sites;
  parts_of<NC, false>(a, blockIdx.x * kPartsThreads + threadIdx.x, (int)blockIdx.y);
}

template <int NC>
__global__ void __launch_bounds__(kPartsThreads, 4) k_step_plaq_links_group(const __grid_constant__ PartsGroup b) {
  follow_last();
  const PartsEvent& e = b.ev[blockIdx.z];
  PartLinksArgs l = b.l;
  l.part = e.part;
  l.s.U = (const double2*)e.U[0];
  l.s.Un = (double2*)e.U[1];
  l.s.E = e.E;
  l.s.QA = e.QA;
  l.s.QB = e.QB;
  l.s.hop = e.hop;
  l.s.zA0 = e.zA0;
  l.s.WA = e.WA;
  l.s.zB0 = e.zB0;
  l.s.WB = e.WB;
  links_of_parts<NC>(l, blockIdx.x * kPartsThreads + threadIdx.x, (int)blockIdx.y);
}

// The scratch of an FP64 leapfrog context.  Where the allocator refuses it, half
// the slices are tried, down to two: results do not depend on the ring, where
// stepping with another kernel would change their rounding (and on one rank of
// several, the slabs).  Two slices are a part 1.2 / nz (SU(3)) or 2.9 / nz (SU(2))
// of the links and fields, less than the initial state's scratch, which is free by
// then, on lattices of 20 slices.
int parts_alloc(glasma_ctx* c) {
  if (c->rs != 8 || c->p.scheme != GLASMA_LEAPFROG) return GLASMA_OK;
  const size_t slice = sizeof(double) * (size_t)part_doubles(c->na) * (size_t)c->g.nxy;
  const size_t whole = (size_t)(c->hi - c->lo) + 1;
  size_t r = kPartsBytes / slice;
  if (r > whole) r = whole;
  if (r < 2) r = 2;
  while (!(c->part = (double*)ctx_alloc(c, slice * r))) {
    if (r == 2) return set_error(GLASMA_ERR_OOM, "step scratch allocation failed");
    r = r / 2 > 2 ? r / 2 : 2;
  }
  c->ring = (int)r;
  return GLASMA_OK;
}

// The parts of the slices [z0, z1), of z0 - 1 as well with `below`; at most
// ring - 1 slices.
template <int NC, bool NORM>
static int launch_parts_pass(glasma_ctx* c, int z0, int z1, bool below) {
  PartsArgs p;
  p.U = (const double2*)c->U[c->cur];
  p.part = c->part;
  p.g = c->g;
  p.ring = c->ring;
  p.z0 = z0;
  p.zfirst = below ? z0 - 1 : z0;
  p.sites = (uint32_t)((z1 - p.zfirst) * c->g.nxy);
  return launch_following("k_step_plaq_parts launch", k_step_plaq_parts<NC, NORM>,
                          dim3((p.sites + kPartsThreads - 1) / kPartsThreads, 3), kPartsThreads, 0, c->stream, p);
}

int launch_parts_norms(glasma_ctx* c, int z0, int z1) {
  return c->p.nc == 2 ? launch_parts_pass<2, true>(c, z0, z1, false) : launch_parts_pass<3, true>(c, z0, z1, false);
}

static void links_args(const glasma_ctx* c, bool hop, PartLinksArgs& l) {
  StepArgs<double>& a = l.s;
  a.U = (const double2*)c->U[c->cur];
  a.Un = (double2*)c->U[1 - c->cur];
  a.E = (double*)c->E;
  a.QA = (double*)c->QA;
  a.QB = (double*)c->QB;
  a.g = c->g;
  a.dt = c->p.dt;
  a.w[0] = 2.0 / (c->p.a_t * c->p.a_t);
  a.w[1] = a.w[0];
  a.w[2] = 2.0 / (c->p.a_z * c->p.a_z);
  a.az2 = c->p.a_z * c->p.a_z;
  a.hop = hop ? 1 : 0;
  a.zA0 = c->zA0;
  a.WA = c->WA;
  a.zB0 = c->zB0;
  a.WB = c->WB;
  a.zlo = c->lo;
  l.part = c->part;
  l.ring = c->ring;
}

template <int NC>
static int launch_parts_t(glasma_ctx* c, bool hop, int zlen, int* launches) {
  PartLinksArgs l;
  links_args(c, hop, l);
  if (zlen <= 0 || zlen > l.ring - 1) zlen = l.ring - 1;
  for (int z0 = c->lo; z0 < c->hi; z0 += zlen) {
    const int z1 = z0 + zlen < c->hi ? z0 + zlen : c->hi;
    l.z0 = z0;
    l.sites = (uint32_t)((z1 - z0) * c->g.nxy);
    int st = launch_parts_pass<NC, false>(c, z0, z1, z0 == c->lo && z0 > 0);
    if (!st)
      st = launch_following("k_step_plaq_links launch", k_step_plaq_links<NC>,
                            dim3((l.sites + kPartsThreads - 1) / kPartsThreads, 3), kPartsThreads, 0, c->stream, l);
    if (st) return st;
    *launches += 2;
  }
  return GLASMA_OK;
}

// Events of the context's geometry that share its launches: as many as keep
// their scratches in the L2 cache together, 1 where one event's ring is shorter
// than its lattice.
int parts_group_size(const glasma_ctx* c) {
  if (c->slab || c->ring != c->g.nz + 1 || c->step_zlen != 0) return 1;
  const size_t n = kPartsBytes / (sizeof(double) * (size_t)part_doubles(c->na) * (size_t)c->g.nxy * (size_t)c->ring);
  return n < 1 ? 1 : n > (size_t)kMaxBatch ? kMaxBatch : (int)n;
}

template <int NC>
static int launch_group_t(glasma_ctx* const* c, int n, const bool* hop, int* launches) {
  PartsGroup b;
  links_args(c[0], false, b.l);
  b.l.z0 = 0;
  b.l.sites = (uint32_t)c[0]->g.V;
  for (int k = 0; k < n; ++k) {
    PartsEvent& e = b.ev[k];
    e.U[0] = c[k]->U[c[k]->cur];
    e.U[1] = c[k]->U[1 - c[k]->cur];
    e.part = c[k]->part;
    e.E = (double*)c[k]->E;
    e.QA = (double*)c[k]->QA;
    e.QB = (double*)c[k]->QB;
    e.zA0 = c[k]->zA0;
    e.WA = c[k]->WA;
    e.zB0 = c[k]->zB0;
    e.WB = c[k]->WB;
    e.hop = hop[k] ? 1 : 0;
  }
  const dim3 grid((b.l.sites + kPartsThreads - 1) / kPartsThreads, 3, (unsigned)n);
  int st = launch_following("k_step_plaq_parts_group launch", k_step_plaq_parts_group<NC>, grid, kPartsThreads, 0,
                            c[0]->stream, b);
  if (!st)
    st = launch_following("k_step_plaq_links_group launch", k_step_plaq_links_group<NC>, grid, kPartsThreads, 0,
                          c[0]->stream, b);
  *launches += 2;
  return st;
}

// One step of n events of equal geometry and stream, n at most parts_group_size
// of each
int launch_parts_group(glasma_ctx* const* c, int n, const bool* hop, int* launches) {
  return c[0]->p.nc == 2 ? launch_group_t<2>(c, n, hop, launches) : launch_group_t<3>(c, n, hop, launches);
}

// zlen: slices per chunk (0: as many as the scratch holds)
int launch_step_parts(glasma_ctx* c, bool hop, int zlen, int* launches) {
  return c->p.nc == 2 ? launch_parts_t<2>(c, hop, zlen, launches) : launch_parts_t<3>(c, hop, zlen, launches);
}

}  // namespace glasma
