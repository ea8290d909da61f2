// FP32 SU(2) leapfrog step with the CPIC hop, one thread per site marching
// through z (Sec. 3, Eqs. lattice_1, plaquette, lattice_2, continuity).
//
// What bounds the step is instruction issue: an SU(2) product is 16
// multiply-adds, so 13 loads with their addresses, the staples of each link by
// itself and a sine, cosine, square root and division per exponential made 673
// instructions per link (2020 per site) where memory needs 168 bytes per site.
// Here a thread updates the three links of its site and forms each plaquette
// based there once (form of k_step_plaq64.cu: A = U_b(x+a) U_a^dag(x+b), B =
// U_b^dag(x) U_a(x), corner values vec AB, vec BA and p0):
//   planes xz, yz   p0 for the links of x, vec BA for the x and y links of the
//                   next slice, which stay in registers until the thread gets
//                   there, as do U_x and U_y of the next slice;
//   plane xy        p0 alone;
//   the plaquettes at x - e_x and x - e_y give the four values that are left.
// That is 17 link loads for three links; exponential and unit norm are short
// series.  Measured against the staple kernel, ms per step: SU(2) 1024 x 128^2
// 1.01 -> 0.59, 768 x 64^2 0.192 -> 0.117, 48 x 64^2 0.0138 -> 0.0118 (below that the
// staple kernel stays, glasma_api.cu).
// The fields are loaded at the start of a slice (loaded where they are used,
// behind the stores of the link before, they cost a memory latency per link:
// 0.79 -> 0.61 ms), and the lines of the next slice are brought to L2 (0.60).
#include "dev_su2.cuh"
#include "step_link.cuh"

namespace glasma {

// Bring the line of p from device memory to L2.
__device__ __forceinline__ void prefetch_l2(const void* p) { asm volatile("prefetch.global.L2 [%0];" ::"l"(p)); }

constexpr int kSiteThreads = 256;  // consecutive transverse sites of a block, at most
constexpr int kSiteBlocks = 3;     // blocks per SM

// exp(i dt e.sigma/2) u, of unit norm: cos(th) - 1 and sin(th) / th by their
// series in th^2 <= 1/4 (remainders below 2.5e-11).
__device__ __forceinline__ Dev4 dev_evolve(Vec3 e, float dt, Dev4 u) {
  const float n2 = fma(e.x, e.x, fma(e.y, e.y, e.z * e.z));
  const float x = 0.25f * dt * dt * n2;
  float co, f;
  if (x <= 0.25f) {
    co = fma(x, fma(x, fma(x, fma(x, -1.f / 3628800.f, 1.f / 40320.f), -1.f / 720.f), 1.f / 24.f), -0.5f) * x;
    f = 0.5f * dt * fma(x, fma(x, fma(x, fma(x, 1.f / 362880.f, -1.f / 5040.f), 1.f / 120.f), -1.f / 6.f), 1.f);
  } else {
    const float nrm = sqrtf(n2);
    float sh, ch;
    sincosf(0.25f * dt * nrm, &sh, &ch);
    co = -2.f * sh * sh;
    f = 2.f * sh * ch / nrm;
  }
  const Dev4 r = dev_mul(Dev4{co, f * e.x, f * e.y, f * e.z}, u);
  const float eps = fma(r.w, r.w, fma(r.x, r.x, fma(r.y, r.y, fma(r.z, r.z, 2.f * r.w))));
  // 1 / sqrt(1 + eps) - 1 for the rounding that a link on the group carries
  const float g = eps * fma(eps, fma(eps, -0.3125f, 0.375f), -0.5f);
  const float h = 1.f + g;
  return Dev4{fma(h, r.w, g), h * r.x, h * r.y, h * r.z};
}

// E_i += dt F (+ dt J, given) and the new link of direction i at site s.
__device__ __forceinline__ Vec3 site_field(const StepArgs<float>& a, int i, int64_t s) {
  const float* e = a.E + (int64_t)(3 * i) * a.g.V + s;
  return Vec3{e[0], e[a.g.V], e[2 * a.g.V]};
}
__device__ __forceinline__ void site_update(const StepArgs<float>& a, int i, int64_t s, Vec3 F, Vec3 E, Vec3 dj,
                                            Dev4 u) {
  float* e = a.E + (int64_t)(3 * i) * a.g.V + s;
  const Vec3 v{fma(a.dt, F.x, E.x) + dj.x, fma(a.dt, F.y, E.y) + dj.y, fma(a.dt, F.z, E.z) + dj.z};
  e[0] = v.x;
  e[a.g.V] = v.y;
  e[2 * a.g.V] = v.z;
  const Dev4 n = dev_evolve(v, a.dt, u);
  reinterpret_cast<float4*>(a.Un)[(int64_t)i * a.g.V + s] = make_float4(n.w, n.z, n.y, n.x);
}

// The hop across the z link u of slice iz (step_link.cuh): dt J.
__device__ __forceinline__ Vec3 site_hop(const StepArgs<float>& a, int iz, uint32_t t, Dev4 u) {
  Vec3 dj{0.f, 0.f, 0.f};
  const int kb = iz - a.zB0, ka = iz + 1 - a.zA0;
  const int64_t nxy = a.g.nxy;
  if (kb >= 0 && kb < a.WB) {
    float* q = a.QB + (int64_t)kb * nxy + t;
    const int64_t S = (int64_t)a.WB * nxy;
    const Vec3 v{q[0], q[S], q[2 * S]};
    add3(dj, -a.az2, v);
    Dev4 d = dev_dag(u);
    const Vec3 r = turn3(d, v);
    q[0] = r.x;
    q[S] = r.y;
    q[2 * S] = r.z;
  }
  if (ka >= 0 && ka < a.WA) {
    float* q = a.QA + (int64_t)ka * nxy + t;
    const int64_t S = (int64_t)a.WA * nxy;
    const Vec3 r = turn3(u, Vec3{q[0], q[S], q[2 * S]});
    add3(dj, a.az2, r);
    q[0] = r.x;
    q[S] = r.y;
    q[2 * S] = r.z;
  }
  return dj;
}

// T threads per block (of 32, at 96 registers: 80 would spill 164 B and take 13.2
// us on 4099 x 32 x 1)
template <int T>
__global__ void __launch_bounds__(T, T == 32 ? 20 : kSiteBlocks * kSiteThreads / T) k_step_leapfrog_site(StepArgs<float> a, int zlen,
                                                                                 int zhi) {
  follow();
  const Geom& g = a.g;
  const uint32_t t = blockIdx.x * T + threadIdx.x;
  if (t >= (uint32_t)g.nxy) return;
  const uint32_t nx = (uint32_t)g.nx, ny = (uint32_t)g.ny, iy = t / nx, ix = t - iy * nx;
  const uint32_t xp = ix + 1 == nx ? 0 : ix + 1, xm = ix == 0 ? nx - 1 : ix - 1;
  const uint32_t yp = (iy + 1 == ny ? 0 : iy + 1) * nx, ym = (iy == 0 ? ny - 1 : iy - 1) * nx, y0 = iy * nx;
  const uint32_t txp = y0 + xp, txm = y0 + xm, typ = yp + ix, tym = ym + ix, txmyp = yp + xm, txpym = ym + xp;
  const int z0 = a.zlo + (int)blockIdx.y * zlen, z1 = min(z0 + zlen, zhi);
  const float wt = a.w[0], wz = a.w[2];
  // The slice below the first one is entered only for what it gives to its
  // next slice, by the same instructions, so that results do not depend on
  // where the blocks' ranges begin.
  int z = z0 > 0 ? z0 - 1 : 0;
  const float4* Ux = links_of(a.U) + (int64_t)z * g.nxy;
  Dev4 ux = dev_load_free(Ux + t), uy = dev_load_free(Ux + g.V + t);
  Vec3 cx{0.f, 0.f, 0.f}, cy{0.f, 0.f, 0.f};  // vec BA of the planes xz, yz of the slice below
#pragma unroll 1
  for (; z < z1; ++z, Ux += g.nxy) {
    const float4 *Uy = Ux + g.V, *Uz = Uy + g.V;
    const bool up = z < g.nz - 1, now = z >= z0;
    const int64_t s = (int64_t)z * g.nxy + t;
    Dev4 uz{0.f, 0.f, 0.f, 0.f}, nux = ux, nuy = uy;
    Vec3 Fx{0.f, 0.f, 0.f}, Fy = Fx, Fz = Fx, nx_{0.f, 0.f, 0.f}, ny_ = nx_;
    if (z + 2 < g.nz) {
      prefetch_l2(Ux + 2 * g.nxy + t);
      prefetch_l2(Uy + 2 * g.nxy + t);
      prefetch_l2(Uz + g.nxy + t);
#pragma unroll
      for (int c = 0; c < 9; ++c) prefetch_l2(a.E + (int64_t)c * g.V + s + g.nxy);
    }
    Vec3 Ex{0.f, 0.f, 0.f}, Ey = Ex, Ez = Ex;
    if (now) {
      Ex = site_field(a, 0, s);
      Ey = site_field(a, 1, s);
      Ez = site_field(a, 2, s);
    }
    if (up) {
      uz = dev_load_free(Uz + t);
      nux = dev_load_free(Ux + g.nxy + t);
      nuy = dev_load_free(Uy + g.nxy + t);
      // planes xz and yz based here: A = U_z(x+a) U_a^dag(x+z), B = U_z^dag U_a
      {
        const Dev4 A = dev_mul(dev_load_free(Uz + txp), dev_dag(nux)), B = dev_mul(dev_dag(uz), ux);
        const Vec3 m = sym3(A, B), c = cross3(vec3(A), vec3(B));
        nx_ = Vec3{m.x + c.x, m.y + c.y, m.z + c.z};
        const Vec3 p = turn3(ux, Vec3{m.x - c.x, m.y - c.y, m.z - c.z});
        add3(Fx, -wz, p);
        add3(Fz, wt, p);
      }
      {
        const Dev4 A = dev_mul(dev_load_free(Uz + typ), dev_dag(nuy)), B = dev_mul(dev_dag(uz), uy);
        const Vec3 m = sym3(A, B), c = cross3(vec3(A), vec3(B));
        ny_ = Vec3{m.x + c.x, m.y + c.y, m.z + c.z};
        const Vec3 p = turn3(uy, Vec3{m.x - c.x, m.y - c.y, m.z - c.z});
        add3(Fy, -wz, p);
        add3(Fz, wt, p);
      }
    }
    if (now) {
      add3(Fx, wz, cx);
      add3(Fy, wz, cy);
      // plane xy based here: Im tr t (U_x U_y(x+x)) (U_y U_x(x+y))^dag
      {
        const Dev4 A = dev_mul(ux, dev_load_free(Uy + txp)), B = dev_mul(uy, dev_load_free(Ux + typ));
        const Vec3 p = vec_ab(A, dev_dag(B));
        add3(Fx, -wt, p);
        add3(Fy, wt, p);
      }
      // plaquettes at x - e_x: vec AB of the planes xy (link y) and xz (link z)
      {
        const Dev4 vx = dev_load_free(Ux + txm);
        add3(Fy, -wt, vec_ab(dev_mul(uy, dev_dag(dev_load_free(Ux + txmyp))), dev_mul(dev_dag(dev_load_free(Uy + txm)), vx)));
        if (up)
          add3(Fz, -wt,
               vec_ab(dev_mul(uz, dev_dag(dev_load_free(Ux + g.nxy + txm))), dev_mul(dev_dag(dev_load_free(Uz + txm)), vx)));
      }
      // plaquettes at x - e_y: vec BA of the plane xy (link x), vec AB of yz (link z)
      {
        const Dev4 vy = dev_load_free(Uy + tym);
        add3(Fx, wt, vec_ab(dev_mul(dev_dag(vy), dev_load_free(Ux + tym)), dev_mul(dev_load_free(Uy + txpym), dev_dag(ux))));
        if (up)
          add3(Fz, -wt,
               vec_ab(dev_mul(uz, dev_dag(dev_load_free(Uy + g.nxy + tym))), dev_mul(dev_dag(dev_load_free(Uz + tym)), vy)));
      }
      const Vec3 zero{0.f, 0.f, 0.f};
      site_update(a, 0, s, Fx, Ex, zero, ux);
      site_update(a, 1, s, Fy, Ey, zero, uy);
      if (up) site_update(a, 2, s, Fz, Ez, a.hop ? site_hop(a, z, t, uz) : zero, uz);
    }
    cx = nx_;
    cy = ny_;
    ux = nux;
    uy = nuy;
  }
}

// Threads of a block, all on one slice: the most that leave at most a tenth more
// of them without a site than the fewest do.  Planes of 32 sites ran one warp of
// eight per block of 256 (us per step: 4099 x 32 x 1 14.6 -> 9.3, 65535 x 1 x 3 168 ->
// 76, 2048 x 8^2 12.0 -> 9.2, 512 x 17^2 13.2 -> 11.2).
// Threads numbered through several ranges of slices fill any block, but then a
// slice is a thread's own number: 80 registers and spills, 1024 x 128^2 0.59 ->
// 0.82 ms.
static int site_threads(int64_t nxy) {
  const int64_t least = (nxy + 31) / 32 * 32;
  static_assert(kSiteThreads == 256, "launch_step_site lists the kernels");
  for (int b = kSiteThreads; b > 32; b /= 2)
    if (10 * ((nxy + b - 1) / b * b) <= 11 * least) return b;
  return 32;
}

int launch_step_site(glasma_ctx* c, bool hop) {
  if (c->rs != 4 || c->p.nc != 2) return set_error(GLASMA_ERR_INTERNAL, "the site kernel is FP32 SU(2) only");
  StepArgs<float> a;
  a.U = (const float2*)c->U[c->cur];
  a.Un = (float2*)c->U[1 - c->cur];
  a.E = (float*)c->E;
  a.QA = (float*)c->QA;
  a.QB = (float*)c->QB;
  a.g = c->g;
  a.dt = (float)c->p.dt;
  a.w[0] = (float)(2.0 / (c->p.a_t * c->p.a_t));
  a.w[1] = a.w[0];
  a.w[2] = (float)(2.0 / (c->p.a_z * c->p.a_z));
  a.az2 = (float)(c->p.a_z * c->p.a_z);
  a.hop = hop ? 1 : 0;
  a.zA0 = c->zA0;
  a.WA = c->WA;
  a.zB0 = c->zB0;
  a.WB = c->WB;
  a.zlo = c->lo;
  const int threads = site_threads(c->g.nxy);
  // about four waves of blocks; a range of n slices enters n + 1
  const int64_t tiles = (c->g.nxy + threads - 1) / threads, nsl = c->hi - c->lo;
  int64_t zlen = tiles * threads * nsl / (4 * (int64_t)c->sms * kSiteBlocks * kSiteThreads);
  if (zlen < 1) zlen = 1;
  if (zlen > 32) zlen = 32;
  auto kernel = threads == 256   ? k_step_leapfrog_site<256>
                : threads == 128 ? k_step_leapfrog_site<128>
                : threads == 64  ? k_step_leapfrog_site<64>
                                 : k_step_leapfrog_site<32>;
  return launch_following("k_step_leapfrog_site launch", kernel,
                          dim3((unsigned)tiles, (unsigned)((nsl + zlen - 1) / zlen)), threads, 0, c->stream, a,
                          (int)zlen, c->hi);
}

}  // namespace glasma
