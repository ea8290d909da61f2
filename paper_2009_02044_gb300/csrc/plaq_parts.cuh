// The scratch between the two passes of the FP64 plaquette-centric kernels
// (k_step_plaq64.cu): per site nine algebra vectors and three plaquette norms,
// vecs[(v * NA + c) * S + slot * nxy + t] and vecs[(kPartVecs * NA + plane) * S + ...],
// S = ring * nxy, slot = z % ring.
#pragma once
#include "lattice.cuh"

namespace glasma {

// p0 of the planes xy, xz, yz, then their pAB, then pBA
enum { kP0 = 0, kPAB = 3, kPBA = 6, kPartVecs = 9 };

// doubles per site of the scratch
GL_HD constexpr int part_doubles(int na) { return kPartVecs * na + 3; }

// Force on link i of site t of slice z from the scratch.
template <int NA>
__device__ __forceinline__ void part_force(const double* part, const Geom& g, int ring, const SiteNbr& n, uint32_t t,
                                           int z, int i, const double* w, double* F) {
  const int64_t S = (int64_t)ring * g.nxy, here = (int64_t)(z % ring) * g.nxy;
#pragma unroll
  for (int c = 0; c < NA; ++c) F[c] = 0.0;
#pragma unroll 1
  for (int j = 0; j < 3; ++j) {
    if (j == i) continue;
    const int pl = i + j - 1;
    const double sgn = i < j ? -w[j] : w[j];
    if (j != 2 || z < g.nz - 1) {
      const double* p = part + (int64_t)(kP0 + pl) * NA * S + here + t;
#pragma unroll
      for (int c = 0; c < NA; ++c) F[c] = fma(sgn, p[c * S], F[c]);
    }
    if (j != 2 || z > 0) {
      const int64_t at = j == 2 ? (int64_t)((z - 1) % ring) * g.nxy + t : here + (nbr_m(n, j) - (n.s - t));
      const double* p = part + (int64_t)((i < j ? kPBA : kPAB) + pl) * NA * S + at;
#pragma unroll
      for (int c = 0; c < NA; ++c) F[c] = fma(-sgn, p[c * S], F[c]);
    }
  }
}

}  // namespace glasma
