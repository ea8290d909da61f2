// FP32 SU(2) links as quaternions of their deviation from 1 (link_alg.cuh):
// (w, x, y, z) of alpha = 1 + w + i z, beta = y + i x, one 16-byte word each.
// Every product is (1+a)(1+b) - 1 = b + a (1+b), so rounding stays of the size
// of the deviations.
#pragma once
#include <cuda_runtime.h>

namespace glasma {

struct Dev4 {  // a link, less 1
  float w, x, y, z;
};

// Loads for kernels that begin with follow(), which are placed while the step
// before them still writes the links: no read-only loads, those are for data that
// nothing writes in the kernel's lifetime.
__device__ __forceinline__ Dev4 dev_of(float4 v) {  // (alpha.re - 1, alpha.im, beta.re, beta.im)
  return Dev4{v.x, v.w, v.z, v.y};
}
__device__ __forceinline__ Dev4 dev_load(const float4* p) { return dev_of(*p); }
// The same for a kernel that writes no link of the array it reads: the load need
// not keep its place among the kernel's stores, as dev_load does (1024 x 128^2
// 0.601 for 0.593 ms per step).  links_of, on whose result every address depends,
// keeps it behind follow()'s wait.
__device__ __forceinline__ const float4* links_of(const float2* U) {
  const float4* p = reinterpret_cast<const float4*>(U);
  asm volatile("" : "+l"(p));
  return p;
}
__device__ __forceinline__ Dev4 dev_load_free(const float4* p) {
  float4 v;
  asm("ld.global.v4.f32 {%0, %1, %2, %3}, [%4];" : "=f"(v.x), "=f"(v.y), "=f"(v.z), "=f"(v.w) : "l"(p));
  return dev_of(v);
}
__device__ __forceinline__ Dev4 dev_dag(Dev4 a) { return Dev4{a.w, -a.x, -a.y, -a.z}; }
// (w + i a.s)(v + i b.s) = (w v - a.b) + i (w b + v a - a x b).s, the products
// of two deviations first, so that each entry rounds twice at their own size;
// rounding four times (dev_mulq, for T^{mu nu}, whose squares are averaged)
// the step took 0.596 for 0.603 ms on 1024 x 128^2, with 1.4 times the error of E
// and 1.3 times that of U
__device__ __forceinline__ Dev4 dev_mul(Dev4 a, Dev4 b) {
  const float v = 1.f + b.w, u = 1.f + a.w;
  return Dev4{fma(a.w, v, fma(-a.x, b.x, fma(-a.y, b.y, -a.z * b.z))) + b.w,
              fma(u, b.x, fma(v, a.x, fma(-a.y, b.z, a.z * b.y))),
              fma(u, b.y, fma(v, a.y, fma(-a.z, b.x, a.x * b.z))),
              fma(u, b.z, fma(v, a.z, fma(-a.x, b.y, a.y * b.x)))};
}
__device__ __forceinline__ Dev4 dev_mulq(Dev4 a, Dev4 b) {
  const float v = 1.f + b.w;
  return Dev4{fma(a.w, v, fma(-a.x, b.x, fma(-a.y, b.y, fma(-a.z, b.z, b.w)))),
              fma(a.w, b.x, fma(v, a.x, fma(-a.y, b.z, fma(a.z, b.y, b.x)))),
              fma(a.w, b.y, fma(v, a.y, fma(-a.z, b.x, fma(a.x, b.z, b.y)))),
              fma(a.w, b.z, fma(v, a.z, fma(-a.x, b.y, fma(a.y, b.x, b.z))))};
}

struct Vec3 {
  float x, y, z;
};
__device__ __forceinline__ Vec3 cross3(Vec3 a, Vec3 b) {
  return Vec3{fma(a.y, b.z, -(a.z * b.y)), fma(a.z, b.x, -(a.x * b.z)), fma(a.x, b.y, -(a.y * b.x))};
}
__device__ __forceinline__ void add3(Vec3& f, float w, Vec3 v) {
  f.x = fma(w, v.x, f.x);
  f.y = fma(w, v.y, f.y);
  f.z = fma(w, v.z, f.z);
}
// the part of vec AB and vec BA that is the same, a (1 + B.w) + b (1 + A.w)
__device__ __forceinline__ Vec3 sym3(Dev4 A, Dev4 B) {
  return Vec3{fma(A.w, B.x, fma(B.w, A.x, A.x + B.x)), fma(A.w, B.y, fma(B.w, A.y, A.y + B.y)),
              fma(A.w, B.z, fma(B.w, A.z, A.z + B.z))};
}
__device__ __forceinline__ Vec3 vec3(Dev4 a) { return Vec3{a.x, a.y, a.z}; }
// vec AB = sym - a x b
__device__ __forceinline__ Vec3 vec_ab(Dev4 A, Dev4 B) {
  const Vec3 s = sym3(A, B), c = cross3(vec3(A), vec3(B));
  return Vec3{s.x - c.x, s.y - c.y, s.z - c.z};
}
// v <- U v U^+, operation for operation Group<2>::rotate: a slab's halo charge
// hops there (k_slab_halo_hop), and its owner's here
__device__ __forceinline__ Vec3 turn3(Dev4 u, Vec3 v) {
  const Vec3 c = cross3(vec3(u), v);
  const float w = 1.f + u.w;
  return Vec3{fma(2.f, fma(u.y, c.z, fma(-u.z, c.y, -(w * c.x))), v.x),
              fma(2.f, fma(u.z, c.x, fma(-u.x, c.z, -(w * c.y))), v.y),
              fma(2.f, fma(u.x, c.y, fma(-u.y, c.x, -(w * c.z))), v.z)};
}

}  // namespace glasma
