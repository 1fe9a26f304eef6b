// Particle-mask predicate and unit-cell lookup shared by the density kernel,
// the fused density + transform row pass and the adjoint row pass (Sec. 2.3).
#pragma once

#include <math.h>
#include <string.h>

#include "ur_common.cuh"

struct ShapeArgs {
  int kind;
  float cx, cy, cz, s;
  float r[9];
  float rb2;  // rows (y, z) with fl(dy dy + dz dz) > rb2 have a zero mask at every x (infinity: unknown)
};

// Per-row part of the predicate: the y and z terms are fixed along a row, so
// they are formed once and only the x term varies.  Every product and sum is rounded separately (no
// contraction), in the order of the ur_build_density contract.
struct RowMask {
  int kind;
  float s, s2;
  float dy2, dz2;      // fl(dy*dy), fl(dz*dz)
  float cx;
  float ry[3], rz[3];  // fl(R[1][a] dy), fl(R[2][a] dz)
  float r0[3];
  __device__ __forceinline__ void init(const ShapeArgs& sh, int y, int z) {
    kind = sh.kind;
    s = sh.s;
    s2 = __fmul_rn(sh.s, sh.s);
    cx = sh.cx;
    const float dy = __fsub_rn((float)y, sh.cy);
    const float dz = __fsub_rn((float)z, sh.cz);
    dy2 = __fmul_rn(dy, dy);
    dz2 = __fmul_rn(dz, dz);
#pragma unroll
    for (int a = 0; a < 3; ++a) {
      r0[a] = sh.r[a];
      ry[a] = __fmul_rn(sh.r[3 + a], dy);
      rz[a] = __fmul_rn(sh.r[6 + a], dz);
    }
  }
  // True when the mask is zero at every x of the row (row_outside)
  __device__ __forceinline__ bool empty(const ShapeArgs& sh) const { return __fadd_rn(dy2, dz2) > sh.rb2; }
  __device__ __forceinline__ bool sphere_empty() const {
    return kind == UR_SHAPE_SPHERE && __fadd_rn(dy2, dz2) > s2;
  }
  // Signed coordinate of axis a at x, rounded as in at; nondecreasing or nonincreasing in x,
  // since rounding to nearest is monotone
  __device__ __forceinline__ float coord(int a, float dx) const {
    return __fadd_rn(__fadd_rn(__fmul_rn(r0[a], dx), ry[a]), rz[a]);
  }
  // Mask values of the W voxels from x on.  Sphere and cube predicates hold on an interval of the
  // row (each side of the sphere's centre and each cube coordinate is monotone in x, roundings
  // included), so a group whose end voxels are both inside is inside, and one whose end voxels fail
  // the same side of the predicate is outside; other groups, and the octahedron (a rounded sum of
  // three coordinates, not an interval), take every voxel.
  template <int W>
  __device__ __forceinline__ void group(int x, float (&m)[W]) const {
    if constexpr (W > 2) {
      if (kind == UR_SHAPE_ALL) {
#pragma unroll
        for (int e = 0; e < W; ++e) m[e] = 1.f;
        return;
      }
      bool in = false, out = false;
      const float da = __fsub_rn((float)x, cx), db = __fsub_rn((float)(x + W - 1), cx);
      if (kind == UR_SHAPE_SPHERE) {
        const bool ia = __fadd_rn(__fadd_rn(__fmul_rn(da, da), dy2), dz2) <= s2;
        const bool ib = __fadd_rn(__fadd_rn(__fmul_rn(db, db), dy2), dz2) <= s2;
        in = ia && ib;
        out = !ia && !ib && (da >= 0.f || db <= 0.f);
      } else if (kind == UR_SHAPE_CUBE) {
        in = true;
#pragma unroll
        for (int a = 0; a < 3; ++a) {
          const float ta = coord(a, da), tb = coord(a, db);
          in = in && fabsf(ta) <= s && fabsf(tb) <= s;
          out = out || (ta > s && tb > s) || (ta < -s && tb < -s);
        }
      }
      if (in || out) {
#pragma unroll
        for (int e = 0; e < W; ++e) m[e] = in ? 1.f : 0.f;
        return;
      }
    }
#pragma unroll
    for (int e = 0; e < W; ++e) m[e] = at(x + e);
  }
  __device__ __forceinline__ float at(int x) const {
    if (kind == UR_SHAPE_ALL) return 1.f;
    const float dx = __fsub_rn((float)x, cx);
    if (kind == UR_SHAPE_SPHERE) return __fadd_rn(__fadd_rn(__fmul_rn(dx, dx), dy2), dz2) <= s2 ? 1.f : 0.f;
    float p[3];
#pragma unroll
    for (int a = 0; a < 3; ++a) p[a] = fabsf(__fadd_rn(__fadd_rn(__fmul_rn(r0[a], dx), ry[a]), rz[a]));
    if (kind == UR_SHAPE_CUBE) return (p[0] <= s && p[1] <= s && p[2] <= s) ? 1.f : 0.f;
    return __fadd_rn(__fadd_rn(p[0], p[1]), p[2]) <= s ? 1.f : 0.f;
  }
};

// Row (y, z) outside the particle: its mask is zero at every x.  Sphere: rb2 = fl(s s); rounding
// to nearest is monotone and fl(dx*dx) >= 0, so fl(fl(fl(dx*dx) + dy2) + dz2) >= fl(dy2 + dz2) for
// every x.  Cube and octahedron: rb2 is the square of a radius beyond their vertices
// (ur_shape_args).
// (Host-callable, for row_range and its test; the volatile results keep the host compiler from
// contracting the product and the sum.)
UR_HD __forceinline__ bool row_outside(float cy, float cz, float rb2, int y, int z) {
#ifdef __CUDA_ARCH__
  const float dy = __fsub_rn((float)y, cy), dz = __fsub_rn((float)z, cz);
  return __fadd_rn(__fmul_rn(dy, dy), __fmul_rn(dz, dz)) > rb2;
#else
  const volatile float dy = (float)y - cy, dz = (float)z - cz;
  const volatile float dy2 = dy * dy, dz2 = dz * dz;
  const volatile float d2 = dy2 + dz2;
  return d2 > rb2;
#endif
}
UR_HD __forceinline__ bool row_outside(const ShapeArgs& sh, int y, int z) {
  return row_outside(sh.cy, sh.cz, sh.rb2, y, z);
}

// Rows y of plane z that the particle can reach, (first, count): those that row_outside does not take
// as outside.  They are neighbours, since row_outside is monotone on either side of the centre.  The
// square root is only where the search starts: the walks inwards drop what is outside, the walks
// outwards find rows of spheres so large (from about 2^14 voxels radius) that the float32 steps of
// rb2 are wider than the margin of the start.  For other particles each walk ends at its first or
// second step.
UR_HD __forceinline__ int2 row_range(const ShapeArgs& sh, int z, int N) {
  const float dz = (float)z - sh.cz;
  const float r = sqrtf(fmaxf(sh.rb2 - dz * dz, 0.f));
  int a = (int)floorf(fminf(fmaxf(sh.cy - r, -1.f), (float)N)) - 1;
  int b = (int)ceilf(fminf(fmaxf(sh.cy + r, -2.f), (float)N)) + 1;
  a = a > 0 ? a : 0;
  b = b < N - 1 ? b : N - 1;
  while (a > 0 && !row_outside(sh, a - 1, z)) --a;
  while (b < N - 1 && !row_outside(sh, b + 1, z)) ++b;
  while (a <= b && row_outside(sh, a, z)) ++a;
  while (b >= a && row_outside(sh, b, z)) --b;
  return make_int2(a, b >= a ? b - a + 1 : 0);
}

// Rotated lattice (Sec. 2.3: the cell sampled on rotated planes with periodic wrap).
// Sample point of voxel (x, y, z) in cell-voxel units: p = R (x - c) + q, c = the shape
// centre; value: trilinear interpolation of the periodic cell at p.  Every product, sum
// and difference is rounded separately in the order below, so the result is the same
// float32 value on every device and in the reference of the tests.
struct LatArgs {
  int on;
  float r[9];
  float q[3];
};

__device__ __forceinline__ int ur_wrap(int i, int U) {
  int m = i % U;
  return m < 0 ? m + U : m;
}

__device__ __forceinline__ float ur_lerp(float a, float b, float f) { return __fadd_rn(a, __fmul_rn(f, __fsub_rn(b, a))); }

__device__ __forceinline__ float lattice_sample(const LatArgs& L, const ShapeArgs& sh, const float* __restrict__ cell,
                                                int U, int x, int y, int z) {
  const float d0 = __fsub_rn((float)x, sh.cx), d1 = __fsub_rn((float)y, sh.cy), d2 = __fsub_rn((float)z, sh.cz);
  float p[3];
#pragma unroll
  for (int a = 0; a < 3; ++a)
    p[a] = __fadd_rn(__fadd_rn(__fadd_rn(__fmul_rn(L.r[3 * a], d0), __fmul_rn(L.r[3 * a + 1], d1)),
                               __fmul_rn(L.r[3 * a + 2], d2)),
                     L.q[a]);
  int i0[3], i1[3];
  float f[3];
#pragma unroll
  for (int a = 0; a < 3; ++a) {
    const float fl = floorf(p[a]);
    f[a] = __fsub_rn(p[a], fl);
    i0[a] = ur_wrap((int)fl, U);
    i1[a] = i0[a] + 1 == U ? 0 : i0[a] + 1;
  }
  // cell[z][y][x]; axis 0 = x
  const float* c00 = cell + ((long long)i0[2] * U + i0[1]) * U;
  const float* c01 = cell + ((long long)i0[2] * U + i1[1]) * U;
  const float* c10 = cell + ((long long)i1[2] * U + i0[1]) * U;
  const float* c11 = cell + ((long long)i1[2] * U + i1[1]) * U;
  const float v00 = ur_lerp(__ldg(c00 + i0[0]), __ldg(c00 + i1[0]), f[0]);
  const float v01 = ur_lerp(__ldg(c01 + i0[0]), __ldg(c01 + i1[0]), f[0]);
  const float v10 = ur_lerp(__ldg(c10 + i0[0]), __ldg(c10 + i1[0]), f[0]);
  const float v11 = ur_lerp(__ldg(c11 + i0[0]), __ldg(c11 + i1[0]), f[0]);
  return ur_lerp(ur_lerp(v00, v01, f[1]), ur_lerp(v10, v11, f[1]), f[2]);
}

static inline LatArgs ur_lattice_args(const ur_lattice* lat) {
  LatArgs L;
  memset(&L, 0, sizeof L);
  if (!lat) return L;
  L.on = 1;
  for (int i = 0; i < 9; ++i) L.r[i] = lat->rot[i];
  for (int i = 0; i < 3; ++i) L.q[i] = lat->offset[i];
  return L;
}

static inline ShapeArgs ur_shape_args(const ur_shape* shape) {
  ShapeArgs sh;
  sh.kind = shape->kind;
  sh.cx = shape->center[0];
  sh.cy = shape->center[1];
  sh.cz = shape->center[2];
  sh.s = shape->size;
  for (int i = 0; i < 9; ++i) sh.r[i] = shape->rot[i];
  sh.rb2 = INFINITY;
  if (sh.kind == UR_SHAPE_SPHERE) {
    sh.rb2 = sh.s * sh.s;
  } else if (sh.kind == UR_SHAPE_CUBE || sh.kind == UR_SHAPE_OCTAHEDRON) {
    // Inside, |p|^2 <= 3 s^2 (cube) or s^2 (octahedron), and |d|^2 <= |p|^2 / (1 - e) where e bounds
    // |R R^T - 1|; the slack covers the predicate's float32 roundings (relative 1e-6 of |d|, and 2.5e-4
    // voxels of a rounded coordinate below 4096).  A matrix that is not nearly a rotation has no bound.
    double e = 0.0;
    for (int i = 0; i < 3; ++i) {
      double row = 0.0;
      for (int j = 0; j < 3; ++j) {
        double v = i == j ? -1.0 : 0.0;
        for (int k = 0; k < 3; ++k) v += (double)sh.r[3 * i + k] * (double)sh.r[3 * j + k];
        row += fabs(v);
      }
      if (!(row <= e)) e = row;
    }
    if (e < 0.01 && sh.s < 1e6f) {
      const double s = sh.s > 0.f ? (double)sh.s : 0.0;
      const double r = s * (sh.kind == UR_SHAPE_CUBE ? 1.7320508075688772 : 1.0) / sqrt(1.0 - e) * 1.0001 + 0.05;
      sh.rb2 = (float)(r * r);
    }
  }
  return sh;
}

// [lo, hi): the coordinates i of an axis (particle centre c) that the mask can reach (all of
// [0, n) when unknown), with the roundings of row_outside
static inline void ur_mask_range(const ShapeArgs& sh, float c, int n, int* lo, int* hi) {
  auto out = [&](int i) {
    const float d = (float)i - c;
    const float d2 = d * d;
    return d2 > sh.rb2;
  };
  int a = 0, b = n;
  while (a < n && out(a)) ++a;
  while (b > a && out(b - 1)) --b;
  *lo = a;
  *hi = b;
}
