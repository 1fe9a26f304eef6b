// Electron-density generation (Sec. 2.3).
//
// k_density  ED-1: the unit cell repeated with periodic wrap, times the
//            particle mask, written plane by plane (FP32 or FP16).
// k_zoom     ED-2/ED-3: block integration of ED-1 over f^3 blocks, placed
//            in the centre of a zero box (the two orthogonal block steps of
//            the paper are one exact sum here).
#include <math.h>
#include <string.h>

#include <type_traits>

#include "ur_forward.cuh"
#include "ur_density.cuh"

// W neighbouring voxels of a row (W = 2, or 8 where every row starts on a 16-byte boundary)
template <typename T, int W>
__device__ __forceinline__ void store_row(T* out, const float (&v)[W]) {
  if constexpr (W == 2 && sizeof(T) == 4) {
    *reinterpret_cast<float2*>(out) = make_float2(v[0], v[1]);
  } else if constexpr (W == 2) {
    *reinterpret_cast<__half2*>(out) = __halves2half2(__float2half_rn(v[0]), __float2half_rn(v[1]));
  } else if constexpr (sizeof(T) == 4) {
    reinterpret_cast<float4*>(out)[0] = make_float4(v[0], v[1], v[2], v[3]);
    reinterpret_cast<float4*>(out)[1] = make_float4(v[4], v[5], v[6], v[7]);
  } else {
    __half2 h[4];
#pragma unroll
    for (int i = 0; i < 4; ++i) h[i] = __halves2half2(__float2half_rn(v[2 * i]), __float2half_rn(v[2 * i + 1]));
    *reinterpret_cast<uint4*>(out) = *reinterpret_cast<const uint4*>(h);
  }
}

struct DensityArgs {
  int N, U, ox, oy, z_begin, z_org;  // cell plane of plane blockIdx.y: (z_org + blockIdx.y) mod U
  const float* cell;
  int vec;        // 1: every group of 4 voxels is one aligned 16-byte read of the cell row
  int lg_lanes;   // threads per row: 2^lg_lanes
  FastDiv fu;     // division by U
  ShapeArgs sh;
  LatArgs lat;
  const float* weights;
};

// Plane z holds density: extend the range (min z, max z).  Every thread of the block calls it.
__device__ __forceinline__ void mark_plane(bool nonzero, int z, int* __restrict__ nz_range) {
  if (__syncthreads_or(nonzero) && threadIdx.x == 0) {
    atomicMin(nz_range, z);
    atomicMax(nz_range + 1, z);
  }
}

// Grid (rows of a plane / rows per block, z_count); 2^lg_lanes neighbouring threads write a row in
// groups of W voxels.  Bound by the writes of the density, so what a row shares (cell row, the y and
// z terms of the mask) is formed once per thread and a group's mask costs two voxels, not W, where
// the float32 predicate is an interval along the row (RowMask::group); the values are always u * m.
// 1024^3 FP16 cube filling the box: 4294 -> 615 us (two voxels per thread with 64-bit divisions,
// every voxel's mask evaluated; one group per thread, 938 us).
template <typename T, int W>
__global__ void __launch_bounds__(256) k_density(const __grid_constant__ DensityArgs a, T* __restrict__ out,
                                                 int* __restrict__ nz_range) {
  const int N = a.N, U = a.U;
  const int z = a.z_begin + blockIdx.y;
  const int lanes = 1 << a.lg_lanes;
  const int y = (int)(blockIdx.x * (256u >> a.lg_lanes) + (threadIdx.x >> a.lg_lanes));
  bool nonzero = false;
  if (y < N) {
    const float* crow = a.cell + ((long long)a.fu.mod((uint32_t)(a.z_org + (int)blockIdx.y)) * U +
                                  a.fu.mod((uint32_t)(y + a.oy))) * U;
    const int x0 = (threadIdx.x & (lanes - 1)) * W;
    int c = (int)a.fu.mod((uint32_t)(x0 + a.ox));
    const int cstep = (int)a.fu.mod((uint32_t)(lanes * W));
    RowMask rm;
    rm.init(a.sh, y, z);
    T* orow = out + ((long long)blockIdx.y * N + y) * N;
    for (int x = x0; x < N; x += lanes * W) {
      float u[W], m[W], v[W];
      int ce = c;
      if (W == 8 && a.vec) {
#pragma unroll
        for (int h = 0; h < W / 4; ++h) {
          const float4 t = __ldg(reinterpret_cast<const float4*>(crow + ce));
          u[4 * h] = t.x;
          u[4 * h + 1] = t.y;
          u[4 * h + 2] = t.z;
          u[4 * h + 3] = t.w;
          ce = ce + 4 == U ? 0 : ce + 4;
        }
      } else {
#pragma unroll
        for (int e = 0; e < W; ++e) {
          u[e] = __ldg(crow + ce);
          ce = ce + 1 == U ? 0 : ce + 1;
        }
      }
      c += cstep;
      if (c >= U) c -= U;
      if (a.sh.kind == UR_SHAPE_WEIGHTS) {
        const float* wrow = a.weights + ((long long)z * N + y) * N + x;
#pragma unroll
        for (int e = 0; e < W; ++e) m[e] = __ldg(wrow + e);
      } else {
        rm.group<W>(x, m);
      }
#pragma unroll
      for (int e = 0; e < W; ++e) v[e] = __fmul_rn(u[e], m[e]);
      if (nz_range) {
        // nonzero as stored (an FP16 value may round to zero)
#pragma unroll
        for (int e = 0; e < W; ++e) nonzero |= (sizeof(T) == 2 ? __half2float(__float2half_rn(v[e])) : v[e]) != 0.f;
      }
      store_row<T, W>(orow + x, v);
    }
  }
  if (nz_range) mark_plane(nonzero, z, nz_range);
}

// Voxels sampled on a rotated lattice: one pair of neighbours per thread, numbered through the plane, so that
// no thread is idle at a row's end.  Bound by the eight cell reads of a sample and their index arithmetic.
// As another case of k_density, a warp per row, it held 62 registers instead of 32 and left up to a third of
// the threads idle: 5 to 15 % slower on 64^3 and 100^3, 4 % on 250^3 (137 us now).
template <typename T>
__global__ void __launch_bounds__(256) k_density_lattice(const __grid_constant__ DensityArgs a, FastDiv half,
                                                         T* __restrict__ out, int* __restrict__ nz_range) {
  const int N = a.N, z = a.z_begin + blockIdx.y;
  const uint32_t pair = blockIdx.x * 256u + threadIdx.x;
  bool nonzero = false;
  if (pair < (uint32_t)N * half.d) {
    const int y = (int)half.div(pair), x = 2 * (int)(pair - (uint32_t)y * half.d);
    float m[2], v[2];
    if (a.sh.kind == UR_SHAPE_WEIGHTS) {
      const float* w = a.weights + ((long long)z * N + y) * N + x;
      m[0] = __ldg(w);
      m[1] = __ldg(w + 1);
    } else {
      RowMask rm;
      rm.init(a.sh, y, z);
      m[0] = rm.at(x);
      m[1] = rm.at(x + 1);
    }
#pragma unroll
    for (int e = 0; e < 2; ++e) {
      v[e] = __fmul_rn(lattice_sample(a.lat, a.sh, a.cell, a.U, x + e, y, z), m[e]);
      // nonzero as stored (an FP16 value may round to zero)
      nonzero |= (sizeof(T) == 2 ? __half2float(__float2half_rn(v[e])) : v[e]) != 0.f;
    }
    store_row<T, 2>(out + ((long long)blockIdx.y * N + y) * N + x, v);
  }
  if (nz_range) mark_plane(nonzero, z, nz_range);
}

static ur_status shape_args(const ur_shape* shape, ShapeArgs* sh) {
  UR_REQUIRE(shape, "ur_build_density: null shape");
  UR_REQUIRE(shape->kind >= UR_SHAPE_SPHERE && shape->kind <= UR_SHAPE_WEIGHTS, "ur_build_density: bad shape kind %d",
             shape->kind);
  *sh = ur_shape_args(shape);
  return UR_OK;
}

static ur_status build_density(int32_t n, const float* cell, int32_t ucell, const int32_t* origin,
                               const ur_lattice* lattice, const ur_shape* shape, const float* weights, int32_t z_begin,
                               int32_t z_count, int32_t out_dtype, void* ed_out, int32_t* nz_range, void* stream) {
  UR_REQUIRE(n >= 2 && n % 2 == 0 && n <= 65536, "ur_build_density: grid edge %d must be even", n);
  UR_REQUIRE(cell && ed_out && ucell >= 1, "ur_build_density: null cell/output or empty cell");
  UR_REQUIRE(z_begin >= 0 && z_count >= 0 && z_begin + z_count <= n, "ur_build_density: planes [%d, %d) outside [0, %d)",
             z_begin, z_begin + z_count, n);
  UR_REQUIRE(out_dtype == UR_F32 || out_dtype == UR_F16, "ur_build_density: out_dtype must be UR_F32 or UR_F16");
  UR_REQUIRE(((uintptr_t)ed_out % 8) == 0, "ur_build_density: ed_out must be 8-byte aligned");
  ShapeArgs sh;
  UR_TRY(shape_args(shape, &sh));
  UR_REQUIRE(sh.kind != UR_SHAPE_WEIGHTS || weights, "ur_build_density: weights required for UR_SHAPE_WEIGHTS");
  int ox = 0, oy = 0, oz = 0;
  if (origin) {
    UR_REQUIRE(origin[0] >= 0 && origin[1] >= 0 && origin[2] >= 0, "ur_build_density: origin must be >= 0");
    ox = origin[0];
    oy = origin[1];
    oz = origin[2];
  }
  const LatArgs lat = ur_lattice_args(lattice);
  if (z_count == 0) return UR_OK;
  cudaStream_t s = (cudaStream_t)stream;
  DensityArgs a;
  memset(&a, 0, sizeof a);
  a.N = n;
  a.U = ucell;
  // cell indices by multiply-shift need x + origin < 2^31: the origin reduced modulo the cell edge
  a.ox = ox % ucell;
  a.oy = oy % ucell;
  a.z_begin = z_begin;
  a.z_org = oz % ucell + z_begin;
  a.cell = cell;
  a.fu = FastDiv((uint32_t)ucell);
  a.sh = sh;
  a.lat = lat;
  a.weights = weights;
  ur_timing_begin("density", s);
  int* nzr = nz_range;
  if (lat.on) {
    const FastDiv half((uint32_t)(n / 2));
    const dim3 grid((unsigned)(((long long)n * (n / 2) + 255) / 256), (unsigned)z_count);
    if (out_dtype == UR_F32) k_density_lattice<float><<<grid, 256, 0, s>>>(a, half, (float*)ed_out, nzr);
    else k_density_lattice<__half><<<grid, 256, 0, s>>>(a, half, (__half*)ed_out, nzr);
  } else {
    // groups of eight voxels need 16-byte row starts; edges that are no multiple of 8 take pairs
    const bool wide = n % 8 == 0 && ((uintptr_t)ed_out % 16) == 0;
    a.vec = (ucell % 4 == 0 && a.ox % 4 == 0 && ((uintptr_t)cell % 16) == 0) ? 1 : 0;
    // a warp per row, or as many threads (a power of two) as a short row has groups
    const int per_row = n / (wide ? 8 : 2);
    while (a.lg_lanes < 5 && (1 << a.lg_lanes) < per_row) ++a.lg_lanes;
    const int rows = 256 >> a.lg_lanes;
    const dim3 grid((unsigned)((n + rows - 1) / rows), (unsigned)z_count);
    const bool f32 = out_dtype == UR_F32;
    if (wide && f32) k_density<float, 8><<<grid, 256, 0, s>>>(a, (float*)ed_out, nzr);
    else if (wide) k_density<__half, 8><<<grid, 256, 0, s>>>(a, (__half*)ed_out, nzr);
    else if (f32) k_density<float, 2><<<grid, 256, 0, s>>>(a, (float*)ed_out, nzr);
    else k_density<__half, 2><<<grid, 256, 0, s>>>(a, (__half*)ed_out, nzr);
  }
  UR_LAUNCH_CHECK("k_density");
  ur_timing_end(s);
  return UR_OK;
}

extern "C" ur_status ur_build_density(int32_t n, const float* cell, int32_t ucell, const int32_t* origin,
                                      const ur_shape* shape, const float* weights, int32_t z_begin, int32_t z_count,
                                      int32_t out_dtype, void* ed_out, int32_t* nz_range, void* stream) {
  return build_density(n, cell, ucell, origin, nullptr, shape, weights, z_begin, z_count, out_dtype, ed_out, nz_range,
                       stream);
}

// Test hook: the squared radius beyond which the rows of a shape are taken as outside (row_outside)
extern "C" float ur_selftest_row_bound(const ur_shape* shape) { return ur_shape_args(shape).rb2; }

// Test hook: the rows of planes 0 .. n - 1 that the column passes take as the particle's, (first, count) pairs
extern "C" void ur_selftest_row_ranges(const ur_shape* shape, int32_t n, int32_t* out) {
  const ShapeArgs sh = ur_shape_args(shape);
  for (int z = 0; z < n; ++z) {
    const int2 r = row_range(sh, z, n);
    out[2 * z] = r.x;
    out[2 * z + 1] = r.y;
  }
}

extern "C" ur_status ur_build_density_lattice(int32_t n, const float* cell, int32_t ucell, const ur_lattice* lattice,
                                              const ur_shape* shape, const float* weights, int32_t z_begin,
                                              int32_t z_count, int32_t out_dtype, void* ed_out, int32_t* nz_range,
                                              void* stream) {
  UR_REQUIRE(lattice, "ur_build_density_lattice: null lattice");
  return build_density(n, cell, ucell, nullptr, lattice, shape, weights, z_begin, z_count, out_dtype, ed_out, nz_range,
                       stream);
}

// ---------------------------------------------------------------------------
// Zoom-out by block integration
// ---------------------------------------------------------------------------
// Round v = S * 2^-24 (S an integer) to binary16, ties to even.
__device__ __forceinline__ unsigned short half_bits_from_fixed24(long long S) {
  unsigned short sign = 0;
  unsigned long long a;
  if (S < 0) {
    sign = 0x8000;
    a = (unsigned long long)(-S);
  } else {
    a = (unsigned long long)S;
  }
  if (a < 1024ull) return sign | (unsigned short)a;  // subnormal or zero: exact
  int e = 63 - __clzll((long long)a);               // a in [2^e, 2^(e+1)), e >= 10
  const int shift = e - 10;
  unsigned long long q = a >> shift;
  if (shift > 0) {
    const unsigned long long rem = a & ((1ull << shift) - 1);
    const unsigned long long half = 1ull << (shift - 1);
    if (rem > half || (rem == half && (q & 1ull))) ++q;
    if (q == 2048ull) {
      q = 1024ull;
      ++e;
    }
  }
  const int ex = e - 9;  // biased exponent of q * 2^(e - 10 - 24)
  if (ex >= 31) return sign | 0x7C00;
  return sign | (unsigned short)((ex << 10) | (int)(q - 1024ull));
}

// FP16 block sums for f = 2, 4, 8, 16 and rows of whole 16-byte groups.  One block per output row
// (Z, Y) of the particle, then blocks that zero the other rows; a thread sums the f^2 source rows of 8
// neighbouring x.  Bound by the reads of the source, so the exact integer sum must be cheap: with C = 1.5 2^17 every t = v + C lies in
// [2^17, 2^18), where floats are multiples of 2^-6, so the bits of t count v rounded to 2^-6
// (summed as int32) and v - (t - C), a multiple of 2^-24 of at most 2^-7, is summed exactly in
// float32 over up to 128 terms before it is added to an integer.  A source row with an infinity or
// NaN shows as a NaN remainder; its outputs take the conversion of k_zoom.
// 1024^3 -> 512^3 box by 4 / by 16: 1847 / 1918 -> 461 / 395 us (two-byte loads, a
// 64-bit conversion per value, 64-bit shared atomics).
#define UR_ZOOM_C 196608.0f
#define UR_ZOOM_ZROWS 16  // rows of the box per zero-filling block
template <int F, typename TO>
__global__ void __launch_bounds__(256) k_zoom_half(const __half* __restrict__ src, int n_src, int n_out,
                                                   TO* __restrict__ out) {
  extern __shared__ __align__(16) unsigned char smraw[];
  long long* acc = reinterpret_cast<long long*>(smraw);
  const int m = n_src / F, o = (n_out - m) / 2;
  const bool wide = n_out % 8 == 0 && ((uintptr_t)out % 16) == 0;  // rows start on 16-byte boundaries
  if (blockIdx.x >= (unsigned)(m * m)) {  // rows that no source row reaches
    const unsigned r0 = (blockIdx.x - m * m) * UR_ZOOM_ZROWS;
    int Z = (int)(r0 / (unsigned)n_out), Y = (int)(r0 - (unsigned)Z * n_out);
    for (int i = 0; i < UR_ZOOM_ZROWS && Z < n_out; ++i, Z += Y + 1 == n_out, Y = Y + 1 == n_out ? 0 : Y + 1) {
      if ((unsigned)(Z - o) < (unsigned)m && (unsigned)(Y - o) < (unsigned)m) continue;
      TO* row = out + ((long long)Z * n_out + Y) * n_out;
      if (wide) {
        for (int X = threadIdx.x; X < n_out * (int)sizeof(TO) / 16; X += blockDim.x)
          reinterpret_cast<uint4*>(row)[X] = make_uint4(0u, 0u, 0u, 0u);
      } else {
        for (int X = threadIdx.x; X < n_out; X += blockDim.x) row[X] = TO(0.f);
      }
    }
    return;
  }
  const int zs = blockIdx.x / m, ys = blockIdx.x - (blockIdx.x / m) * m;
  TO* orow = out + ((long long)(zs + o) * n_out + (ys + o)) * n_out;
  constexpr int PER = 8 / F > 0 ? 8 / F : 1;   // outputs per thread (F = 16: two threads share one)
  constexpr int NV = F < 8 ? F : 8;            // values of a thread's row group per output
  constexpr int FOLD = 128 < F * F ? 128 / F : F;  // dz per fold: at most 128 terms per float32 sum
  {
    const int groups = n_src / 8;
    const int rounds = (groups + (int)blockDim.x - 1) / (int)blockDim.x;
    for (int it = 0; it < rounds; ++it) {
      const int g = threadIdx.x + it * blockDim.x;
      long long S[PER];
#pragma unroll
      for (int p = 0; p < PER; ++p) S[p] = 0;
      if (g < groups) {
        const __half* base = src + ((long long)F * zs * n_src + (long long)F * ys) * n_src + 8 * g;
        int hi[8], lo[8];
        bool bad = false;
#pragma unroll
        for (int e = 0; e < 8; ++e) hi[e] = lo[e] = 0;
        const ur_f2 C = f2_pack(UR_ZOOM_C, UR_ZOOM_C);
        for (int z0 = 0; z0 < F; z0 += FOLD) {
          ur_f2 rem[4];
#pragma unroll
          for (int q = 0; q < 4; ++q) rem[q] = f2_pack(0.f, 0.f);
#pragma unroll(F <= 4 ? FOLD : 1)
          for (int dz = z0; dz < z0 + FOLD; ++dz) {
#pragma unroll
            for (int dy = 0; dy < F; ++dy) {
              const uint4 w = __ldg(reinterpret_cast<const uint4*>(base + ((long long)dz * n_src + dy) * n_src));
              const uint32_t ww[4] = {w.x, w.y, w.z, w.w};
#pragma unroll
              for (int q = 0; q < 4; ++q) {
                const float2 f = __half22float2(*reinterpret_cast<const __half2*>(&ww[q]));
                const ur_f2 v = f2_pack(f.x, f.y);
                const ur_f2 t = f2_add(v, C);
                rem[q] = f2_add(rem[q], f2_sub(v, f2_sub(t, C)));
                const float2 tt = f2_get(t);
                hi[2 * q] += __float_as_int(tt.x) - __float_as_int(UR_ZOOM_C);
                hi[2 * q + 1] += __float_as_int(tt.y) - __float_as_int(UR_ZOOM_C);
              }
            }
          }
#pragma unroll
          for (int q = 0; q < 4; ++q) {
            const float2 r = f2_get(rem[q]);
            bad |= r.x != r.x || r.y != r.y;
            lo[2 * q] += __float2int_rn(r.x * 16777216.0f);
            lo[2 * q + 1] += __float2int_rn(r.y * 16777216.0f);
          }
        }
#pragma unroll
        for (int e = 0; e < 8; ++e) S[e / NV] += ((long long)hi[e] << 18) + (long long)lo[e];
        if (bad) {
#pragma unroll
          for (int p = 0; p < PER; ++p) S[p] = 0;
          for (int dz = 0; dz < F; ++dz)
            for (int dy = 0; dy < F; ++dy)
#pragma unroll
              for (int e = 0; e < 8; ++e)
                S[e / NV] += __float2ll_rn(__half2float(base[((long long)dz * n_src + dy) * n_src + e]) * 16777216.0f);
        }
      }
      if constexpr (F == 16) S[0] += __shfl_xor_sync(0xffffffffu, S[0], 1);  // rounds are uniform over the block
      if (g < groups) {
        if constexpr (F == 16) {
          if ((g & 1) == 0) acc[g / 2] = S[0];
        } else {
#pragma unroll
          for (int p = 0; p < PER; ++p) acc[g * PER + p] = S[p];
        }
      }
    }
    __syncthreads();
  }
  // eight outputs per thread where rows start on 16-byte boundaries, else one
  const int step = wide ? 8 : 1;
  for (int X = threadIdx.x * step; X < n_out; X += blockDim.x * step) {
    float vf[8];
    unsigned short hb[8];
    for (int e = 0; e < step; ++e) {
      const int xs = X + e - o;
      const long long S = (xs >= 0 && xs < m) ? acc[xs] : 0;
      if constexpr (sizeof(TO) == 2) hb[e] = half_bits_from_fixed24(S);
      else vf[e] = __double2float_rn((double)S * 5.9604644775390625e-08);  // * 2^-24, exact in double
    }
    if (wide) {
      if constexpr (sizeof(TO) == 2) {
        *reinterpret_cast<uint4*>(orow + X) =
            make_uint4(hb[0] | (uint32_t)hb[1] << 16, hb[2] | (uint32_t)hb[3] << 16, hb[4] | (uint32_t)hb[5] << 16,
                       hb[6] | (uint32_t)hb[7] << 16);
      } else {
        reinterpret_cast<float4*>(orow + X)[0] = make_float4(vf[0], vf[1], vf[2], vf[3]);
        reinterpret_cast<float4*>(orow + X)[1] = make_float4(vf[4], vf[5], vf[6], vf[7]);
      }
    } else {
      if constexpr (sizeof(TO) == 2) orow[X] = __ushort_as_half(hb[0]);
      else orow[X] = vf[0];
    }
  }
}

// One block per output row (Z, Y) of the n_out^3 box.
template <typename TS, typename TO>
__global__ void __launch_bounds__(256) k_zoom(const TS* __restrict__ src, int n_src, int f, int n_out,
                                              TO* __restrict__ out) {
  extern __shared__ __align__(16) unsigned char smraw[];
  const int Z = blockIdx.x / n_out, Y = blockIdx.x - (blockIdx.x / n_out) * n_out;
  const int m = n_src / f, o = (n_out - m) / 2;
  const int zs = Z - o, ys = Y - o;
  TO* orow = out + ((long long)Z * n_out + Y) * n_out;
  const bool inside = zs >= 0 && zs < m && ys >= 0 && ys < m;
  constexpr bool EXACT = sizeof(TS) == 2;
  using Acc = typename std::conditional<EXACT, unsigned long long, double>::type;
  Acc* acc = reinterpret_cast<Acc*>(smraw);
  if (inside) {
    for (int i = threadIdx.x; i < m; i += blockDim.x) acc[i] = 0;
    __syncthreads();
    for (int x = threadIdx.x; x < n_src; x += blockDim.x) {
      Acc part = 0;
      for (int dz = 0; dz < f; ++dz) {
        for (int dy = 0; dy < f; ++dy) {
          const long long row = ((long long)(f * zs + dz) * n_src + (f * ys + dy)) * n_src;
          if constexpr (EXACT) {
            const float v = __half2float(src[row + x]);
            part += (unsigned long long)__float2ll_rn(v * 16777216.0f);  // v * 2^24, an exact integer
          } else {
            part += (double)src[row + x];
          }
        }
      }
      atomicAdd(acc + x / f, part);
    }
    __syncthreads();
  }
  for (int X = threadIdx.x; X < n_out; X += blockDim.x) {
    const int xs = X - o;
    float vf = 0.f;
    unsigned short hb = 0;
    if (inside && xs >= 0 && xs < m) {
      if constexpr (EXACT) {
        const long long S = (long long)acc[xs];
        hb = half_bits_from_fixed24(S);
        vf = __double2float_rn((double)S * 5.9604644775390625e-08);  // * 2^-24, exact in double
      } else {
        const double d = (double)acc[xs];
        vf = __double2float_rn(d);
        hb = __half_as_ushort(__double2half(d));
      }
    }
    if constexpr (sizeof(TO) == 2) orow[X] = __ushort_as_half(hb);
    else orow[X] = vf;
  }
}

extern "C" ur_status ur_zoom_density(int32_t n_src, int32_t src_dtype, const void* src, int32_t f, int32_t n_out,
                                     int32_t out_dtype, void* out, void* stream) {
  UR_REQUIRE(src && out, "ur_zoom_density: null argument");
  UR_REQUIRE(f >= 1 && n_src >= f && n_src % f == 0, "ur_zoom_density: source edge %d not divisible by factor %d", n_src, f);
  UR_REQUIRE(n_out >= n_src / f, "ur_zoom_density: box %d smaller than the zoomed particle %d", n_out, n_src / f);
  UR_REQUIRE(src_dtype == UR_F32 || src_dtype == UR_F16, "ur_zoom_density: bad source type");
  UR_REQUIRE(out_dtype == UR_F32 || out_dtype == UR_F16, "ur_zoom_density: bad output type");
  UR_REQUIRE(src_dtype == UR_F32 || (long long)f * f * f <= 4096, "ur_zoom_density: FP16 exact sums need f^3 <= 4096");
  cudaStream_t s = (cudaStream_t)stream;
  const int m = n_src / f;
  const size_t smem = (size_t)m * 8;
  UR_REQUIRE(smem <= 200 * 1024, "ur_zoom_density: zoomed row too long");
  const unsigned grid = (unsigned)((long long)n_out * n_out);
#define UR_ZOOM(TS, TO)                                                                                   \
  do {                                                                                                    \
    if (smem > 48 * 1024)                                                                                 \
      UR_CUDA_CHECK(cudaFuncSetAttribute(k_zoom<TS, TO>, cudaFuncAttributeMaxDynamicSharedMemorySize, (int)smem)); \
    k_zoom<TS, TO><<<grid, 256, smem, s>>>((const TS*)src, n_src, f, n_out, (TO*)out);                    \
  } while (0)
  ur_timing_begin("zoom", s);
  // FP16 sources with the usual factors and rows of whole 16-byte groups: k_zoom_half; every other
  // factor, edge, alignment and FP32 sources: k_zoom.  Halving short rows without a box around them
  // leaves k_zoom_half too few loads in flight (48 -> 24 3.3 us against 2.9, 96 -> 48 5.5 against 5.1, but
  // 128 -> 64 5.9 against 8.6, and 7.2 against 15.4 in a box of 128).
  const bool fast = src_dtype == UR_F16 && n_src % 8 == 0 && ((uintptr_t)src % 16) == 0 &&
                    (f > 2 || n_src >= 128 || n_out > m);
#define UR_ZOOM_HALF(F)                                                                                   \
  do {                                                                                                    \
    const int threads = n_src / 8 >= 256 ? 256 : (n_src / 8 + 31) / 32 * 32;                              \
    if (smem > 48 * 1024) {                                                                               \
      UR_CUDA_CHECK(cudaFuncSetAttribute(k_zoom_half<F, __half>, cudaFuncAttributeMaxDynamicSharedMemorySize, (int)smem)); \
      UR_CUDA_CHECK(cudaFuncSetAttribute(k_zoom_half<F, float>, cudaFuncAttributeMaxDynamicSharedMemorySize, (int)smem));  \
    }                                                                                                     \
    const unsigned zgrid = (unsigned)((long long)m * m +                                                  \
                                      (n_out > m ? ((long long)n_out * n_out + UR_ZOOM_ZROWS - 1) / UR_ZOOM_ZROWS : 0));     \
    if (out_dtype == UR_F16)                                                                              \
      k_zoom_half<F, __half><<<zgrid, threads, smem, s>>>((const __half*)src, n_src, n_out, (__half*)out); \
    else k_zoom_half<F, float><<<zgrid, threads, smem, s>>>((const __half*)src, n_src, n_out, (float*)out); \
  } while (0)
  if (fast && f == 2) UR_ZOOM_HALF(2);
  else if (fast && f == 4) UR_ZOOM_HALF(4);
  else if (fast && f == 8) UR_ZOOM_HALF(8);
  else if (fast && f == 16) UR_ZOOM_HALF(16);
  else if (src_dtype == UR_F16 && out_dtype == UR_F16) UR_ZOOM(__half, __half);
  else if (src_dtype == UR_F16) UR_ZOOM(__half, float);
  else if (out_dtype == UR_F16) UR_ZOOM(float, __half);
  else UR_ZOOM(float, float);
#undef UR_ZOOM
#undef UR_ZOOM_HALF
  UR_LAUNCH_CHECK("k_zoom");
  ur_timing_end(s);
  return UR_OK;
}
