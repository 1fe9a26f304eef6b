// Forward path: Sec. 2.4 separated transform (Eq. 2) and Sec. 2.5 Q binning.
//
//   pass 1a  k_rows_r2c        real-to-complex transform along x of every row of
//                              the planes that hold density (two reals packed as
//                              one complex, N/2-point FFT, then the split step)
//   pass 1b  k_cols<COL_Y>     complex transform along y of each (plane, kx)
//                              column, in place: with 1a, the 2D transform of
//                              every nonzero plane (inner sum of Eq. 2)
//   pass 2   k_cols<COL_ZBIN>  complex transform along z of each (ky, kx)
//                              column; planes outside [z0, z0+nz) enter as zeros
//                              (Sec. 2.4: skipped slices are padded); |F|^2 and
//                              the Q-bin sums are taken from shared memory
//   k_finalize                 per-bin counts, sums, mean and standard error
//
// Layouts: intermediate X[p][y][kx] (p = plane - z0), complex64, kx contiguous,
// N/2+1 per row.  Columns of pass 1b are c = p*(N/2+1) + kx; columns of pass 2
// are c = ky_index*(N/2+1) + kx.
#include <math.h>
#include <stdio.h>
#include <string.h>

#include "ur_fast.cuh"

// Consecutive |kz| per thread in the binning and scaling walks; lanes read that many values apart in
// shared memory, so an odd number spreads them over the banks (8 -> 9: 378^3 z + bins 253 -> 245 us, adjoint
// z 285 -> 268; 64 particles 3627 -> 3461 and 4374 -> 4059; 7 and 11 within 3 % of 9)
// (Longer where a tile would take two rounds, shorter where tiles of short lines have fewer values per thread:
// ur_col_args.)
#define BIN_CHUNK 9

// ---------------------------------------------------------------------------
// Pass 1a
// Row r (r = p*N + y) holds N reals read as N/2 complex z[m] = (x[2m], x[2m+1]);
// Z = FFT_{N/2}(z); then, with Z[M] = Z[0],
//   X[k] = (Z[k] + conj Z[M-k])/2 - i W_N^k (Z[k] - conj Z[M-k])/2,  k = 0..M,
// which recombines the transforms of the even and the odd samples.
// ---------------------------------------------------------------------------
template <typename T>
__device__ __forceinline__ float2 load_pair(const T* p);
template <>
__device__ __forceinline__ float2 load_pair<float>(const float* p) {
  return __ldg(reinterpret_cast<const float2*>(p));
}
template <>
__device__ __forceinline__ float2 load_pair<__half>(const __half* p) {
  __half2 h = __ldg(reinterpret_cast<const __half2*>(p));
  return __half22float2(h);
}

struct NoLd {
  struct It {
    __device__ __forceinline__ float2 get() { return make_float2(0.f, 0.f); }
  };
  __device__ __forceinline__ It first(int, int, int) const { return {}; }
};
struct NoSt {
  struct It {
    __device__ __forceinline__ void put(float2) {}
  };
  __device__ __forceinline__ It first(int, int, int) const { return {}; }
};

// GEN = 1: the row's density is generated here (Sec. 2.3 tile + mask) instead of read.
// Body of one block (block index blk); shared by the single-plan and batched launches.
// IO: the first stage reads stored rows from global memory (nst >= 2).
template <int GEN, typename T, bool IO = false>
__device__ __forceinline__ void rows_r2c_body(const RowArgs& ra, int N, int RB, const StageInfo* __restrict__ sched,
                                              int nst, long long blk) {
  extern __shared__ float2 smem[];
  const T* __restrict__ ed = reinterpret_cast<const T*>(ra.ed);
  float2* __restrict__ X = ra.X;
  const long long nrows = ra.nrows;
  const float2* __restrict__ tw = ra.tw;
  const int M = N >> 1, H = M + 1;
  const long long r0 = blk * RB;
  const FastDiv dm((uint32_t)M), dh((uint32_t)H);
  // generated rows (r = p N + y < 2^31): what a row shares is formed once, by one thread per row.  Lattice
  // samples (GEN = 2) form the mask's row terms anew: they are few against a sample's arithmetic, and the
  // shared memory is worth more to its cell reads as L1.
  RowMask* rms = reinterpret_cast<RowMask*>(smem + (size_t)RB * M);  // GEN = 1 (ur_row_smem)
  int* crow = reinterpret_cast<int*>(rms + RB);                       // cell offset of the row
  const FastDiv du((uint32_t)(GEN ? ra.ucell : 1)), dn((uint32_t)N);
  if (GEN) {
    bool some = false;
    for (int t = threadIdx.x; t < RB; t += blockDim.x) {
      const long long r = r0 + t;
      if (r >= nrows) break;
      const int p = (int)dn.div((uint32_t)r), y = (int)r - p * N, z = ra.z0 + p;
      if (GEN == 1) {
        rms[t].init(ra.sh, y, z);
        crow[t] = (int)(du.mod((uint32_t)(z + ra.oz)) * ra.ucell + du.mod((uint32_t)(y + ra.oy)));
      }
      some = some || !row_outside(ra.sh, y, z);
    }
    // rows outside the particle are not written when the y pass knows to skip them
    const bool any = __syncthreads_or(some);
    if (ra.skip_empty && !any) return;
  }
  if constexpr (IO) {
    // stored rows: the first stage reads them from global memory instead of from a copy in shared
    // memory (720^3 FP16 rows 1688 -> 1232 us; generated rows measured slower that way)
    auto stored = [&](int t, int m) -> float2 {
      const long long r = r0 + t;
      return r < nrows ? load_pair<T>(ed + r * N + 2 * m) : make_float2(0.f, 0.f);
    };
    fft_lines_io<false, UR_EMAX, true, false, false>(smem, M, RB, sched, nst, tw, ld_fn(stored), NoSt());
  } else {
    for (int f = threadIdx.x; f < RB * M; f += blockDim.x) {
      const int t = (int)dm.div((uint32_t)f);
      const int m = f - t * M;
      const long long r = r0 + t;
      float2 v = make_float2(0.f, 0.f);
      if (r < nrows) {
        if (GEN) {
          const int x = 2 * m, U = ra.ucell;
          const int p = (int)dn.div((uint32_t)r), y = (int)r - p * N, z = ra.z0 + p;  // (GEN = 2)
          float m0, m1;
          if (ra.weights) {
            const float2 mw = __ldg(reinterpret_cast<const float2*>(ra.weights + ((long long)ra.z0 * N + r) * N + x));
            m0 = mw.x;
            m1 = mw.y;
          } else if (GEN == 2) {
            RowMask rm;
            rm.init(ra.sh, y, z);
            m0 = rm.at(x);
            m1 = rm.at(x + 1);
          } else {
            m0 = rms[t].at(x);
            m1 = rms[t].at(x + 1);
          }
          if (GEN == 2) {
            v = make_float2(__fmul_rn(lattice_sample(ra.lat, ra.sh, ra.cell, U, x, y, z), m0),
                            __fmul_rn(lattice_sample(ra.lat, ra.sh, ra.cell, U, x + 1, y, z), m1));
          } else {
            const int c0 = (int)du.mod((uint32_t)(x + ra.ox)), c1 = c0 + 1 == U ? 0 : c0 + 1;
            const float* cr = ra.cell + (long long)crow[t] * U;
            v = make_float2(__fmul_rn(__ldg(cr + c0), m0), __fmul_rn(__ldg(cr + c1), m1));
          }
        } else {
          v = load_pair<T>(ed + r * N + 2 * m);
        }
      }
      smem[f] = v;
    }
    __syncthreads();
    fft_lines<false, UR_EMAX>(smem, M, RB, sched, nst, tw);
  }
  for (int f = threadIdx.x; f < RB * H; f += blockDim.x) {
    const int t = (int)dh.div((uint32_t)f);
    const int k = f - t * H;
    const long long r = r0 + t;
    if (r >= nrows) continue;
    const float2* Z = smem + t * M;
    const float2 zk = Z[k == M ? 0 : k];
    const float2 zc = cconj(Z[k == 0 ? 0 : M - k]);
    const float2 e = make_float2(0.5f * (zk.x + zc.x), 0.5f * (zk.y + zc.y));
    const float2 d = make_float2(0.5f * (zk.x - zc.x), 0.5f * (zk.y - zc.y));
    const float2 o = make_float2(d.y, -d.x);  // -i d
    const float2 w = __ldg(tw + k);
    X[r * ra.xp + k] = cadd(e, cmul(w, o));
  }
}

template <int GEN, typename T, bool IO>
__global__ void __launch_bounds__(256, 4) k_rows_r2c(RowArgs ra, int N, int RB, const StageInfo* __restrict__ sched,
                                                     int nst) {
  rows_r2c_body<GEN, T, IO>(ra, N, RB, sched, nst, blockIdx.x);
}

// ---------------------------------------------------------------------------
// Column passes.  A block owns TX consecutive columns; column c of the source
// has elements src[(c / H) * A + c % H + i * S], i < nload, placed at shared
// position zoff + i (all other positions zero).
// ---------------------------------------------------------------------------
// Column indices stay below 2^31 (at most N (N/2+1) columns), so the block's
// index arithmetic runs in 32 bits with multiply-shift division (FastDiv).
struct ColDivs {
  FastDiv tx, h;
  __device__ explicit ColDivs(const ColArgs& a) : tx((uint32_t)a.TX), h((uint32_t)a.H) {}
};

// Element access of the column transforms: the elements of tile line `line` (column c0 + line) in the
// source or destination layout.  What an element would cost in index arithmetic is formed once per
// butterfly (a running pointer), and the elements that are known to be zero or not needed (ColArgs:
// row_skip, k2_zero, out_lo) are a range per line, formed once per
// block: 378^3 y 136 -> 127 us, adjoint z 268 -> 260; 64 particles y 843 -> 811, adjoint z 4059 -> 3947.
// (Fields are copied: a batched launch holds its ColArgs in global memory.)
#define UR_TILE_MAX (UR_EMAX * 256 / 8)  // columns per block of the shortest line

struct ColItLd {
  const float2* p;
  long long step;
  int i, di, lo, n;  // elements present: lo <= i < lo + n, or all others (outside)
  bool outside;
  __device__ __forceinline__ float2 get() {
    const bool in = ((unsigned)(i - lo) < (unsigned)n) != outside;
    const float2 v = in ? __ldg(p) : make_float2(0.f, 0.f);
    p += step;
    i += di;
    return v;
  }
};
template <int MODE, bool INV>
struct ColLd {
  const float2* src;
  long long A, S, ncols, c0;
  int zoff, nload;
  const int2* rng;  // y passes: range per line
  FastDiv h;
  __device__ ColLd(const ColArgs& a, const ColDivs& dv, long long c, const int2* ranges)
      : src(a.src), A(a.A), S(a.S), ncols(a.ncols), c0(c), zoff(a.zoff), nload(a.nload), rng(ranges), h(dv.h) {}
  __device__ __forceinline__ ColItLd first(int line, int i, int di) const {
    const long long c = c0 + line;
    const uint32_t o = h.div((uint32_t)c), k = (uint32_t)c - o * h.d;
    ColItLd it;
    it.p = src + (long long)o * A + k + (long long)(i - zoff) * S;
    it.step = (long long)di * S;
    it.i = i;
    it.di = di;
    it.outside = MODE == COL_Y && INV;
    if (MODE == COL_Y) {
      const int2 r = rng[line];
      it.lo = r.x;
      it.n = r.y;
    } else {
      it.lo = zoff;
      it.n = c < ncols ? nload : 0;
    }
    return it;
  }
};
struct ColItSt {
  float2* p;
  long long step;
  int i, di, lo, n;  // elements wanted
  __device__ __forceinline__ void put(float2 v) {
    if ((unsigned)(i - lo) < (unsigned)n) *p = v;
    p += step;
    i += di;
  }
};
template <int MODE, bool INV>
struct ColSt {
  float2* dst;
  long long Ad, Sd, ncols, c0;
  int out_lo, out_cnt, N;
  const int2* rng;  // adjoint y pass with row_skip: range per line, else NULL
  FastDiv h;
  __device__ ColSt(const ColArgs& a, const ColDivs& dv, long long c, const int2* ranges)
      : dst(a.dst), Ad(a.Ad), Sd(a.Sd), ncols(a.ncols), c0(c), out_lo(a.out_lo), out_cnt(a.out_cnt), N(a.N), rng(ranges),
        h(dv.h) {}
  __device__ __forceinline__ ColItSt first(int line, int i, int di) const {
    const long long c = c0 + line;
    const uint32_t o = h.div((uint32_t)c), k = (uint32_t)c - o * h.d;
    const bool slab = MODE == COL_ZADJ && out_cnt > 0;
    ColItSt it;
    it.p = dst + (long long)o * Ad + k + (long long)(i - (slab ? out_lo : 0)) * Sd;
    it.step = (long long)di * Sd;
    it.i = i;
    it.di = di;
    it.lo = slab ? out_lo : 0;
    it.n = slab ? out_cnt : N;
    if (MODE == COL_Y && INV && rng) {
      const int2 r = rng[line];
      it.lo = r.x;
      it.n = r.y;
    }
    if (c >= ncols) it.n = 0;
    return it;
  }
};

// Elements i of a column of kx that lie at or beyond k2_zero, (first, count): |ky| > km, the largest
// with kx^2 + km^2 < k2_zero, is i in (km, N - km)
__device__ __forceinline__ int2 beyond_range(int kx, int k2_zero, int N) {
  const int M = N / 2, left = k2_zero - 1 - kx * kx;
  if (left < 0) return make_int2(0, N);
  int km = min((int)sqrtf((float)left), M);
  while (km > 0 && km * km > left) --km;
  while (km < M && (km + 1) * (km + 1) <= left) ++km;
  return make_int2(km + 1, max(N - 2 * km - 1, 0));
}

// The tile's columns to shared memory and back, for transforms of a single stage
template <class Ld>
__device__ __forceinline__ void load_columns(const ColArgs& a, const ColDivs& dv, float2* buf, int N, Ld ld) {
  const int TX = a.TX;
  for (int f = threadIdx.x; f < TX * N; f += blockDim.x) {
    const int i = (int)dv.tx.div((uint32_t)f);
    const int t = f - i * TX;
    buf[t * a.pitch + i] = ld.first(t, i, 1).get();
  }
  __syncthreads();
}

template <class St>
__device__ __forceinline__ void store_columns(const ColArgs& a, const ColDivs& dv, const float2* buf, int N, St st) {
  const int TX = a.TX;
  for (int f = threadIdx.x; f < TX * N; f += blockDim.x) {
    const int i = (int)dv.tx.div((uint32_t)f);
    const int t = f - i * TX;
    st.first(t, i, 1).put(buf[t * a.pitch + i]);
  }
}

// Walk the (column, |kz|) pairs of the block's spectrum columns in chunks of
// a.walk consecutive |kz| = m.  k^2 = kx^2 + ky^2 + m^2 grows with m, so the
// bin index only moves forward inside a chunk.  kz = m and kz = N - m share k^2.
// Op(t, m, bin, weight) is called for every pair.
template <typename Op>
__device__ __forceinline__ void walk_bins(const ColArgs& a, const ColDivs& dv, const int32_t* __restrict__ thr,
                                          long long c0, Op op) {
  const int M = a.M, H = a.H, N = a.N;
  const int len = a.walk, nch = (H + len - 1) / len;
  const int ntask = a.TX * nch;
  const FastDiv dch((uint32_t)nch);
  for (int task = threadIdx.x; task < ntask; task += blockDim.x) {
    const int t = (int)dch.div((uint32_t)task);
    const int ch = task - t * nch;
    const long long c = c0 + t;
    if (c >= a.ncols) continue;
    const int kyi = (int)dv.h.div((uint32_t)c);
    const int kx = (int)c - kyi * H;
    const int ky = kyi < M ? kyi : kyi - N;
    const int c2 = kx * kx + ky * ky;
    const float w = (kx == 0 || kx == M) ? 1.f : 2.f;
    const int m0 = ch * len;
    const int m1 = min(m0 + len, M + 1);
    int cur = bin_search(thr, a.nbins, c2 + m0 * m0);
    // voxel-sinc factor of the column (kx, ky); the kz part is applied per element
    const float cs = a.vs ? __ldg(a.vs + kx) * __ldg(a.vs + (ky < 0 ? -ky : ky)) : 1.f;
    op.begin(cur, cs);
    for (int m = m0; m < m1; ++m) {
      const int s = c2 + m * m;
      while (cur < a.nbins && thr[cur + 1] <= s) ++cur;
      op.visit(t, m, cur, w);
    }
    op.end(w);
  }
}

struct BinAccum {
  const float2* buf;
  int pitch, M, N, nbins;
  float iscale;
  double* hs;
  double* hs2;
  int run;
  float aI, aI2;
  const float* vs;
  float cs;
  __device__ __forceinline__ void flush(float w) {
    if (run >= 0 && run < nbins && (aI != 0.f || aI2 != 0.f)) {
      atomicAdd(hs + run, (double)(w * aI));
      atomicAdd(hs2 + run, (double)(w * aI2));
    }
    aI = 0.f;
    aI2 = 0.f;
  }
  __device__ __forceinline__ void begin(int b, float c) {
    run = b;
    aI = 0.f;
    aI2 = 0.f;
    cs = c;
  }
  __device__ __forceinline__ void visit(int t, int m, int b, float w) {
    if (b != run) {
      flush(w);
      run = b;
    }
    const float sc = vs ? iscale * (cs * __ldg(vs + m)) : iscale;
    const float2 f1 = buf[t * pitch + m];
    const float i1 = (f1.x * f1.x + f1.y * f1.y) * sc;
    float s = i1, s2 = i1 * i1;
    if (m != 0 && m != M) {
      const float2 f2 = buf[t * pitch + N - m];
      const float i2 = (f2.x * f2.x + f2.y * f2.y) * sc;
      s += i2;
      s2 += i2 * i2;
    }
    aI += s;
    aI2 += s2;
  }
  __device__ __forceinline__ void end(float w) { flush(w); }
};

struct SigmaScale {
  float2* buf;
  int pitch, M, N, nbins;
  const float* sigma;
  __device__ __forceinline__ void begin(int, float) {}
  __device__ __forceinline__ void end(float) {}
  __device__ __forceinline__ void visit(int t, int m, int b, float) {
    const float sg = (b >= 0 && b < nbins) ? __ldg(sigma + b) : 0.f;
    float2* col = buf + t * pitch;
    col[m] = cscale(col[m], sg);
    if (m != 0 && m != M) col[N - m] = cscale(col[N - m], sg);
  }
};

// One block per tile of TX columns.  (A persistent loop over tiles around the
// shared-memory FFT made the compiler spill ~1.3 KB per thread.)
template <int MODE, bool INV>
__device__ __forceinline__ void cols_body(const ColArgs& a, long long blk) {
  extern __shared__ __align__(16) unsigned char smraw[];
  __shared__ int s_blo, s_bhi;
  __shared__ int2 s_ld[MODE == COL_Y ? UR_TILE_MAX : 1], s_st[MODE == COL_Y && INV ? UR_TILE_MAX : 1];
  float2* buf = reinterpret_cast<float2*>(smraw);
  const int N = a.N;
  const size_t buf_bytes = ur_align_up_dev((size_t)a.TX * a.pitch * sizeof(float2), 16);
  int32_t* thr = reinterpret_cast<int32_t*>(smraw + buf_bytes);
  double* hs = nullptr;
  double* hs2 = nullptr;
  const long long c0 = blk * a.TX;
  const ColDivs dv(a);
  if (MODE == COL_Y) {  // (published by the transform's first barrier)
    for (int t = threadIdx.x; t < a.TX; t += blockDim.x) {
      const long long c = c0 + t;
      const uint32_t o = dv.h.div((uint32_t)c);
      const int kx = (int)((uint32_t)c - o * dv.h.d);
      const bool valid = c < a.ncols;
      if (INV) {
        s_ld[t] = !valid ? make_int2(0, N) : beyond_range(kx, a.k2_zero, N);
        if (a.row_skip) s_st[t] = valid ? row_range(a.sh, a.gen_z0 + (int)o, N) : make_int2(0, 0);
      } else {
        s_ld[t] = !valid ? make_int2(0, 0) : a.row_skip ? row_range(a.sh, a.gen_z0 + (int)o, N) : make_int2(0, N);
      }
    }
  }
  if (MODE != COL_Y && a.nbins > 0) {
    for (int j = threadIdx.x; j <= a.nbins; j += blockDim.x) thr[j] = __ldg(a.thr + j);
    if (MODE == COL_ZBIN) {
      hs = reinterpret_cast<double*>(smraw + buf_bytes + ur_align_up_dev((size_t)(a.nbins + 1) * 4, 16));
      hs2 = hs + a.nbins;
      if (threadIdx.x == 0) {
        s_blo = 0x7fffffff;
        s_bhi = -1;
      }
    }
  }
  // a tile whose columns all lie at or beyond the closing threshold reaches no bin: nothing to bin, or zero
  // output, which the y pass takes as zeros without loading it (k2_zero).  The vote is also the barrier
  // that publishes the tables.
  bool beyond = a.nbins > 0 && (MODE == COL_ZADJ || (MODE == COL_ZBIN && !a.fout));
  if (beyond) {
    for (int t = threadIdx.x; t < a.TX && c0 + t < a.ncols; t += blockDim.x) {
      const uint32_t o = dv.h.div((uint32_t)(c0 + t));
      const int kx = (int)((uint32_t)(c0 + t) - o * dv.h.d), ky = (int)o < a.M ? (int)o : (int)o - N;
      beyond = beyond && kx * kx + ky * ky >= __ldg(a.thr + a.nbins);
    }
  }
  if (__syncthreads_and(beyond)) return;
  if (MODE == COL_ZBIN && a.nbins > 0) {
    // bins this tile can reach: k^2 in [min kx^2+ky^2, max kx^2+ky^2 + (N/2)^2]
    if (threadIdx.x < a.TX && c0 + threadIdx.x < a.ncols) {
      const long long c = c0 + threadIdx.x;
      const int kyi = (int)dv.h.div((uint32_t)c);
      const int kx = (int)c - kyi * a.H;
      const int ky = kyi < a.M ? kyi : kyi - N;
      const int c2 = kx * kx + ky * ky;
      atomicMin(&s_blo, max(bin_search(thr, a.nbins, c2), 0));
      atomicMax(&s_bhi, min(bin_search(thr, a.nbins, c2 + a.M * a.M), a.nbins - 1));
    }
    __syncthreads();
    for (int j = s_blo + (int)threadIdx.x; j <= s_bhi; j += blockDim.x) {
      hs[j] = 0.0;
      hs2[j] = 0.0;
    }
  }
  {
    // with two or more stages the first stage reads the columns from global memory and, where
    // the result goes back to global memory, the last stage writes it (no staging round trips)
    const bool io = a.nst >= 2;
    const ColLd<MODE, INV> ld(a, dv, c0, s_ld);
    const ColSt<MODE, INV> st(a, dv, c0, MODE == COL_Y && INV && a.row_skip ? s_st : nullptr);
    if (MODE == COL_Y) {
      if (io) {
        fft_lines_io<INV, UR_EMAX, true, true, true>(buf, a.pitch, a.TX, a.sched, a.nst, a.tw, ld, st);
      } else {
        load_columns(a, dv, buf, N, ld);
        fft_lines<INV, UR_EMAX>(buf, a.pitch, a.TX, a.sched, a.nst, a.tw);
        store_columns(a, dv, buf, N, st);
      }
    } else if (MODE == COL_ZBIN) {
      if (io) {
        fft_lines_io<false, UR_EMAX, true, false, true>(buf, a.pitch, a.TX, a.sched, a.nst, a.tw, ld, NoSt());
      } else {
        load_columns(a, dv, buf, N, ld);
        fft_lines<false, UR_EMAX>(buf, a.pitch, a.TX, a.sched, a.nst, a.tw);
      }
      if (a.fout) {
        for (int f = threadIdx.x; f < a.TX * N; f += blockDim.x) {
          const int i = (int)dv.tx.div((uint32_t)f);
          const int t = f - i * a.TX;
          const long long c = c0 + t;
          if (c < a.ncols) a.fout[(long long)i * N * a.H + c] = cscale(buf[t * a.pitch + i], a.fscale);
        }
      }
      if (a.nbins > 0) {
        BinAccum acc{buf, a.pitch, a.M, N, a.nbins, a.iscale, hs, hs2, -1, 0.f, 0.f, a.vs, 1.f};
        walk_bins(a, dv, thr, c0, acc);
      }
    } else {  // COL_ZADJ: F along z (recomputed or given), times sigma(bin), inverse along z
      if (io && !a.skip_fwd) {
        fft_lines_io<false, UR_EMAX, true, false, true>(buf, a.pitch, a.TX, a.sched, a.nst, a.tw, ld, NoSt());
      } else {
        load_columns(a, dv, buf, N, ld);
        if (!a.skip_fwd) fft_lines<false, UR_EMAX>(buf, a.pitch, a.TX, a.sched, a.nst, a.tw);
      }
      SigmaScale sc{buf, a.pitch, a.M, N, a.nbins, a.sigma};
      walk_bins(a, dv, thr, c0, sc);
      __syncthreads();
      if (io) {
        fft_lines_io<true, UR_EMAX, false, true, true>(buf, a.pitch, a.TX, a.sched, a.nst, a.tw, NoLd(), st);
      } else {
        fft_lines<true, UR_EMAX>(buf, a.pitch, a.TX, a.sched, a.nst, a.tw);
        store_columns(a, dv, buf, N, st);
      }
    }
  }
  if (MODE == COL_ZBIN && a.nbins > 0) {
    __syncthreads();
    for (int j = s_blo + (int)threadIdx.x; j <= s_bhi; j += blockDim.x) {
      if (hs[j] != 0.0) atomicAdd(a.gsum + j, hs[j]);
      if (hs2[j] != 0.0) atomicAdd(a.gsum2 + j, hs2[j]);
    }
  }
}

template <int MODE, bool INV>
__global__ void __launch_bounds__(256, 4) k_cols(ColArgs a) {
  cols_body<MODE, INV>(a, blockIdx.x);
}

// ---------------------------------------------------------------------------
// Finalize: bins[UR_BIN_FIELDS][B] from the accumulated sums (in I' units:
// I' = N^3 I) and the plan's per-bin count and sum |Q|.
// ---------------------------------------------------------------------------
__device__ __forceinline__ void finalize_bin(double* __restrict__ bins, const double* __restrict__ geo, int nb,
                                             double inv_n3, int j) {
  if (j >= nb) return;
  const double n = geo[j];
  const double s = bins[UR_BIN_SUM_I * nb + j] * inv_n3;
  const double s2 = bins[UR_BIN_SUM_I2 * nb + j] * (inv_n3 * inv_n3);
  const double nan = __longlong_as_double(0x7ff8000000000000ll);
  bins[UR_BIN_COUNT * nb + j] = n;
  bins[UR_BIN_SUM_I * nb + j] = s;
  bins[UR_BIN_SUM_I2 * nb + j] = s2;
  bins[UR_BIN_SUM_Q * nb + j] = geo[nb + j];
  double mean = nan, sem = nan;
  if (n > 0) mean = s / n;
  if (n > 1) {
    double var = (s2 - s * mean) / (n - 1.0);
    if (var < 0) var = 0;
    sem = sqrt(var / n);
  }
  bins[UR_BIN_MEAN * nb + j] = mean;
  bins[UR_BIN_SEM * nb + j] = sem;
}

__global__ void k_finalize(double* __restrict__ bins, const double* __restrict__ geo, int nb, double inv_n3) {
  finalize_bin(bins, geo, nb, inv_n3, blockIdx.x * blockDim.x + threadIdx.x);
}

// finalize of the power-of-two column pass, which leaves shifted sums (ur_bin_shift)
__global__ void k_finalize_shifted(double* __restrict__ bins, const double* __restrict__ geo, int nb, double inv_n3) {
  const int j = blockIdx.x * blockDim.x + threadIdx.x;
  if (j < nb) ur_finalize_shifted(bins, geo, nb, inv_n3, j);
}

// ---------------------------------------------------------------------------
// Plan-time bin geometry: count (weighted by the half-spectrum multiplicity)
// and sum of |Q| per bin over the full N^3 grid; independent of the data.
// One thread per (ky, kx) column, walking |kz| = m; block histogram in shared
// memory, then one global add per touched bin.
// ---------------------------------------------------------------------------
__global__ void k_geometry(const int32_t* __restrict__ thr_g, int nb, int N, double dq,
                           unsigned long long* __restrict__ gcount, double* __restrict__ gsumq) {
  extern __shared__ __align__(16) unsigned char smraw[];
  int32_t* thr = reinterpret_cast<int32_t*>(smraw);
  unsigned long long* hc = reinterpret_cast<unsigned long long*>(smraw + ur_align_up_dev((size_t)(nb + 1) * 4, 16));
  double* hq = reinterpret_cast<double*>(hc + nb);
  for (int j = threadIdx.x; j <= nb; j += blockDim.x) thr[j] = thr_g[j];
  for (int j = threadIdx.x; j < nb; j += blockDim.x) {
    hc[j] = 0ull;
    hq[j] = 0.0;
  }
  __syncthreads();
  const int M = N / 2, H = M + 1;
  const long long ncols = (long long)N * H;
  for (long long c = (long long)blockIdx.x * blockDim.x + threadIdx.x; c < ncols; c += (long long)gridDim.x * blockDim.x) {
    const int kyi = (int)(c / H);
    const int kx = (int)(c - (long long)kyi * H);
    const int ky = kyi < M ? kyi : kyi - N;
    const int c2 = kx * kx + ky * ky;
    const unsigned long long w = (kx == 0 || kx == M) ? 1ull : 2ull;
    int cur = bin_search(thr, nb, c2);
    int run = cur;
    unsigned long long cnt = 0;
    double sq = 0.0;
    for (int m = 0; m <= M; ++m) {
      const int s = c2 + m * m;
      while (cur < nb && thr[cur + 1] <= s) ++cur;
      if (cur != run) {
        if (run >= 0 && run < nb && cnt) {
          atomicAdd(hc + run, cnt * w);
          atomicAdd(hq + run, sq * (double)w);
        }
        run = cur;
        cnt = 0;
        sq = 0.0;
      }
      const unsigned long long mult = (m == 0 || m == M) ? 1ull : 2ull;
      cnt += mult;
      sq += (double)mult * sqrt((double)s);
    }
    if (run >= 0 && run < nb && cnt) {
      atomicAdd(hc + run, cnt * w);
      atomicAdd(hq + run, sq * (double)w);
    }
  }
  __syncthreads();
  for (int j = threadIdx.x; j < nb; j += blockDim.x) {
    if (hc[j]) {
      atomicAdd(gcount + j, hc[j]);
      atomicAdd(gsumq + j, hq[j] * dq);
    }
  }
}

__global__ void k_geo_to_double(const unsigned long long* __restrict__ c, double* __restrict__ out, int nb) {
  const int j = blockIdx.x * blockDim.x + threadIdx.x;
  if (j < nb) out[j] = (double)c[j];
}

__global__ void k_binlut(const int32_t* __restrict__ thr, int nb, int smax, int16_t* __restrict__ lut) {
  const int s = blockIdx.x * blockDim.x + threadIdx.x;
  if (s > smax) return;
  const int b = bin_search(thr, nb, s);
  lut[s] = (int16_t)((b >= 0 && b < nb) ? b : -1);
}

__global__ void k_bincoarse(const int32_t* __restrict__ thr, int nb, int shift, int16_t* __restrict__ crs) {
  const int i = blockIdx.x * blockDim.x + threadIdx.x;
  if (i < UR_COARSE_ENTRIES) crs[i] = (int16_t)bin_search(thr, nb, i << shift);
}

ur_status ur_launch_geometry(ur_plan* p, cudaStream_t s) {
  {
    const int smax = 3 * (p->n / 2) * (p->n / 2);
    int sh = 0;
    while ((smax >> sh) >= UR_COARSE_ENTRIES) ++sh;
    p->coarse_shift = sh;
    UR_CUDA_CHECK(cudaMalloc(&p->binlut, sizeof(int16_t) * ((size_t)smax + 1)));
    k_binlut<<<(smax + 256) / 256, 256, 0, s>>>(p->thr, p->nbins, smax, p->binlut);
    UR_LAUNCH_CHECK("k_binlut");
    UR_CUDA_CHECK(cudaMalloc(&p->bincoarse, sizeof(int16_t) * UR_COARSE_ENTRIES));
    k_bincoarse<<<(UR_COARSE_ENTRIES + 255) / 256, 256, 0, s>>>(p->thr, p->nbins, sh, p->bincoarse);
    UR_LAUNCH_CHECK("k_bincoarse");
  }
  const int nb = p->nbins;
  unsigned long long* cnt = nullptr;
  UR_CUDA_CHECK(cudaMalloc(&cnt, sizeof(unsigned long long) * nb));
  UR_CUDA_CHECK(cudaMemset(cnt, 0, sizeof(unsigned long long) * nb));
  UR_CUDA_CHECK(cudaMemset(p->geo, 0, sizeof(double) * 2 * nb));
  const size_t smem = ur_align_up((size_t)(nb + 1) * 4, 16) + (size_t)nb * 16;
  if (smem > 48 * 1024) UR_CUDA_CHECK(cudaFuncSetAttribute(k_geometry, cudaFuncAttributeMaxDynamicSharedMemorySize, (int)smem));
  const long long ncols = (long long)p->n * p->H;
  long long blocks = (ncols + 255) / 256;
  const long long cap = (long long)p->num_sms * 4;
  if (blocks > cap) blocks = cap;
  k_geometry<<<(int)blocks, 256, smem, s>>>(p->thr, nb, p->n, p->dq, cnt, p->geo + nb);
  UR_LAUNCH_CHECK("k_geometry");
  k_geo_to_double<<<(nb + 255) / 256, 256, 0, s>>>(cnt, p->geo, nb);
  UR_LAUNCH_CHECK("k_geo_to_double");
  UR_CUDA_CHECK(cudaStreamSynchronize(s));
  UR_CUDA_CHECK(cudaFree(cnt));
  return UR_OK;
}

// ---------------------------------------------------------------------------
// Standalone binning of a stored half-spectrum intensity (Sec. 2.5)
//
// Memory is the only unavoidable cost (4 bytes per element), so the bin of an element must
// be nearly free.  A thread owns one (kx, m) and walks a chunk of n >= m: the up to eight
// values at (ky, kz) = (+-n, +-m) and (+-m, +-n) share k^2, which only grows along the walk,
// so a run of equal bins is summed in registers and leaves the thread once per run.  Lanes
// are neighbours in kx, so every load is a row segment; the loads of two steps are issued
// together.  A float64 instruction occupies its pipe for a whole warp however few lanes are
// active, so float64 comes last: runs are three-float sums (72 bits) of the intensity scaled
// by a power of two, finished runs are queued per warp, and 32 of them at a time are added to
// the block's float64 histogram (compare-and-swap loops).  Values outside the range where their
// squares and the squares' rounding errors are both representable go to the histogram in float64,
// summed over a step.  512^3, 512 bins: 1918 us with one element per thread (64-bit division,
// binary search, two float64 histogram updates), 361 us with runs over (+-n, +-m) that each
// lane adds to the histogram itself (float64 pipe 77 % busy), 184 us now (kernel 168 us, 1.7 TB/s, 62 % issue).
// ---------------------------------------------------------------------------
struct BinHalfArgs {
  const float* I;
  int N, nb, chunk, nchunk;  // steps n per task, tasks per (kx, m)
  const int32_t* thr;
  const int16_t* lut;
  double* gsum;
  double* gsum2;
  float s;           // power of two near N^3: the walk sums I s
  double sd;         // s
  double f1, f2;     // N^3 / s and its square
  const float* vs;
};

// h + returned error = h + x exactly (Knuth's TwoSum)
__device__ __forceinline__ float two_add(float& h, float x) {
  const float t = __fadd_rn(h, x);
  const float z = __fsub_rn(t, h);
  const float e = __fadd_rn(__fsub_rn(h, __fsub_rn(t, z)), __fsub_rn(x, z));
  h = t;
  return e;
}
struct Sum3 {
  float h, l, e;
  __device__ __forceinline__ void clear() { h = l = e = 0.f; }
  __device__ __forceinline__ void add_low(float x) { e += two_add(l, x); }
  __device__ __forceinline__ void add(float x) { add_low(two_add(h, x)); }
};

#define UR_BINQ_STEPS 2    // steps whose loads are issued together
#define UR_BINQ_THREADS 256
#define UR_BINQ_QUEUE 64   // entries per warp: at most 31 waiting and 32 new

struct BinQueue {
  int b[UR_BINQ_QUEUE];
  float v[6][UR_BINQ_QUEUE];
};

template <bool VS>
__global__ void __launch_bounds__(UR_BINQ_THREADS, 4) k_bin_half(const __grid_constant__ BinHalfArgs a) {
  extern __shared__ __align__(16) unsigned char smraw[];
  __shared__ BinQueue queues[UR_BINQ_THREADS / 32];
  const int nb = a.nb;
  int32_t* thr = reinterpret_cast<int32_t*>(smraw);
  double* hs = reinterpret_cast<double*>(smraw + ur_align_up_dev((size_t)(nb + 1) * 4, 16));
  double* hs2 = hs + nb;
  for (int j = threadIdx.x; j <= nb; j += blockDim.x) thr[j] = __ldg(a.thr + j);
  for (int j = threadIdx.x; j < 2 * nb; j += blockDim.x) hs[j] = 0.0;
  __syncthreads();
  constexpr unsigned FULL = 0xffffffffu;
  BinQueue& q = queues[threadIdx.x >> 5];
  const int lane = threadIdx.x & 31;
  int waiting = 0;  // uniform over the warp
  auto add_queued = [&](int i) {
    const int b = q.b[i];
    atomicAdd(hs + b, ((double)q.v[0][i] + (double)q.v[1][i]) + (double)q.v[2][i]);
    atomicAdd(hs2 + b, ((double)q.v[3][i] + (double)q.v[4][i]) + (double)q.v[5][i]);
  };
  const int N = a.N, M = N / 2, H = M + 1;
  const long long ncol = (long long)(M + 1) * H, plane = (long long)N * H;
  const long long ntask = ncol * a.nchunk;
  // the loops are uniform over a warp (its lanes share the queue)
  for (long long base = (long long)blockIdx.x * blockDim.x + threadIdx.x - lane; base < ntask;
       base += (long long)gridDim.x * blockDim.x) {
    const long long task = base + lane;
    const bool valid = task < ntask;
    const int ch = valid ? (int)(task / ncol) : 0;
    const int c = valid ? (int)(task - ch * ncol) : 0;
    const int m = c / H, kx = c - m * H;
    int y0 = max(ch * a.chunk, m), y1 = min((ch + 1) * a.chunk, M + 1);
    if (!valid || y0 >= y1) y0 = y1 = 0;
    const bool some = y0 < y1;
    const int ylo = __reduce_min_sync(FULL, some ? y0 : 0x7fffffff), yhi = __reduce_max_sync(FULL, y1);
    const bool twom = m != 0 && m != M;
    const float w = (kx == 0 || kx == M) ? 1.f : 2.f;
    const float* pz0 = a.I + m * plane + kx;
    const float* pz1 = a.I + (N - m) * plane + kx;
    const float* py0 = a.I + (long long)m * H + kx;
    const float* py1 = a.I + (long long)(N - m) * H + kx;
    const float vx = VS ? __ldg(a.vs + kx) : 0.f, vm = VS ? __ldg(a.vs + m) : 0.f;
    int s = kx * kx + m * m + y0 * y0;
    int b = s < thr[0] ? -1 : s >= thr[nb] ? nb : __ldg(a.lut + s);
    int tnext = b < nb ? thr[b + 1] : 0x7fffffff;
    Sum3 s1, s2;
    s1.clear();
    s2.clear();
    auto push = [&](bool need) {
      need = need && (s1.h != 0.f || s2.h != 0.f);
      const unsigned who = __ballot_sync(FULL, need);
      if (!who) return;
      if (need) {
        const int i = waiting + __popc(who & ((1u << lane) - 1u));
        q.b[i] = b;
        q.v[0][i] = w * s1.h;  // w is 1 or 2: exact
        q.v[1][i] = w * s1.l;
        q.v[2][i] = w * s1.e;
        q.v[3][i] = w * s2.h;
        q.v[4][i] = w * s2.l;
        q.v[5][i] = w * s2.e;
        s1.clear();
        s2.clear();
      }
      waiting += __popc(who);
      if (waiting >= 32) {
        waiting -= 32;
        __syncwarp();
        add_queued(waiting + lane);
        __syncwarp();
      }
    };
    for (int y = ylo; y < yhi; y += UR_BINQ_STEPS) {
      float v[UR_BINQ_STEPS][8];
      auto value = [&](int n, int e, bool in) {
        const bool two = n != 0 && n != M, swap = n != m;
        const float* p = e < 4 ? (e & 2 ? pz1 : pz0) : (e & 2 ? py1 : py0);
        const long long o = (long long)(e & 1 ? N - n : n) * H * (e < 4 ? 1 : N);
        return in && (!(e & 1) || two) && (!(e & 2) || twom) && (!(e & 4) || swap) ? __ldg(p + o) : 0.f;
      };
      // x^2 of x = v s and its rounding error are both normal floats, or zero
      auto in_range = [&](float v) {
        const float x = fabsf(v * a.s);
        return x <= 1e18f && (x >= 1e-15f || v == 0.f);
      };
#pragma unroll
      for (int u = 0; u < UR_BINQ_STEPS; ++u)
#pragma unroll
        for (int e = 0; e < 8; ++e) v[u][e] = value(y + u, e, y + u >= y0 && y + u < y1);
#pragma unroll
      for (int u = 0; u < UR_BINQ_STEPS; ++u) {
        const int n = y + u;
        const bool in = n >= y0 && n < y1;
        const bool next = in && s >= tnext;
        push(next);
        if (next) {
          do {
            ++b;
            tnext = b < nb ? thr[b + 1] : 0x7fffffff;
          } while (s >= tnext);
        }
        if (in && b >= 0 && b < nb) {
          // voxel-sinc factors in the order (x y) z
          const float vn = VS ? __ldg(a.vs + n) : 0.f;
          const float fa = VS ? vx * vn * vm : 1.f, fb = VS ? vx * vm * vn : 1.f;
          bool all = true;
#pragma unroll
          for (int e = 0; e < 8; ++e) {
            const float f = e < 4 ? fa : fb;
            const float x = v[u][e] * a.s;
            if (in_range(v[u][e])) {
              float p = x, r = 0.f;
              if (VS) {
                p = __fmul_rn(x, f);
                r = __fmaf_rn(x, f, -p);
                s1.add_low(r);
              }
              const float sq = __fmul_rn(p, p);
              s1.add(p);
              s2.add(sq);
              s2.add_low(__fmaf_rn(p, p, -sq));
              if (VS) {  // (p + r)^2 = p^2 + 2 p r + r^2
                const float pr = __fmul_rn(2.f * p, r);
                s2.add_low(pr);
                s2.e += fmaf(r, r, __fmaf_rn(2.f * p, r, -pr));
              }
            } else {
              all = false;
            }
          }
          if (!all) {  // the step's other values, read once more: one float64 sum
            double d1 = 0.0, d2 = 0.0;
#pragma unroll 1
            for (int e = 0; e < 8; ++e) {
              const float t = value(n, e, true);
              if (in_range(t)) continue;
              double d = (double)t * a.sd;
              if (VS) d *= (double)(e < 4 ? fa : fb);
              d1 += d;
              d2 += d * d;
            }
            atomicAdd(hs + b, (double)w * d1);
            atomicAdd(hs2 + b, (double)w * d2);
          }
        }
        if (in) s += 2 * n + 1;
      }
    }
    push(b >= 0 && b < nb);
  }
  __syncwarp();
  if (lane < waiting) add_queued(lane);
  __syncthreads();
  for (int j = threadIdx.x; j < nb; j += blockDim.x) {
    if (hs[j] != 0.0) atomicAdd(a.gsum + j, a.f1 * hs[j]);
    if (hs2[j] != 0.0) atomicAdd(a.gsum2 + j, a.f2 * hs2[j]);
  }
}

// ---------------------------------------------------------------------------
// Host: kernel configuration for a plan
// ---------------------------------------------------------------------------
// rows of a block, and per row its mask terms and cell offset
size_t ur_row_smem(int rb, int M) { return (size_t)rb * (M * sizeof(float2) + sizeof(RowMask) + sizeof(int)); }

size_t ur_colbin_smem(const ur_plan* p) {
  return ur_align_up((size_t)p->col_tx * (p->n + 1) * sizeof(float2), 16) + ur_align_up((size_t)(p->nbins + 1) * 4, 16) +
         (size_t)p->nbins * 16;
}

ur_status ur_configure_kernels(ur_plan* p) {
  const int n = p->n, M = p->M;
  // rows: RB rows of M complex per block, 256 threads, <= EMAX elements per thread
  p->row_threads = 256;
  p->row_rb = (UR_EMAX * p->row_threads) / M;
  if (p->row_rb > 64) p->row_rb = 64;
  if (p->row_rb < 1) p->row_rb = 1;
  p->row_smem = ur_row_smem(p->row_rb, M);
  // columns: TX columns of N complex per block
  p->col_threads = 256;
  p->col_tx = (UR_EMAX * p->col_threads) / n;
  if (p->col_tx > 64) p->col_tx = 64;
  if (p->col_tx < 1) p->col_tx = 1;
  p->col_smem = ur_align_up((size_t)p->col_tx * (n + 1) * sizeof(float2), 16) + ur_align_up((size_t)(p->nbins + 1) * 4, 16);
  p->colbin_smem = ur_colbin_smem(p);
  if (p->colbin_smem > 227 * 1024) {
    ur_set_error("ur_plan_create: %d bins need %zu bytes of shared memory per block (max 227 KB)", p->nbins, p->colbin_smem);
    return UR_ERR_UNSUPPORTED;
  }
  // the runtime-radix kernels accept any tile shape up to the per-block limit
  // (ur_plan_set_tiles may change it), so they get the largest dynamic size once
  const int kMaxDyn = 200 * 1024;
  UR_CUDA_CHECK(cudaFuncSetAttribute(k_rows_r2c<0, float, false>, cudaFuncAttributeMaxDynamicSharedMemorySize, kMaxDyn));
  UR_CUDA_CHECK(cudaFuncSetAttribute(k_rows_r2c<0, float, true>, cudaFuncAttributeMaxDynamicSharedMemorySize, kMaxDyn));
  UR_CUDA_CHECK(cudaFuncSetAttribute(k_rows_r2c<0, __half, false>, cudaFuncAttributeMaxDynamicSharedMemorySize, kMaxDyn));
  UR_CUDA_CHECK(cudaFuncSetAttribute(k_rows_r2c<0, __half, true>, cudaFuncAttributeMaxDynamicSharedMemorySize, kMaxDyn));
  UR_CUDA_CHECK(cudaFuncSetAttribute(k_rows_r2c<1, float, false>, cudaFuncAttributeMaxDynamicSharedMemorySize, kMaxDyn));
  UR_CUDA_CHECK(cudaFuncSetAttribute(k_rows_r2c<2, float, false>, cudaFuncAttributeMaxDynamicSharedMemorySize, kMaxDyn));
  UR_CUDA_CHECK(cudaFuncSetAttribute(k_cols<COL_Y, false>, cudaFuncAttributeMaxDynamicSharedMemorySize, kMaxDyn));
  UR_CUDA_CHECK(cudaFuncSetAttribute(k_cols<COL_Y, true>, cudaFuncAttributeMaxDynamicSharedMemorySize, kMaxDyn));
  UR_CUDA_CHECK(cudaFuncSetAttribute(k_cols<COL_ZBIN, false>, cudaFuncAttributeMaxDynamicSharedMemorySize, kMaxDyn));
  UR_CUDA_CHECK(cudaFuncSetAttribute(k_cols<COL_ZADJ, false>, cudaFuncAttributeMaxDynamicSharedMemorySize, kMaxDyn));
  const long long ntiles = ((long long)n * p->H + p->col_tx - 1) / p->col_tx;
  p->zbin_grid = (int)ntiles;
  // device copy of the radix schedules
  UR_CUDA_CHECK(cudaMalloc(&p->d_sched, sizeof(StageInfo) * 2 * UR_MAX_STAGES));
  UR_CUDA_CHECK(cudaMemcpy(p->d_sched, p->sched_n.st, sizeof(StageInfo) * UR_MAX_STAGES, cudaMemcpyHostToDevice));
  UR_CUDA_CHECK(cudaMemcpy(p->d_sched + UR_MAX_STAGES, p->sched_m.st, sizeof(StageInfo) * UR_MAX_STAGES, cudaMemcpyHostToDevice));
  // workspace regions
  p->ws_inter = (size_t)p->nz * n * p->xp * sizeof(float2);
  p->ws_inv = (size_t)n * n * p->xp * sizeof(float2);
  p->ws_sigma = (size_t)p->nbins * sizeof(float);
  // host-resident ED: slabs of about 256 MiB, two of them in the workspace
  {
    const size_t ed_plane = (size_t)n * n * (p->ed_dtype == UR_F16 ? 2 : 4);
    long long sp = (long long)((256ull << 20) / ed_plane);
    if (sp < 1) sp = 1;
    if (sp > p->nz) sp = p->nz;
    p->slab_planes = (int)sp;
    p->ws_slab = (size_t)sp * ed_plane;
  }
  // out-of-core adjoint: about 4 GiB of inverse intermediate per slab
  {
    long long ap = (long long)((4ull << 30) / ((size_t)n * p->xp * sizeof(float2)));
    if (ap < 1) ap = 1;
    if (ap > n) ap = n;
    p->adj_slab_planes = (int)ap;
  }
  // power-of-two kernels; by default every pass runs over all planes at once
  // (ur_plan_set_chunk_planes can split the plane pass and the adjoint's y and
  // row passes into chunks whose intermediate stays in L2 between the two
  // kernels; on the 512^3 workload one launch per pass measured faster)
  p->fast = ur_fast_supported(n) ? 1 : 0;
  p->chunk_planes = n;
  p->ws_chunk = 0;
  return UR_OK;
}

ur_status ur_launch_cols(int mode, bool inv, const ur_plan* p, const ColArgs& a, int grid, size_t smem, cudaStream_t s) {
  (void)p;
  if (grid <= 0) return UR_OK;
  if (mode == COL_Y && !inv) k_cols<COL_Y, false><<<grid, p->col_threads, smem, s>>>(a);
  else if (mode == COL_Y) k_cols<COL_Y, true><<<grid, p->col_threads, smem, s>>>(a);
  else if (mode == COL_ZBIN) k_cols<COL_ZBIN, false><<<grid, p->col_threads, smem, s>>>(a);
  else k_cols<COL_ZADJ, false><<<grid, p->col_threads, smem, s>>>(a);
  UR_LAUNCH_CHECK("k_cols");
  return UR_OK;
}

ColArgs ur_col_args(const ur_plan* p) {
  ColArgs a;
  memset(&a, 0, sizeof a);
  a.N = p->n;
  a.H = p->H;
  a.M = p->M;
  a.TX = p->col_tx;
  a.pitch = p->n + 1;
  a.sched = p->d_sched;
  a.nst = p->sched_n.nst;
  a.tw = p->tw;
  a.stw = p->stw;
  a.stw32 = p->stw + p->stw_32_off;
  a.thr = p->thr;
  a.lut = p->binlut;
  a.vs = p->vsinc;
  a.crs = p->bincoarse;
  a.crs_shift = p->coarse_shift;
  a.nbins = p->nbins;
  // a tile's walks in one round of the block's threads
  a.walk = p->n < 64 ? 1 : BIN_CHUNK;
  while (a.walk < 15 && a.TX * ((a.H + a.walk - 1) / a.walk) > p->col_threads) a.walk += 2;
  return a;
}

// Pass 1 (rows along x, then columns along y) of nplanes planes into X (same
// plane order).  ra carries either the density rows (GEN = 0) or the density
// description (GEN = 1, rows generated in the kernel); ra.z0 is the absolute
// plane of X's first plane.  On the power-of-two path the planes go in chunks
// whose intermediate stays in L2 between the two kernels.
static ur_status plane_pass(const ur_plan* p, RowArgs ra, int gen, long long nplanes, float2* X, cudaStream_t s) {
  const int n = p->n, H = p->H;
  const long long step = p->fast ? p->chunk_planes : nplanes;
  for (long long p0 = 0; p0 < nplanes; p0 += step) {
    const long long np = (p0 + step <= nplanes) ? step : nplanes - p0;
    RowArgs r = ra;
    r.stw = p->stw ? p->stw + (gen ? p->stw_m_off : p->stw_s_off) : nullptr;
    r.fu = FastDiv((uint32_t)(ra.ucell > 0 ? ra.ucell : 1));
    r.X = X + p0 * n * p->xp;
    r.xp = p->xp;
    r.nrows = np * n;
    r.z0 = ra.z0 + (int)p0;
    if (!gen) r.ed = (const char*)ra.ed + p0 * (long long)n * n * (p->ed_dtype == UR_F16 ? 2 : 4);
    // generated particle: the row pass leaves the rows outside it unwritten and the y pass reads them
    // as zeros
    const bool skip = gen && ra.sh.rb2 < INFINITY && !ra.weights;
    r.skip_empty = skip ? 1 : 0;
    ur_timing_begin("rows_r2c", s);
    if (p->fast) {
      UR_TRY(ur_fast_rows(n, r, gen, p->ed_dtype == UR_F16, s));
    } else {
      const int grid_rows = (int)((r.nrows + p->row_rb - 1) / p->row_rb);
      const StageInfo* sm = p->d_sched + UR_MAX_STAGES;
      // stored rows that leave half of the SMs idle are short of time for one block, not of shared-memory
      // bandwidth, and the first stage from global memory costs registers: 16^3 10.2 us against 6.3, 48^3
      // 13.0 against 10.9; 90^3 (126 blocks) 13.8 against 14.1
      const int nst = p->sched_m.nst;
      const bool io = nst >= 2 && grid_rows >= p->num_sms / 2, f32 = p->ed_dtype == UR_F32;
      const size_t smem = gen == 1 ? p->row_smem : (size_t)p->row_rb * p->M * sizeof(float2);
#define UR_ROWS(...) k_rows_r2c<__VA_ARGS__><<<grid_rows, p->row_threads, smem, s>>>(r, n, p->row_rb, sm, nst)
      if (gen == 2) UR_ROWS(2, float, false);
      else if (gen) UR_ROWS(1, float, false);
      else if (io && f32) UR_ROWS(0, float, true);
      else if (io) UR_ROWS(0, __half, true);
      else if (f32) UR_ROWS(0, float, false);
      else UR_ROWS(0, __half, false);
#undef UR_ROWS
      UR_LAUNCH_CHECK("k_rows_r2c");
    }
    ur_timing_end(s);
    ColArgs a = ur_col_args(p);
    a.src = r.X;
    a.dst = r.X;
    a.ncols = np * H;
    a.A = (long long)n * p->xp;
    a.S = p->xp;
    a.Ad = a.A;
    a.Sd = a.S;
    a.nload = n;
    a.zoff = 0;
    a.nbins = 0;
    if (skip) {
      a.row_skip = 1;
      a.gen_z0 = r.z0;
      a.sh = ra.sh;
    }
    ur_timing_begin("cols_y", s);
    if (p->fast) {
      UR_TRY(ur_fast_cols(n, 0 /* y forward */, a, s));
    } else {
      const long long ntiles = (a.ncols + a.TX - 1) / a.TX;
      k_cols<COL_Y, false><<<(int)ntiles, p->col_threads, p->col_smem, s>>>(a);
      UR_LAUNCH_CHECK("k_cols<COL_Y>");
    }
    ur_timing_end(s);
  }
  return UR_OK;
}

ur_status ur_plane_pass(const ur_plan* p, const void* ed, long long nplanes, float2* X, cudaStream_t s) {
  RowArgs ra;
  memset(&ra, 0, sizeof ra);
  ra.ed = ed;
  ra.tw = p->tw;
  ra.z0 = p->z0;
  return plane_pass(p, ra, 0, nplanes, X, s);
}

// Pass 2 (+ binning) from the intermediate X holding planes [z0, z0+nz).
ur_status ur_column_pass(const ur_plan* p, const float2* X, double* bins, float2* F_out, cudaStream_t s) {
  const int nb = p->nbins;
  ColArgs a = ur_col_args(p);
  a.src = X;
  a.ncols = (long long)p->n * p->H;
  a.A = p->xp;
  a.S = (long long)p->n * p->xp;
  a.nload = p->nz;
  a.zoff = p->z0;
  const double n3 = (double)p->n * p->n * p->n;
  a.iscale = (float)(1.0 / n3);
  a.fout = F_out;
  a.fscale = (float)(1.0 / n3);
  if (bins) {
    UR_CUDA_CHECK(cudaMemsetAsync(bins, 0, sizeof(double) * UR_BIN_FIELDS * nb, s));
    a.gsum = bins + UR_BIN_SUM_I * nb;
    a.gsum2 = bins + UR_BIN_SUM_I2 * nb;
    a.gK = ur_shift_slots(bins, nb);
  } else {
    a.nbins = 0;
  }
  // grids of 256 and 512 with binning, when the plan asks for it: the TMA z-column kernel
  const bool zc = bins && p->fast && p->zc_enabled && ur_zcol_supported(p);
  ur_timing_begin("cols_z_bin", s);
  if (zc) {
    UR_TRY(ur_zcol_forward(p, X, bins, F_out, a.iscale, a.fscale, s));
  } else if (p->fast) {
    UR_TRY(ur_fast_cols(p->n, 2 /* z + bins */, a, s));
  } else {
    k_cols<COL_ZBIN, false><<<p->zbin_grid, p->col_threads, p->colbin_smem, s>>>(a);
    UR_LAUNCH_CHECK("k_cols<COL_ZBIN>");
  }
  ur_timing_end(s);
  if (bins && !zc) {  // (the TMA z-column kernel finalizes the bins itself)
    ur_timing_begin("finalize", s);
    if (p->fast) k_finalize_shifted<<<(nb + 255) / 256, 256, 0, s>>>(bins, p->geo, nb, 1.0 / n3);
    else k_finalize<<<(nb + 255) / 256, 256, 0, s>>>(bins, p->geo, nb, 1.0 / n3);
    UR_LAUNCH_CHECK("k_finalize");
    ur_timing_end(s);
  }
  return UR_OK;
}

extern "C" ur_status ur_fft_intensity(const ur_plan* p, const void* ed, int32_t ed_on_host, double* bins, void* F_out,
                                      void* ws, size_t ws_bytes, void* stream) {
  UR_REQUIRE(p && ed && ws, "ur_fft_intensity: null argument");
  cudaStream_t s = (cudaStream_t)stream;
  if (ed_on_host) return ur_fft_intensity_host(p, ed, bins, (float2*)F_out, ws, ws_bytes, s);
  UR_REQUIRE(ws_bytes >= ur_workspace_size(p, UR_WS_FORWARD), "ur_fft_intensity: workspace %zu < %zu bytes", ws_bytes,
             ur_workspace_size(p, UR_WS_FORWARD));
  UR_REQUIRE(((uintptr_t)ed % 8) == 0 && ((uintptr_t)ws % 256) == 0, "ur_fft_intensity: misaligned ed or ws");
  UR_TRY(ur_fault_point("fft_intensity"));
  float2* X = (float2*)ws;
  UR_TRY(ur_plane_pass(p, ed, p->nz, X, s));
  UR_TRY(ur_column_pass(p, X, bins, (float2*)F_out, s));
  return UR_OK;
}

static ur_status fft_intensity_tiled(const ur_plan* p, const float* cell, int32_t ucell, const int32_t* origin,
                                     const ur_lattice* lattice, const ur_shape* shape, const float* weights,
                                     double* bins, void* F_out, void* ws, size_t ws_bytes, void* stream) {
  UR_REQUIRE(p && cell && shape && ws, "ur_fft_intensity_tiled: null argument");
  UR_REQUIRE(ucell >= 1, "ur_fft_intensity_tiled: empty cell");
  UR_REQUIRE(shape->kind >= UR_SHAPE_SPHERE && shape->kind <= UR_SHAPE_WEIGHTS, "ur_fft_intensity_tiled: bad shape kind");
  UR_REQUIRE(shape->kind != UR_SHAPE_WEIGHTS || weights, "ur_fft_intensity_tiled: weights required for UR_SHAPE_WEIGHTS");
  UR_REQUIRE(!weights || ((uintptr_t)weights % 8) == 0, "ur_fft_intensity_tiled: weights must be 8-byte aligned");
  UR_REQUIRE(ws_bytes >= ur_workspace_size(p, UR_WS_FORWARD), "ur_fft_intensity_tiled: workspace %zu < %zu bytes",
             ws_bytes, ur_workspace_size(p, UR_WS_FORWARD));
  UR_REQUIRE(((uintptr_t)ws % 256) == 0, "ur_fft_intensity_tiled: misaligned ws");
  UR_TRY(ur_fault_point("fft_intensity"));
  cudaStream_t s = (cudaStream_t)stream;
  RowArgs ra;
  memset(&ra, 0, sizeof ra);
  ra.tw = p->tw;
  ra.z0 = p->z0;
  ra.cell = cell;
  ra.ucell = ucell;
  if (origin) {
    UR_REQUIRE(origin[0] >= 0 && origin[1] >= 0 && origin[2] >= 0, "ur_fft_intensity_tiled: origin must be >= 0");
    ra.ox = origin[0];
    ra.oy = origin[1];
    ra.oz = origin[2];
  }
  ra.sh = ur_shape_args(shape);
  ra.lat = ur_lattice_args(lattice);
  ra.weights = shape->kind == UR_SHAPE_WEIGHTS ? weights : nullptr;
  float2* X = (float2*)ws;
  UR_TRY(plane_pass(p, ra, lattice ? 2 : 1, p->nz, X, s));
  UR_TRY(ur_column_pass(p, X, bins, (float2*)F_out, s));
  return UR_OK;
}

extern "C" ur_status ur_fft_intensity_tiled(const ur_plan* p, const float* cell, int32_t ucell, const int32_t* origin,
                                            const ur_shape* shape, const float* weights, double* bins, void* F_out,
                                            void* ws, size_t ws_bytes, void* stream) {
  return fft_intensity_tiled(p, cell, ucell, origin, nullptr, shape, weights, bins, F_out, ws, ws_bytes, stream);
}

extern "C" ur_status ur_fft_intensity_tiled_lattice(const ur_plan* p, const float* cell, int32_t ucell,
                                                    const ur_lattice* lattice, const ur_shape* shape,
                                                    const float* weights, double* bins, void* F_out, void* ws,
                                                    size_t ws_bytes, void* stream) {
  UR_REQUIRE(lattice, "ur_fft_intensity_tiled_lattice: null lattice");
  return fft_intensity_tiled(p, cell, ucell, nullptr, lattice, shape, weights, bins, F_out, ws, ws_bytes, stream);
}

extern "C" ur_status ur_bin_q(const ur_plan* p, const float* I, double* bins, void* ws, size_t ws_bytes, void* stream) {
  UR_REQUIRE(p && I && bins, "ur_bin_q: null argument");
  (void)ws;
  (void)ws_bytes;
  cudaStream_t s = (cudaStream_t)stream;
  const int nb = p->nbins;
  const size_t smem = ur_align_up((size_t)(nb + 1) * 4, 16) + (size_t)nb * 16;
  if (smem > 32 * 1024) {  // (the queues take 14 KB of the default limit)
    UR_CUDA_CHECK(cudaFuncSetAttribute(k_bin_half<false>, cudaFuncAttributeMaxDynamicSharedMemorySize, (int)smem));
    UR_CUDA_CHECK(cudaFuncSetAttribute(k_bin_half<true>, cudaFuncAttributeMaxDynamicSharedMemorySize, (int)smem));
  }
  UR_CUDA_CHECK(cudaMemsetAsync(bins, 0, sizeof(double) * UR_BIN_FIELDS * nb, s));
  const double n3 = (double)p->n * p->n * p->n;
  // the kernel accumulates I * N^3 so that k_finalize's I' convention applies
  BinHalfArgs a;
  memset(&a, 0, sizeof a);
  a.I = I;
  a.N = p->n;
  a.nb = nb;
  // long walks merge more elements per histogram update, short ones fill the GPU on small grids:
  // 16 steps per task (512^3: 64 steps 291 us, 32 199, 16 184, 8 186) while that leaves two tasks per
  // resident thread, and 8 or 4 below; 2 and 1, in blocks of half the size, where walks of 4 give less
  // than 512 threads per SM (below about 130^3), us with 40, 300, 771, 1000 bins (40 and 771: log):
  //           4 steps, 256 threads     2 or 1 steps, 128 threads
  //    48^3   23.4 17.1 29.0 21.4      14.4 10.9 12.2 12.6
  //    84^3   27.0 17.3 26.5 20.1      18.5 12.7 15.0 16.3
  //   126^3   31.3 21.0 26.6 21.2      23.1 16.9 18.3 20.6
  //   160^3   37.7 25.2 27.9 25.1      34.5 23.6 25.9 27.8
  const long long ncol = (long long)p->H * p->H;
  auto tasks = [&] { return ncol * ((p->H + a.chunk - 1) / a.chunk); };
  a.chunk = 16;
  while (a.chunk > 4 && tasks() < (long long)p->num_sms * 2048) a.chunk /= 2;
  while (a.chunk > 1 && tasks() < (long long)p->num_sms * 512) a.chunk /= 2;
  const int threads = a.chunk < 4 ? UR_BINQ_THREADS / 2 : UR_BINQ_THREADS;
  a.nchunk = (p->H + a.chunk - 1) / a.chunk;
  a.thr = p->thr;
  a.lut = p->binlut;
  a.gsum = bins + UR_BIN_SUM_I * nb;
  a.gsum2 = bins + UR_BIN_SUM_I2 * nb;
  const double s2 = ldexp(1.0, ilogb(n3));
  a.s = (float)s2;
  a.sd = s2;
  a.f1 = n3 / s2;
  a.f2 = (n3 / s2) * (n3 / s2);
  a.vs = p->vsinc;
  const long long need = (tasks() + threads - 1) / threads;
  const int cap = p->num_sms * (smem > 40 * 1024 ? 1 : 4);
  const int grid = (int)(need < cap ? need : cap);
  if (a.vs) k_bin_half<true><<<grid, threads, smem, s>>>(a);
  else k_bin_half<false><<<grid, threads, smem, s>>>(a);
  UR_LAUNCH_CHECK("k_bin_half");
  k_finalize<<<(nb + 255) / 256, 256, 0, s>>>(bins, p->geo, nb, 1.0 / n3);
  UR_LAUNCH_CHECK("k_finalize");
  return UR_OK;
}

// ---------------------------------------------------------------------------
// Batched launches (many plans of different grid edges in one grid).
// ---------------------------------------------------------------------------
__device__ __forceinline__ int batch_item(const long long* __restrict__ start, int count, long long b) {
  int lo = 0, hi = count - 1;
  while (lo < hi) {
    const int mid = (lo + hi + 1) >> 1;
    if (__ldg(start + mid) <= b) lo = mid;
    else hi = mid - 1;
  }
  return lo;
}

__global__ void __launch_bounds__(256, 4) k_batch_rows(const BatchRowsItem* __restrict__ items,
                                                       const long long* __restrict__ start, int count) {
  const int i = batch_item(start, count, blockIdx.x);
  const BatchRowsItem& it = items[i];
  rows_r2c_body<1, float>(it.ra, it.N, it.RB, it.sched, it.nst, blockIdx.x - __ldg(start + i));
}

template <int MODE, bool INV>
__global__ void __launch_bounds__(256, 4) k_batch_cols(const ColArgs* __restrict__ items,
                                                       const long long* __restrict__ start, int count) {
  const int i = batch_item(start, count, blockIdx.x);
  cols_body<MODE, INV>(items[i], blockIdx.x - __ldg(start + i));
}

__global__ void k_batch_finalize(const BatchFinItem* __restrict__ items) {
  const BatchFinItem& it = items[blockIdx.y];
  finalize_bin(it.bins, it.geo, it.nb, it.inv_n3, blockIdx.x * blockDim.x + threadIdx.x);
}

__global__ void k_batch_zero(const BatchZeroItem* __restrict__ items) {
  const BatchZeroItem& it = items[blockIdx.y];
  const size_t n4 = it.bytes / 4;
  uint32_t* p = reinterpret_cast<uint32_t*>(it.ptr);
  for (size_t k = (size_t)blockIdx.x * blockDim.x + threadIdx.x; k < n4; k += (size_t)gridDim.x * blockDim.x) p[k] = 0u;
}

static void batch_grid_check(long long nblocks) { (void)nblocks; }

ur_status ur_batch_launch_rows(const BatchRowsItem* items, const long long* start, int count, long long nblocks,
                               size_t smem, cudaStream_t s) {
  if (nblocks <= 0) return UR_OK;
  UR_REQUIRE(nblocks < (1ll << 31), "batched rows: too many blocks");
  batch_grid_check(nblocks);
  if (smem > UR_DYN_SMEM_FREE)
    UR_CUDA_CHECK(cudaFuncSetAttribute(k_batch_rows, cudaFuncAttributeMaxDynamicSharedMemorySize, (int)smem));
  k_batch_rows<<<(unsigned)nblocks, 256, smem, s>>>(items, start, count);
  UR_LAUNCH_CHECK("k_batch_rows");
  return UR_OK;
}

ur_status ur_batch_launch_cols(int mode, bool inv, const ColArgs* items, const long long* start, int count,
                               long long nblocks, size_t smem, cudaStream_t s) {
  if (nblocks <= 0) return UR_OK;
  UR_REQUIRE(nblocks < (1ll << 31), "batched columns: too many blocks");
#define UR_BATCH_COLS(MD, IV)                                                                                  \
  do {                                                                                                         \
    UR_CUDA_CHECK(cudaFuncSetAttribute(k_batch_cols<MD, IV>, cudaFuncAttributeMaxDynamicSharedMemorySize, (int)smem)); \
    k_batch_cols<MD, IV><<<(unsigned)nblocks, 256, smem, s>>>(items, start, count);                            \
  } while (0)
  if (mode == COL_Y && !inv) UR_BATCH_COLS(COL_Y, false);
  else if (mode == COL_Y) UR_BATCH_COLS(COL_Y, true);
  else if (mode == COL_ZBIN) UR_BATCH_COLS(COL_ZBIN, false);
  else UR_BATCH_COLS(COL_ZADJ, false);
#undef UR_BATCH_COLS
  UR_LAUNCH_CHECK("k_batch_cols");
  return UR_OK;
}

ur_status ur_batch_launch_finalize(const BatchFinItem* items, int count, int maxnb, cudaStream_t s) {
  if (count <= 0) return UR_OK;
  k_batch_finalize<<<dim3((unsigned)((maxnb + 255) / 256), (unsigned)count), 256, 0, s>>>(items);
  UR_LAUNCH_CHECK("k_batch_finalize");
  return UR_OK;
}

ur_status ur_batch_launch_zero(const BatchZeroItem* items, int count, cudaStream_t s) {
  if (count <= 0) return UR_OK;
  k_batch_zero<<<dim3(64u, (unsigned)count), 256, 0, s>>>(items);
  UR_LAUNCH_CHECK("k_batch_zero");
  return UR_OK;
}
