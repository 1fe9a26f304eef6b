// Column passes of power-of-two grid edges 64 <= N <= 512: two columns per thread group, in
// packed float32 pairs.
//
// The column kernels are short of issue slots, not of float32 lanes or memory (60-66 % issue
// at 37-73 % of HBM with one column per thread group), and add/mul/fma.f32x2 do two IEEE
// operations per slot.  So a group of N/8 threads transforms two columns A and B at once: a
// value is (re A, re B), (im A, im B), and every butterfly, exchange, address and table
// lookup is shared by the two.  The pairs are chosen so that the rest is shared too:
//   z passes  A = (kx, ky), B = (kx, -ky): the same k^2 at every kz, so one walk of the bins
//             (one lookup of the adjoint's scale) serves four values instead of two.
//             ky = 0 and ky = N/2 have no partner (B is zero and weighs nothing).
//   y passes  A and B are the same kx in neighbouring planes: the same zero columns.
// A block is TXP pairs of neighbouring kx (32- or 64-byte row segments at 512; the rows of
// the intermediates start on 32-byte boundaries).  The transform is the Stockham schedule of
// ur_fast.cu with 8 values per thread; an exchange moves a pair's value as one 16-byte word
// at i + i/8 with a column pitch that spreads the eight lanes of a shared-memory phase over
// the banks.  Twiddles are stored twice over (wx, wx, wy, wy), stage by stage, so that a
// 16-byte load is a packed operand and neighbouring lanes read neighbouring words.
//
// Measured against one column per group, us: z + bins of a 256^3 forward 62 -> 49; 512^3 step: y 106 -> 90, z + bins 258 -> 240, adjoint z 322 -> 276, adjoint y 220 -> 203.  The
// shared-memory and L1 data pipe is now the busiest unit (65-68 %).  At 1024 pairs are slower than
// single columns with 16 and 32 values per thread (y 723 -> 1362, z + bins 2154 -> 2890, of a full grid 2305 ->
// 4114, adjoint z 2469 -> 3382, adjoint y 1730 -> 1986 us: row segments of 16 and 32 bytes, and rows ky and -ky
// of a plane lie in different 2 MB pages), so from 1024 on the columns are transformed one by one
// (ur_fast.cu).
#include <vector>

#include "ur_fast.cuh"

struct C2 {  // one complex value of columns A and B
  ur_f2 x, y;
};
__device__ __forceinline__ C2 c2_add(C2 a, C2 b) { return {f2_add(a.x, b.x), f2_add(a.y, b.y)}; }
__device__ __forceinline__ C2 c2_sub(C2 a, C2 b) { return {f2_sub(a.x, b.x), f2_sub(a.y, b.y)}; }
// a - i b (forward) / a + i b (inverse), and the other sign
template <bool INV>
__device__ __forceinline__ C2 c2_add_ni(C2 a, C2 b) {
  return INV ? C2{f2_sub(a.x, b.y), f2_add(a.y, b.x)} : C2{f2_add(a.x, b.y), f2_sub(a.y, b.x)};
}
template <bool INV>
__device__ __forceinline__ C2 c2_sub_ni(C2 a, C2 b) {
  return c2_add_ni<!INV>(a, b);
}
// a * w, w = (wx, wx, wy, wy) the forward twiddle (inverse: its conjugate); both components end in a
// fused multiply-add, so that one product of each is not rounded
template <bool INV>
__device__ __forceinline__ C2 c2_twmul(C2 a, ulonglong2 w) {
  const ur_f2 p = f2_mul(a.x, w.x), q = f2_mul(a.y, w.x), n = f2_neg(w.y);
  return INV ? C2{f2_fma(a.y, w.y, p), f2_fma(a.x, n, q)} : C2{f2_fma(a.y, n, p), f2_fma(a.x, w.y, q)};
}
template <bool INV>
__device__ __forceinline__ void c2_dft4(C2& a0, C2& a1, C2& a2, C2& a3) {
  const C2 t0 = c2_add(a0, a2), t1 = c2_sub(a0, a2), t2 = c2_add(a1, a3), t3 = c2_sub(a1, a3);
  a0 = c2_add(t0, t2);
  a2 = c2_sub(t0, t2);
  a1 = c2_add_ni<INV>(t1, t3);
  a3 = c2_sub_ni<INV>(t1, t3);
}

template <int R, bool INV>
__device__ __forceinline__ void c2_dft(C2* a) {
  if constexpr (R == 2) {
    const C2 t = a[0];
    a[0] = c2_add(t, a[1]);
    a[1] = c2_sub(t, a[1]);
  } else if constexpr (R == 4) {
    c2_dft4<INV>(a[0], a[1], a[2], a[3]);
  } else {
    static_assert(R == 8, "radix 2, 4 or 8");
    C2 e0 = a[0], e1 = a[2], e2 = a[4], e3 = a[6];
    C2 o0 = a[1], o1 = a[3], o2 = a[5], o3 = a[7];
    c2_dft4<INV>(e0, e1, e2, e3);
    c2_dft4<INV>(o0, o1, o2, o3);
    const float r = 0.70710678118654752f;
    const ur_f2 pr = f2_pack(r, r), nr = f2_pack(-r, -r);
    a[0] = c2_add(e0, o0);
    a[4] = c2_sub(e0, o0);
    a[2] = c2_add_ni<INV>(e2, o2);
    a[6] = c2_sub_ni<INV>(e2, o2);
    // W8 o1 = r (s1, d1) and W8^3 o3 = r (d3, -s3) (forward), folded into the last additions
    const ur_f2 s1 = f2_add(o1.x, o1.y), s3 = f2_add(o3.x, o3.y);
    const ur_f2 d1 = f2_sub(o1.y, o1.x), d3 = f2_sub(o3.y, o3.x);
    if constexpr (!INV) {
      a[1] = {f2_fma(s1, pr, e1.x), f2_fma(d1, pr, e1.y)};
      a[5] = {f2_fma(s1, nr, e1.x), f2_fma(d1, nr, e1.y)};
      a[3] = {f2_fma(d3, pr, e3.x), f2_fma(s3, nr, e3.y)};
      a[7] = {f2_fma(d3, nr, e3.x), f2_fma(s3, pr, e3.y)};
    } else {
      a[1] = {f2_fma(d1, nr, e1.x), f2_fma(s1, pr, e1.y)};
      a[5] = {f2_fma(d1, pr, e1.x), f2_fma(s1, nr, e1.y)};
      a[3] = {f2_fma(s3, nr, e3.x), f2_fma(d3, nr, e3.y)};
      a[7] = {f2_fma(s3, pr, e3.x), f2_fma(d3, pr, e3.y)};
    }
  }
}

// ---------------------------------------------------------------------------
// Configuration: 8 values per column and thread (64 registers), 1024 threads per SM.  At 512 the
// passes that write the whole grid take blocks of 512 threads, eight pairs (64-byte row
// segments): adjoint z 326 -> 276 us, adjoint y 215 -> 203; the forward passes, which write less
// or nothing, are faster with blocks of 256 (y 104 -> 90 us, z + bins 242 -> 240).
// ---------------------------------------------------------------------------
template <int N, int MODE>
struct PairCfg {
  static constexpr int E = 8, LE = 3;
  static constexpr int T = N / E;
  static constexpr int THREADS = N == 512 && (MODE == P2_Y_INV || MODE == P2_Y_INV_ROWS || MODE == P2_Z_ADJ) ? 512 : 256;
  static constexpr int TXP = THREADS / T;
  static constexpr int MINB = 1024 / THREADS;
  // column pitch in 16-byte words: the eight lanes of a phase are TXP columns of 8 / TXP positions
  static constexpr int PITCH = N + N / E + (TXP == 4 ? 2 : 1);
  static constexpr int CW = (N / 2 + 4) / 4 * 4;  // columns per row of the flattened index (H rounded up to 4)
  static_assert(TXP == 4 ? PITCH % 8 == 2 : PITCH % 2 == 1, "conflict-free exchange");
};

__device__ __forceinline__ int pair_pad(int i) { return i + (i >> 3); }

constexpr int pair_pow(int e, int s) { return s == 0 ? 1 : e * pair_pow(e, s - 1); }
// radix of stage S of an L = 2^LOG point transform with E = 2^LE values per thread
constexpr int pair_radix(int log, int le, int S) { return (S + 1) * le <= log ? 1 << le : 1 << (log - S * le); }
// offset (16-byte words) of stage S >= 1 in the twiddle table: [r - 1][k], k < E^S
constexpr int pair_off(int log, int le, int S) {
  return S <= 1 ? 0 : pair_off(log, le, S - 1) + (pair_radix(log, le, S - 1) - 1) * pair_pow(1 << le, S - 1);
}
constexpr int pair_log(int n) { return n <= 1 ? 0 : 1 + pair_log(n / 2); }

template <int N, bool INV, int S>
__device__ __forceinline__ void pair_stages(C2 (&v)[8], int j, ulonglong2* line,
                                            const ulonglong2* __restrict__ tw) {
  constexpr int E = 8, LE = 3, T = N / E, LOG = pair_log(N);
  constexpr int NST = (LOG + LE - 1) / LE;
  if constexpr (S < NST) {
    constexpr int R = pair_radix(LOG, LE, S), NS = pair_pow(E, S), NB = E / R, OFF = pair_off(LOG, LE, S);
#pragma unroll
    for (int i = 0; i < NB; ++i) {
      const int k = (j + i * T) & (NS - 1);
      C2 a[R];
#pragma unroll
      for (int r = 0; r < R; ++r) a[r] = v[i + NB * r];
      if constexpr (S > 0) {
#pragma unroll
        for (int r = 1; r < R; ++r) a[r] = c2_twmul<INV>(a[r], __ldg(tw + OFF + (r - 1) * NS + k));
      }
      c2_dft<R, INV>(a);
#pragma unroll
      for (int r = 0; r < R; ++r) v[i + NB * r] = a[r];
    }
    if constexpr (S + 1 < NST) {
#pragma unroll
      for (int i = 0; i < NB; ++i) {
        const int b = j + i * T, k = b & (NS - 1);
#pragma unroll
        for (int r = 0; r < R; ++r)
          line[pair_pad((b - k) * R + k + r * NS)] = make_ulonglong2(v[i + NB * r].x, v[i + NB * r].y);
      }
      __syncthreads();
#pragma unroll
      for (int q = 0; q < E; ++q) {
        const ulonglong2 t = line[pair_pad(j + q * T)];
        v[q] = {t.x, t.y};
      }
      __syncthreads();
    }
    pair_stages<N, INV, S + 1>(v, j, line, tw);
  }
}

// Element q of a column: base + (unsigned)q * step bytes (step < 2^32: at most 64 planes of 1 MB)
__device__ __forceinline__ const float2* at_step(const float2* p, unsigned q, unsigned step) {
  return reinterpret_cast<const float2*>(reinterpret_cast<const char*>(p) + (unsigned long long)q * step);
}
__device__ __forceinline__ float2* at_step(float2* p, unsigned q, unsigned step) {
  return reinterpret_cast<float2*>(reinterpret_cast<char*>(p) + (unsigned long long)q * step);
}
__device__ __forceinline__ C2 c2_pack(float2 a, float2 b) { return {f2_pack(a.x, b.x), f2_pack(a.y, b.y)}; }
__device__ __forceinline__ void c2_store(float2* pa, float2* pb, bool hasb, C2 v) {
  const float2 x = f2_get(v.x), y = f2_get(v.y);
  *pa = make_float2(x.x, y.x);
  if (hasb) *pb = make_float2(x.y, y.y);
}

template <int N, int MODE>
__global__ void __launch_bounds__(PairCfg<N, MODE>::THREADS, (PairCfg<N, MODE>::MINB)) k_pair_cols(const __grid_constant__ ColArgs a) {
  using Cfg = PairCfg<N, MODE>;
  constexpr int E = Cfg::E, T = Cfg::T, TXP = Cfg::TXP, PITCH = Cfg::PITCH, CW = Cfg::CW, M = N / 2, H = M + 1;
  constexpr bool ZP = MODE == P2_Z_BIN || MODE == P2_Z_ADJ, YINV = MODE == P2_Y_INV || MODE == P2_Y_INV_ROWS;
  extern __shared__ __align__(16) unsigned char smraw[];
  __shared__ int s_blo, s_bhi;
  ulonglong2* buf = reinterpret_cast<ulonglong2*>(smraw);
  constexpr size_t BUF_BYTES = (size_t)TXP * PITCH * 16;
  const int nb = a.nbins;
  int32_t* thr = reinterpret_cast<int32_t*>(smraw + BUF_BYTES);
  float* hs = reinterpret_cast<float*>(smraw + BUF_BYTES + ur_align_up_dev((size_t)(nb + 1) * 4, 16));
  float* hs2 = hs + nb;
  int16_t* crs = reinterpret_cast<int16_t*>(reinterpret_cast<unsigned char*>(hs) + ur_align_up_dev((size_t)nb * 8, 16));
  float* Kb = reinterpret_cast<float*>(crs);  // forward binning: the block's cache of the bin shifts
  const int c = threadIdx.x % TXP, j = threadIdx.x / TXP;
  const int blk = MODE == P2_Z_BIN ? ur_late_first_row(blockIdx.x, gridDim.x, (CW + TXP - 1) / TXP) : blockIdx.x;
  const int cp = blk * TXP + c;
  // row of the flattened index: |ky| in the z passes, plane pair in the y passes
  const int row = cp / CW, kx = cp - row * CW;
  const int ia = ZP ? row : 2 * row;
  const int ib = ZP ? N - row : 2 * row + 1;
  const bool valid = kx < H && (ZP ? row <= M : ia < a.nouter);
  const bool hasb = valid && (ZP ? (row != 0 && row != M) : ib < a.nouter);
  const int c2 = kx * kx + row * row;  // z passes: kx^2 + ky^2
  const bool binning = ZP && nb > 0;
  int lo_bin = 0, hi_bin = 0;
  if (MODE == P2_Z_BIN && binning) {
    if (threadIdx.x == 0) {
      s_blo = 0x7fffffff;
      s_bhi = -1;
    }
    // bins of k^2 = c2 and c2 + M^2: the range that the column reaches
    if (j == 0 && valid) {
      const int t0 = __ldg(a.thr), tn = __ldg(a.thr + nb), s_hi = c2 + M * M;
      lo_bin = c2 < t0 ? 0 : c2 >= tn ? nb - 1 : __ldg(a.lut + c2);
      hi_bin = s_hi < t0 ? 0 : s_hi >= tn ? nb - 1 : __ldg(a.lut + s_hi);
    }
  }
  // z passes: a block whose columns all lie at or beyond the closing threshold reaches no bin
  const bool skip_mode = (MODE == P2_Z_BIN && binning && !a.fout) || (MODE == P2_Z_ADJ && binning);
  float2* const da = a.dst + (long long)ia * a.Ad + kx;
  float2* const db = a.dst + (long long)(hasb ? ib : ia) * a.Ad + kx;
  const unsigned dstep = (unsigned)(T * a.Sd * 8);
  if (skip_mode) {
    const bool beyond = __syncthreads_and(!valid || c2 >= __ldg(a.thr + nb));
    // uniform over the block (adjoint: the output columns are zero, and the y pass takes them as zeros
    // without loading them: k2_zero)
    if (beyond) return;
  }
  if (MODE == P2_Z_ADJ && binning) {
    for (int i = threadIdx.x; i <= nb; i += Cfg::THREADS) thr[i] = __ldg(a.thr + i);
    for (int i = threadIdx.x; i < UR_COARSE_ENTRIES / 8; i += Cfg::THREADS)
      reinterpret_cast<uint4*>(crs)[i] = __ldg(reinterpret_cast<const uint4*>(a.crs) + i);
    for (int i = threadIdx.x; i < nb; i += Cfg::THREADS) hs[i] = __ldg(a.sigma + i);
  }
  C2 v[E];
  {
    // planes zoff .. zoff + nload - 1 are present (z passes), or every element (nload = N)
    const long long off = (long long)(j - a.zoff) * a.S + kx;
    const float2* pa = a.src + (long long)ia * a.A + off;
    const float2* pb = a.src + (long long)(hasb ? ib : ia) * a.A + off;
    const unsigned step = (unsigned)(T * a.S * 8);
    const float2 zero = make_float2(0.f, 0.f);
#pragma unroll
    for (int q = 0; q < E; ++q) {
      const int li = j + q * T;
      bool la = valid, lb = hasb;
      if (ZP) {
        const bool in = (unsigned)(li - a.zoff) < (unsigned)a.nload;
        la = la && in;
        lb = lb && in;
      } else if (MODE == P2_Y_FWD) {
        if (a.row_skip) {  // rows outside the particle were not written
          la = la && !row_outside(a.sh, li, a.gen_z0 + ia);
          lb = lb && !row_outside(a.sh, li, a.gen_z0 + ib);
        }
      } else {  // columns at or beyond k2_zero were not written
        const int ky = li < M ? li : li - N;
        const bool in = kx * kx + ky * ky < a.k2_zero;
        la = la && in;
        lb = lb && in;
      }
      v[q] = c2_pack(la ? __ldg(at_step(pa, q, step)) : zero, lb ? __ldg(at_step(pb, q, step)) : zero);
    }
  }
  // forward z pass: the thresholds are staged after the column loads are issued
  if (MODE == P2_Z_BIN && binning) {
    for (int i = threadIdx.x; i <= nb; i += Cfg::THREADS) thr[i] = __ldg(a.thr + i);
  }
  ulonglong2* line = buf + c * PITCH;
  const ulonglong2* tw = reinterpret_cast<const ulonglong2*>(a.stw);
  if (binning && (MODE == P2_Z_ADJ || !skip_mode)) __syncthreads();  // tables (and the range reset) visible
  if (MODE == P2_Z_BIN && binning && j == 0 && valid) {
    atomicMin(&s_blo, lo_bin);
    atomicMax(&s_bhi, hi_bin);
  }
  if (!ZP) {
    pair_stages<N, YINV, 0>(v, j, line, tw);
    if (MODE == P2_Y_INV_ROWS) {  // rows outside the particle are not needed
#pragma unroll
      for (int q = 0; q < E; ++q) {
        const float2 x = f2_get(v[q].x), y = f2_get(v[q].y);
        const int li = j + q * T;
        if (valid && !row_outside(a.sh, li, a.gen_z0 + ia)) *at_step(da + j * a.Sd, q, dstep) = make_float2(x.x, y.x);
        if (hasb && !row_outside(a.sh, li, a.gen_z0 + ib)) *at_step(db + j * a.Sd, q, dstep) = make_float2(x.y, y.y);
      }
    } else if (valid) {
#pragma unroll
      for (int q = 0; q < E; ++q)
        c2_store(at_step(da + j * a.Sd, q, dstep), at_step(db + j * a.Sd, q, dstep), hasb, v[q]);
    }
  } else if (MODE == P2_Z_BIN) {
    pair_stages<N, false, 0>(v, j, line, tw);
    if (a.fout && valid) {
#pragma unroll
      for (int q = 0; q < E; ++q) {
        const float2 x = f2_get(v[q].x), y = f2_get(v[q].y);
        float2* f = a.fout + (long long)(j + q * T) * N * H + kx;
        f[(long long)ia * H] = cscale(make_float2(x.x, y.x), a.fscale);
        if (hasb) f[(long long)ib * H] = cscale(make_float2(x.y, y.y), a.fscale);
      }
    }
    if (binning) {
      // Task = (pair, chunk of CH consecutive |kz| = m); the last chunk also takes m = M.  The bin of
      // the chunk's first m comes from the k^2 table; after that it only moves forward, when
      // s = c2 + m^2 reaches the next threshold.  The values at kz = +-m of both columns are one run
      // of shifted sums (ur_bin_shift).
      constexpr int CH = M / T;
      static_assert(CH * T == M, "whole chunks");
      const bool has = valid;
      const int m0 = j * CH;
      const float w = (kx == 0 || kx == M) ? 1.f : 2.f;
      float csc = a.iscale;  // I scale of the pair (times its voxel-sinc factor)
      int b = -1;
      if (has) {
        if (a.vs) csc = a.iscale * (__ldg(a.vs + kx) * __ldg(a.vs + row));
        const int s0 = c2 + m0 * m0;
        b = s0 < thr[0] ? -1 : s0 >= thr[nb] ? nb : __ldg(a.lut + s0);
      }
      for (int i = s_blo + (int)threadIdx.x; i <= s_bhi; i += Cfg::THREADS) {
        hs[i] = 0.f;
        hs2[i] = 0.f;
        // the shifts already published for the block's bins, fetched together up front; unset ones
        // are NaN and published on first use
        const unsigned long long g = __ldcg(a.gK + i);
        Kb[i] = g ? __uint_as_float((unsigned)(g & 0xffffffffull)) : __int_as_float(0x7fc00000);
      }
#pragma unroll
      for (int q = 0; q < E; ++q) line[pair_pad(j + q * T)] = make_ulonglong2(v[q].x, v[q].y);
      __syncthreads();
      if (has) {
        int tnext = b < nb ? thr[b + 1] : 0x7fffffff;
        int s = c2 + m0 * m0;
        ur_f2 sI = 0ull, sI2 = 0ull, nK = 0ull;
        bool fresh = true;
        auto flush = [&]() {
          const float2 t = f2_get(sI), t2 = f2_get(sI2);
          // without a partner lane B holds (0 - K)^2, which may have overflowed: left out, not weighed with 0
          atomicAdd(hs + b, w * (hasb ? t.x + t.y : t.x));
          atomicAdd(hs2 + b, w * (hasb ? t2.x + t2.y : t2.x));
          sI = sI2 = 0ull;
          fresh = true;
        };
        auto visit = [&](int mm, bool twice) {
          if (s >= tnext) {
            if (!fresh) flush();
            do {
              ++b;
              tnext = b < nb ? thr[b + 1] : 0x7fffffff;
            } while (s >= tnext);
          }
          if (b >= 0 && b < nb) {
            const float sc = a.vs ? csc * __ldg(a.vs + mm) : csc;
            const ur_f2 sc2 = f2_pack(sc, sc);
            const ulonglong2 f1 = line[pair_pad(mm)];
            const ur_f2 p1 = f2_fma(f1.y, f1.y, f2_mul(f1.x, f1.x));
            if (fresh) {
              const float K = ur_bin_shift(Kb, a.gK, b, f2_get(p1).x * sc);
              nK = f2_pack(-K, -K);
              fresh = false;
            }
            const ur_f2 d1 = f2_fma(p1, sc2, nK);
            sI = f2_add(sI, d1);
            sI2 = f2_fma(d1, d1, sI2);
            if (twice) {
              const ulonglong2 f2 = line[pair_pad(N - mm)];
              const ur_f2 d2 = f2_fma(f2_fma(f2.y, f2.y, f2_mul(f2.x, f2.x)), sc2, nK);
              sI = f2_add(sI, d2);
              sI2 = f2_fma(d2, d2, sI2);
            }
          }
          s += 2 * mm + 1;
        };
#pragma unroll
        for (int u = 0; u < CH; ++u) visit(m0 + u, m0 + u != 0);
        if (j == T - 1) visit(M, false);
        if (!fresh && b >= 0 && b < nb) flush();
      }
      __syncthreads();
      for (int i = s_blo + (int)threadIdx.x; i <= s_bhi; i += Cfg::THREADS) {
        if (hs[i] != 0.f) atomicAdd(a.gsum + i, (double)hs[i]);
        if (hs2[i] != 0.f) atomicAdd(a.gsum2 + i, (double)hs2[i]);
      }
    }
  } else {  // P2_Z_ADJ
    if (!a.skip_fwd) pair_stages<N, false, 0>(v, j, line, tw);
    // scale of element kz: sigma of the bin of k^2 = c2 + m^2, m = |signed kz|
#pragma unroll
    for (int q = 0; q < E; ++q) {
      const int kz = j + q * T;
      const int m = kz <= M ? kz : N - kz;
      const int b = valid ? bin_rank(crs, a.crs_shift, thr, nb, c2 + m * m) : nb;
      const float sg = (b >= 0 && b < nb) ? hs[b] : 0.f;
      const ur_f2 s2 = f2_pack(sg, sg);
      v[q] = {f2_mul(v[q].x, s2), f2_mul(v[q].y, s2)};
    }
    pair_stages<N, true, 0>(v, j, line, tw);
    if (valid) {
      if (a.out_cnt > 0) {  // a slab of output planes
#pragma unroll
        for (int q = 0; q < E; ++q) {
          const int zo = j + q * T - a.out_lo;
          if (zo >= 0 && zo < a.out_cnt) c2_store(da + zo * a.Sd, db + zo * a.Sd, hasb, v[q]);
        }
      } else {
#pragma unroll
        for (int q = 0; q < E; ++q)
          c2_store(at_step(da + j * a.Sd, q, dstep), at_step(db + j * a.Sd, q, dstep), hasb, v[q]);
      }
    }
  }
}

// ---------------------------------------------------------------------------
// Host
// ---------------------------------------------------------------------------
bool ur_pair_supported(int n) { return n == 64 || n == 128 || n == 256 || n == 512; }

// Twiddle table of the N-point column transform: the entries w of ur_stage_twiddles for 8 values per
// thread as (wx, wx, wy, wy).  Returns the number of 16-byte words (out may be NULL to count).
size_t ur_pair_twiddles(int n, float4* out) {
  const size_t cnt = ur_stage_twiddles(pair_log(n), 8, nullptr);
  if (out) {
    std::vector<float2> w(cnt);
    ur_stage_twiddles(pair_log(n), 8, w.data());
    for (size_t i = 0; i < cnt; ++i) out[i] = make_float4(w[i].x, w[i].x, w[i].y, w[i].y);
  }
  return cnt;
}

template <int N, int MODE>
static ur_status launch_pair(const ColArgs& args, cudaStream_t s) {
  using Cfg = PairCfg<N, MODE>;
  ColArgs a = args;
  a.nouter = (int)(args.ncols / (N / 2 + 1));  // planes (y passes)
  const bool zp = MODE == P2_Z_BIN || MODE == P2_Z_ADJ;
  const long long rows = zp ? N / 2 + 1 : ((long long)a.nouter + 1) / 2;
  const long long blocks = (rows * Cfg::CW + Cfg::TXP - 1) / Cfg::TXP;
  if (blocks <= 0) return UR_OK;
  const size_t nb = (size_t)a.nbins;
  const size_t smem = (size_t)Cfg::TXP * Cfg::PITCH * 16 + ur_align_up((nb + 1) * 4, 16) + ur_align_up(nb * 8, 16) +
                      (MODE == P2_Z_ADJ ? (size_t)UR_COARSE_ENTRIES * 2 : 0) + (MODE == P2_Z_BIN ? nb * 4 : 0);
  if (smem > UR_DYN_SMEM_FREE)
    UR_CUDA_CHECK(cudaFuncSetAttribute(k_pair_cols<N, MODE>, cudaFuncAttributeMaxDynamicSharedMemorySize, (int)smem));
  k_pair_cols<N, MODE><<<(unsigned)blocks, Cfg::THREADS, smem, s>>>(a);
  UR_LAUNCH_CHECK("k_pair_cols");
  return UR_OK;
}

template <int N>
static ur_status launch_pair_n(int mode, const ColArgs& a, cudaStream_t s) {
  switch (mode) {
    case P2_Y_FWD: return launch_pair<N, P2_Y_FWD>(a, s);
    case P2_Y_INV: return a.row_skip ? launch_pair<N, P2_Y_INV_ROWS>(a, s) : launch_pair<N, P2_Y_INV>(a, s);
    case P2_Z_BIN: return launch_pair<N, P2_Z_BIN>(a, s);
    default: return launch_pair<N, P2_Z_ADJ>(a, s);
  }
}

ur_status ur_pair_cols(int n, int mode, const ColArgs& a, cudaStream_t s) {
  switch (n) {
    case 64: return launch_pair_n<64>(mode, a, s);
    case 128: return launch_pair_n<128>(mode, a, s);
    case 256: return launch_pair_n<256>(mode, a, s);
    case 512: return launch_pair_n<512>(mode, a, s);
  }
  ur_set_error("ur_pair_cols: unsupported size %d", n);
  return UR_ERR_UNSUPPORTED;
}
