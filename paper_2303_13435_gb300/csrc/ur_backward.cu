// Adjoint of the forward map (not in the paper; the chain rule through
// Sec. 2.3-2.5).  For g_j = dL/d(mean I_j) and G_k = g_j / n_j on bin j:
//
//   dL/drho(x) = (2/N^3) Re sum_k G_k F_k e^{+2 pi i k.x/N}
//              = (1/N^3) Re sum_k sigma_j F~_k e^{+2 pi i k.x/N},  sigma_j = 2 g_j / (n_j N^3)
//
// with F~ the unnormalised transform.  The inverse transform runs in the
// reverse order of the forward passes:
//   B1 k_cols<COL_ZADJ>  per (ky, kx) column: F~ along z recomputed from the
//                        forward intermediate (or F read), times sigma(bin),
//                        inverse transform along z, all N planes written
//   B2 k_cols<COL_Y,inv> inverse transform along y of every plane, in place
//   B3 k_rows_grad       inverse real transform along x of every row, then
//                        dL/dm = dL/drho * u(x mod U) written and
//                        dL/du(c) = sum over tiles of dL/drho * m(x) reduced;
//                        a block takes a batch of the grid rows that wrap
//                        onto one cell row (cz, cy), so its partial sums of
//                        dL/du land on one cell row (one global add each).
#include <math.h>
#include <string.h>

#include "ur_fast.cuh"

// sigma_j = 2 g_j / (n_j N^3) (scale of F~), or 2 g_j / n_j when F (= F~/N^3) is read
__global__ void k_sigma(const double* __restrict__ g, const double* __restrict__ fwd_bins, int nb, double n3, int f_given,
                        float* __restrict__ sigma) {
  const int j = blockIdx.x * blockDim.x + threadIdx.x;
  if (j >= nb) return;
  const double n = fwd_bins[UR_BIN_COUNT * nb + j];
  double v = 0.0;
  if (n > 0) v = 2.0 * g[j] / n / (f_given ? 1.0 : n3);
  sigma[j] = (float)v;
}

// B3.  A block takes up to RB rows (z, y) that wrap onto G neighbouring cell rows of one cell plane:
// (z + oz) mod U = cz, (y + oy) mod U in [cy0, cy0 + G), so that small grids and small particles fill
// its transforms too.  Rows that are not needed (outside the particle, when dL/dm is not wanted) do
// not enter.  Each row: Y[z][y][0..M] (Hermitian half along x) -> Z[k] = E[k] + i O[k],
//   E[k] = X[k] + conj X[M-k],  O[k] = (X[k] - conj X[M-k]) conj(W_N^k),
// then z = IFFT_{M}(Z) gives (g(2m), g(2m+1)) = (Re z[m], Im z[m]).
// dL/du: a thread owns a cell voxel (or a share of its rows), sums its voxels of the block's rows in
// registers and adds the sum to global memory once: a shared-memory float32 addition per voxel is a
// compare-and-swap loop.  64 particles of 96^3-384^3, dL/du only: 8674 -> 678 us (64-row tiles of
// which 1 to 36 rows were used, every row of the box); 378^3 with dL/dm: 311 -> 289 us.
struct NoStore {
  struct It {
    __device__ __forceinline__ void put(float2) {}
  };
  __device__ __forceinline__ It first(int, int, int) const { return {}; }
};

struct GradRow {
  RowMask rm;
  int z, y, g;  // g: cell row of the block
};

__device__ __forceinline__ int first_in(int lo, int c, int o, int U) {  // first i >= lo with (i + o) mod U = c
  int d = (c - o - lo) % U;
  if (d < 0) d += U;
  return lo + d;
}

__device__ __forceinline__ void rows_grad_body(const GenGradArgs& g, int bx, int by) {
  const int N = g.N, RB = g.RB, nst = g.nst, U = g.U, G = g.G, zlo = g.zlo, yp = g.yp, ox = g.ox;
  const float* __restrict__ weights = g.weights;
  float* __restrict__ dl_dmask = g.dl_dmask;
  float* __restrict__ dl_dcell = g.dl_dcell;
  const StageInfo* __restrict__ sched = g.sched;
  const float2* __restrict__ tw = g.tw;
  const ShapeArgs& sh = g.sh;
  const float inv_n3 = g.inv_n3;
  extern __shared__ __align__(16) unsigned char smraw[];
  __shared__ int s_nrow;
  const int M = N >> 1, H = M + 1;
  float2* buf = reinterpret_cast<float2*>(smraw);
  GradRow* rows = reinterpret_cast<GradRow*>(smraw + ur_align_up_dev((size_t)RB * H * sizeof(float2), 16));
  int* gbeg = reinterpret_cast<int*>(rows + RB);  // first row of each of the block's cell rows
  const int ncg = (U + G - 1) / G;
  const int cz = by / ncg, cy0 = (by - cz * ncg) * G;
  const int zf = first_in(g.zlo, cz, g.oz, U);
  if (zf >= g.zhi) return;  // uniform over the block
  // the block's rows, in order of cell row; listed by the first warp
  if (threadIdx.x < 32) {
    const int per = g.nza * g.nyb;
    int n = 0;
    for (int t0 = 0; t0 < RB; t0 += 32) {
      const int q = bx * RB + t0 + (int)threadIdx.x;
      const int gr = q / per, ab = q - gr * per, a = ab / g.nyb, b = ab - a * g.nyb;
      const int z = zf + U * a, cy = cy0 + gr;
      bool use = t0 + (int)threadIdx.x < RB && gr < G && cy < U && z < g.zhi;
      int y = 0;
      if (use) {
        y = first_in(g.ylo, cy, g.oy, U) + U * b;
        use = y < g.yhi && !(g.row_skip && row_outside(sh, y, z));
      }
      const unsigned who = __ballot_sync(0xffffffffu, use);
      if (use) {
        GradRow& r = rows[n + __popc(who & ((1u << threadIdx.x) - 1u))];
        r.rm.init(sh, y, z);
        r.z = z;
        r.y = y;
        r.g = gr;
      }
      n += __popc(who);
    }
    __syncwarp();
    for (int i = threadIdx.x; i <= G; i += 32) {  // rows of cell row i: [gbeg[i], gbeg[i + 1])
      int lo = 0, hi = n;
      while (lo < hi) {
        const int mid = (lo + hi) >> 1;
        if (rows[mid].g < i) lo = mid + 1;
        else hi = mid;
      }
      gbeg[i] = lo;
    }
    if (threadIdx.x == 0) s_nrow = n;
  }
  __syncthreads();
  const int nrow = s_nrow;
  if (nrow == 0) return;
  const float2* __restrict__ Y = g.Y;
  const FastDiv dM((uint32_t)M), dH((uint32_t)H);
  if (nst >= 2) {
    // the first stage packs its inputs straight from the Hermitian half rows (no staging
    // round trip): Z[i] = (X[i] + conj X[M-i]) + i (X[i] - conj X[M-i]) conj(W_N^i), X[M] for i = 0
    auto packed = [&](int t, int i) -> float2 {
      const float2* row = Y + ((long long)(rows[t].z - zlo) * N + rows[t].y) * yp;
      const float2 xa = __ldg(row + i), xb = __ldg(row + (M - i));
      const float2 w = __ldg(tw + i);
      const float2 e = cadd(xa, cconj(xb));
      const float2 d = csub(xa, cconj(xb));
      const float2 o = make_float2(d.x * w.x + d.y * w.y, d.y * w.x - d.x * w.y);  // * conj(W^i)
      return make_float2(e.x - o.y, e.y + o.x);
    };
    fft_lines_io<true, UR_EMAX, true, false, false>(buf, H, nrow, sched, nst, tw, ld_fn(packed), NoStore());
  } else {
    for (int f = threadIdx.x; f < nrow * H; f += blockDim.x) {
      const int t = (int)dH.div((uint32_t)f);
      buf[f] = __ldg(Y + ((long long)(rows[t].z - zlo) * N + rows[t].y) * yp + (f - t * H));
    }
    __syncthreads();
    // Hermitian half -> packed complex sequence, in place by (k, M-k) pairs
    const int half = M / 2 + 1;
    const FastDiv dhalf((uint32_t)half);
    for (int f = threadIdx.x; f < nrow * half; f += blockDim.x) {
      const int t = (int)dhalf.div((uint32_t)f);
      const int k = f - t * half;
      float2* X = buf + t * H;
      const float2 xa = X[k], xb = X[M - k];
      const float2 wa = __ldg(tw + k);
      // Z[k]
      const float2 ea = cadd(xa, cconj(xb));
      const float2 da = csub(xa, cconj(xb));
      const float2 oa = make_float2(da.x * wa.x + da.y * wa.y, da.y * wa.x - da.x * wa.y);  // * conj(W^k)
      const float2 za = make_float2(ea.x - oa.y, ea.y + oa.x);
      if (k != 0 && 2 * k != M) {
        const float2 wb = __ldg(tw + (M - k));
        const float2 eb = cadd(xb, cconj(xa));
        const float2 db = csub(xb, cconj(xa));
        const float2 ob = make_float2(db.x * wb.x + db.y * wb.y, db.y * wb.x - db.x * wb.y);
        X[M - k] = make_float2(eb.x - ob.y, eb.y + ob.x);
      }
      X[k] = za;
    }
    __syncthreads();
    fft_lines<true, UR_EMAX>(buf, H, nrow, sched, nst, tw);
  }
  // dL/dm = dL/drho * u.  Voxel weights are multiplied in here, where neighbouring threads read neighbouring
  // ones, and not by the threads that sum a cell voxel's repeats
  if (dl_dmask || weights) {
    const FastDiv dU((uint32_t)U);
    for (int f = threadIdx.x; f < nrow * M; f += blockDim.x) {
      const int t = (int)dM.div((uint32_t)f);
      const int m = f - t * M;
      const float2 zv = buf[t * H + m];
      const long long vox = ((long long)rows[t].z * N + rows[t].y) * N + 2 * m;
      if (dl_dmask) {
        const int c0 = (int)dU.mod((uint32_t)(2 * m + ox)), c1 = c0 + 1 == U ? 0 : c0 + 1;
        const float* crow = g.cell + ((long long)cz * U + cy0 + rows[t].g) * U;
        *reinterpret_cast<float2*>(dl_dmask + vox) =
            make_float2(zv.x * inv_n3 * __ldg(crow + c0), zv.y * inv_n3 * __ldg(crow + c1));
      }
      if (weights) {
        const float2 w = __ldg(reinterpret_cast<const float2*>(weights + vox));
        buf[t * H + m] = make_float2(w.x != 0.f ? zv.x * inv_n3 * w.x : 0.f, w.y != 0.f ? zv.y * inv_n3 * w.y : 0.f);
      }
    }
    if (weights) __syncthreads();
  }
  // dL/du = sum of dL/drho * m over the repeats: task (cell row, share of its rows, cell column)
  const float* bufr = reinterpret_cast<const float*>(buf);
  const int share = G * U < (int)blockDim.x ? (int)blockDim.x / (G * U) : 1;
  const int ntask = G * share * U;
  for (int task = threadIdx.x; task < ntask; task += blockDim.x) {
    const int gs = task / U, c = task - gs * U;
    const int gr = gs / share, part = gs - gr * share;
    int x0 = (c - ox) % U;
    if (x0 < 0) x0 += U;
    float sum = 0.f;
    for (int t = gbeg[gr] + part; t < gbeg[gr + 1]; t += share) {
      const RowMask& rm = rows[t].rm;
      const float* line = bufr + (size_t)t * 2 * H;
      if (weights) {
        for (int x = x0; x < N; x += U) sum += line[x];
      } else {
        for (int x = x0; x < N; x += U) {
          const float m = rm.at(x);
          if (m != 0.f) sum += line[x] * inv_n3 * m;
        }
      }
    }
    if (sum != 0.f) atomicAdd(dl_dcell + ((long long)cz * U + cy0 + gr) * U + c, sum);
  }
}

__global__ void __launch_bounds__(256, 4) k_rows_grad(GenGradArgs g) { rows_grad_body(g, blockIdx.x, blockIdx.y); }

// Log-I(Q) MSE and its gradient: one thread per bin over blocks of 64 threads
// (the float64 logarithms are the cost, so they are spread over many SMs).
// Every block first counts the valid bins of the whole curve (V, needed by the
// gradient of every bin; a cheap scan), then writes its bins' gradients and
// adds its share of L = sum d^2 / V to *loss (zeroed beforehand).  float64
// throughout.
#define UR_LOSS_THREADS 64
#define UR_LOSS_MAX_BINS 8192
__global__ void __launch_bounds__(UR_LOSS_THREADS) k_log_mse_grad(int nb, const double* __restrict__ bins,
                                                                  const double* __restrict__ target,
                                                                  double* __restrict__ loss, double* __restrict__ g) {
  __shared__ int s_cnt[UR_LOSS_THREADS / 32];
  __shared__ double s_sum[UR_LOSS_THREADS / 32];
  const double* mean = bins + (size_t)UR_BIN_MEAN * nb;
  int cnt = 0;
  for (int j = threadIdx.x; j < nb; j += UR_LOSS_THREADS) {
    const double m = mean[j];
    cnt += (isfinite(m) && m > 0.0) ? 1 : 0;
  }
#pragma unroll
  for (int o = 16; o > 0; o >>= 1) cnt += __shfl_down_sync(0xffffffffu, cnt, o);
  if ((threadIdx.x & 31) == 0) s_cnt[threadIdx.x >> 5] = cnt;
  __syncthreads();
  int ntot = 0;
  for (int w = 0; w < UR_LOSS_THREADS / 32; ++w) ntot += s_cnt[w];
  const double nv = (double)(ntot > 0 ? ntot : 1);
  const int j = blockIdx.x * UR_LOSS_THREADS + threadIdx.x;
  double d2 = 0.0;
  if (j < nb) {
    const double m = mean[j];
    double gj = 0.0;
    if (isfinite(m) && m > 0.0) {
      const double d = log(m) - log(target[j]);
      d2 = d * d;
      gj = 2.0 * d / (m * nv);
    }
    g[j] = gj;
  }
#pragma unroll
  for (int o = 16; o > 0; o >>= 1) d2 += __shfl_down_sync(0xffffffffu, d2, o);
  if ((threadIdx.x & 31) == 0) s_sum[threadIdx.x >> 5] = d2;
  __syncthreads();
  if (threadIdx.x == 0 && loss) {
    double tot = 0.0;
    for (int w = 0; w < UR_LOSS_THREADS / 32; ++w) tot += s_sum[w];
    if (tot != 0.0) atomicAdd(loss, tot / nv);
  }
}

extern "C" ur_status ur_log_mse_grad(int32_t nbins, const double* bins, const double* target, double* loss,
                                     double* dl_dmean, void* stream) {
  UR_REQUIRE(nbins >= 1 && bins && target && dl_dmean, "ur_log_mse_grad: bad argument");
  UR_REQUIRE(nbins <= UR_LOSS_MAX_BINS, "ur_log_mse_grad: %d bins (at most %d)", nbins, UR_LOSS_MAX_BINS);
  cudaStream_t s = (cudaStream_t)stream;
  ur_timing_begin("loss_grad", s);
  if (loss) UR_CUDA_CHECK(cudaMemsetAsync(loss, 0, sizeof(double), s));
  k_log_mse_grad<<<(nbins + UR_LOSS_THREADS - 1) / UR_LOSS_THREADS, UR_LOSS_THREADS, 0, s>>>(nbins, bins, target, loss,
                                                                                              dl_dmean);
  UR_LAUNCH_CHECK("k_log_mse_grad");
  ur_timing_end(s);
  return UR_OK;
}

AdjRange ur_adj_range(const ur_plan* p, const ShapeArgs& sh, bool want_mask) {
  AdjRange r = {0, p->n, 0, p->n, 0};
  if (want_mask || !(sh.rb2 < INFINITY)) return r;
  ur_mask_range(sh, sh.cz, p->n, &r.zlo, &r.zhi);
  ur_mask_range(sh, sh.cy, p->n, &r.ylo, &r.yhi);
  r.row_skip = 1;
  return r;
}

// columns with kx^2 + ky^2 at or beyond the closing threshold have zero scales at every kz: the
// adjoint z pass leaves them unwritten and its y pass reads them as zeros
int ur_k2_zero(const ur_plan* p) { return (int)p->thr_host[p->nbins]; }

// Blocks of the generic row pass: as many cell rows per block as fill its RB rows, but not so many that a
// small grid has fewer than `least` blocks
void ur_grad_blocks(const AdjRange& rg, GenGradArgs* g, int least, int* gx, long long* gy) {
  const int U = g->U;
  g->zlo = rg.zlo;
  g->zhi = rg.zhi;
  g->ylo = rg.ylo;
  g->yhi = rg.yhi;
  g->row_skip = rg.row_skip;
  g->nza = (rg.zhi - rg.zlo + U - 1) / U;
  g->nyb = (rg.yhi - rg.ylo + U - 1) / U;
  const int per = g->nza * g->nyb;
  if (per <= 0) {
    g->nza = g->nyb = g->G = 1;
    *gx = 1;
    *gy = 0;
    return;
  }
  g->G = g->RB / per;
  if (g->G < 1) g->G = 1;
  if (g->G > U) g->G = U;
  while (g->G > 1 && U * ((U + g->G - 1) / g->G) < least) g->G = (g->G + 1) / 2;
  *gx = (g->G * per + g->RB - 1) / g->RB;
  *gy = (long long)U * ((U + g->G - 1) / g->G);
}

size_t ur_grad_smem(const ur_plan* p) {
  const size_t rb = (size_t)p->row_rb;
  return ur_align_up(rb * p->H * sizeof(float2), 16) + rb * sizeof(GradRow) + (rb + 1) * sizeof(int);
}

extern "C" ur_status ur_backward(const ur_plan* p, const double* dl_dmean, const double* fwd_bins, const void* F,
                                 const float* cell, int32_t ucell, const int32_t* origin, const ur_shape* shape,
                                 const float* weights, float* dl_dcell, float* dl_dmask, void* ws, size_t ws_bytes,
                                 void* stream) {
  UR_REQUIRE(p && dl_dmean && fwd_bins && cell && shape && dl_dcell && ws, "ur_backward: null argument");
  UR_REQUIRE(ucell >= 1, "ur_backward: empty cell");
  UR_REQUIRE(!origin || (origin[0] >= 0 && origin[1] >= 0 && origin[2] >= 0), "ur_backward: origin must be >= 0");
  UR_REQUIRE(ws_bytes >= ur_workspace_size(p, UR_WS_FORWARD | UR_WS_BACKWARD), "ur_backward: workspace %zu < %zu bytes",
             ws_bytes, ur_workspace_size(p, UR_WS_FORWARD | UR_WS_BACKWARD));
  UR_REQUIRE(shape->kind >= UR_SHAPE_SPHERE && shape->kind <= UR_SHAPE_WEIGHTS, "ur_backward: bad shape kind");
  UR_REQUIRE(shape->kind != UR_SHAPE_WEIGHTS || weights, "ur_backward: weights required for UR_SHAPE_WEIGHTS");
  UR_REQUIRE(!dl_dmask || ((uintptr_t)dl_dmask % 8) == 0, "ur_backward: dl_dmask must be 8-byte aligned");
  if (p->vsinc) {
    ur_set_error("ur_backward: the adjoint of the voxel-sinc corrected binning is not built");
    return UR_ERR_UNSUPPORTED;
  }
  UR_TRY(ur_fault_point("backward"));
  cudaStream_t s = (cudaStream_t)stream;
  const int n = p->n, H = p->H, nb = p->nbins;
  const double n3 = (double)n * n * n;
  float2* X = (float2*)ws;
  float2* Y = (float2*)((char*)ws + ur_align_up(p->ws_inter, 256));
  float* sigma = (float*)((char*)Y + ur_align_up(p->ws_inv, 256));

  ur_timing_begin("sigma", s);
  k_sigma<<<(nb + 255) / 256, 256, 0, s>>>(dl_dmean, fwd_bins, nb, n3, F != nullptr, sigma);
  UR_LAUNCH_CHECK("k_sigma");
  ur_timing_end(s);

  // B1
  ColArgs a = ur_col_args(p);
  a.ncols = (long long)n * H;
  a.A = p->xp;
  a.S = (long long)n * p->xp;
  a.Ad = p->xp;
  a.Sd = (long long)n * p->xp;
  a.dst = Y;
  a.sigma = sigma;
  if (F) {  // caller's layout: rows of N/2+1
    a.src = (const float2*)F;
    a.A = H;
    a.S = (long long)n * H;
    a.nload = n;
    a.zoff = 0;
    a.skip_fwd = 1;
  } else {
    a.src = X;
    a.nload = p->nz;
    a.zoff = p->z0;
    a.skip_fwd = 0;
  }
  const long long tiles = (a.ncols + a.TX - 1) / a.TX;
  const ShapeArgs sh = ur_shape_args(shape);
  const AdjRange rg = ur_adj_range(p, sh, dl_dmask != nullptr);
  const int cnt = rg.zhi - rg.zlo, k2_zero = ur_k2_zero(p);
  a.k2_zero = k2_zero;
  if (cnt < n) {
    a.out_lo = rg.zlo;
    a.out_cnt = cnt;
  }
  if (!p->fast) UR_REQUIRE((long long)ucell * ucell <= 65535, "ur_backward: cell edge %d too large", ucell);
  UR_CUDA_CHECK(cudaMemsetAsync(dl_dcell, 0, sizeof(float) * (size_t)ucell * ucell * ucell, s));
  if (p->fast) UR_REQUIRE(!weights || ((uintptr_t)weights % 8) == 0, "ur_backward: weights must be 8-byte aligned");
  if (cnt <= 0) return UR_OK;  // the mask is zero everywhere and dL/dm is not wanted
  ur_timing_begin("adj_cols_z", s);
  if (p->fast) {
    UR_TRY(ur_fast_cols(n, P2_Z_ADJ, a, s));
  } else {
    UR_TRY(ur_launch_cols(COL_ZADJ, false, p, a, (int)tiles, p->col_smem, s));
  }
  ur_timing_end(s);

  if (p->fast) {
    // B2 + B3, over all planes with the y-inverse in place, or in plane chunks
    // whose y-inverse goes to a chunk buffer that the row pass of the same chunk
    // reads while it is still in L2.
    const bool whole = p->chunk_planes >= n;
    float2* C = (float2*)((char*)sigma + ur_align_up(p->ws_sigma, 256));
    GradArgs g;
    memset(&g, 0, sizeof g);
    g.tw = p->tw;
    g.stw = p->stw + p->stw_m_off;
    g.cell = cell;
    g.ucell = ucell;
    if (origin) {  // the row kernel takes the origin reduced modulo the cell edge
      g.ox = origin[0] % ucell;
      g.oy = origin[1] % ucell;
      g.oz = origin[2] % ucell;
    }
    g.sh = sh;
    g.weights = shape->kind == UR_SHAPE_WEIGHTS ? weights : nullptr;
    g.inv_n3 = (float)(1.0 / n3);
    g.dl_dmask = dl_dmask;
    g.dl_dcell = dl_dcell;
    for (int p0 = 0; p0 < cnt; p0 += p->chunk_planes) {
      const int np = (p0 + p->chunk_planes <= cnt) ? p->chunk_planes : cnt - p0;
      ColArgs b = ur_col_args(p);
      b.src = Y + (long long)p0 * n * p->xp;
      b.dst = whole ? Y : C;
      b.ncols = (long long)np * H;
      b.A = (long long)n * p->xp;
      b.S = p->xp;
      b.Ad = b.A;
      b.Sd = b.S;
      b.nload = n;
      b.zoff = 0;
      b.nbins = 0;
      b.k2_zero = k2_zero;
      b.row_skip = rg.row_skip;
      b.gen_z0 = rg.zlo + p0;
      b.sh = sh;
      ur_timing_begin("adj_cols_y", s);
      UR_TRY(ur_fast_cols(n, P2_Y_INV, b, s));
      ur_timing_end(s);
      g.Y = whole ? Y : C;
      g.yp = p->xp;
      g.ybase_z = rg.zlo + p0;
      g.z0 = rg.zlo + p0;
      ur_timing_begin("adj_rows_grad", s);
      UR_TRY(ur_fast_rows_grad(n, g, np, s));
      ur_timing_end(s);
    }
    return UR_OK;
  }

  // B2
  ColArgs b = ur_col_args(p);
  b.src = Y;
  b.dst = Y;
  b.ncols = (long long)cnt * H;
  b.A = (long long)n * p->xp;
  b.S = p->xp;
  b.Ad = b.A;
  b.Sd = b.S;
  b.nload = n;
  b.zoff = 0;
  b.nbins = 0;
  b.k2_zero = k2_zero;
  b.row_skip = rg.row_skip;
  b.gen_z0 = rg.zlo;
  b.sh = sh;
  ur_timing_begin("adj_cols_y", s);
  UR_TRY(ur_launch_cols(COL_Y, true, p, b, (int)((b.ncols + b.TX - 1) / b.TX), p->col_smem, s));
  ur_timing_end(s);

  // B3
  GenGradArgs ga;
  memset(&ga, 0, sizeof ga);
  ga.Y = Y;
  ga.yp = p->xp;
  ga.N = n;
  ga.RB = p->row_rb;
  ga.nst = p->sched_m.nst;
  ga.sched = p->d_sched + UR_MAX_STAGES;
  ga.tw = p->tw;
  ga.cell = cell;
  ga.U = ucell;
  if (origin) {  // reduced modulo the cell edge, as the cell indices are
    ga.ox = origin[0] % ucell;
    ga.oy = origin[1] % ucell;
    ga.oz = origin[2] % ucell;
  }
  ga.sh = sh;
  ga.weights = shape->kind == UR_SHAPE_WEIGHTS ? weights : nullptr;
  ga.inv_n3 = (float)(1.0 / n3);
  ga.dl_dmask = dl_dmask;
  ga.dl_dcell = dl_dcell;
  int gx = 0;
  long long gy = 0;
  ur_grad_blocks(rg, &ga, p->num_sms, &gx, &gy);
  if (gy == 0) return UR_OK;
  const size_t smem = ur_grad_smem(p);
  UR_CUDA_CHECK(cudaFuncSetAttribute(k_rows_grad, cudaFuncAttributeMaxDynamicSharedMemorySize, (int)smem));
  ur_timing_begin("adj_rows_grad", s);
  k_rows_grad<<<dim3((unsigned)gx, (unsigned)gy), 256, smem, s>>>(ga);
  UR_LAUNCH_CHECK("k_rows_grad");
  ur_timing_end(s);
  return UR_OK;
}

// ---------------------------------------------------------------------------
// Batched adjoint launches
// ---------------------------------------------------------------------------
__global__ void k_batch_sigma(const BatchSigmaItem* __restrict__ items) {
  const BatchSigmaItem& it = items[blockIdx.y];
  const int j = blockIdx.x * blockDim.x + threadIdx.x;
  if (j >= it.nb) return;
  const double n = it.bins[UR_BIN_COUNT * it.nb + j];
  it.sigma[j] = (float)(n > 0 ? 2.0 * it.g[j] / n / it.n3 : 0.0);
}

__global__ void __launch_bounds__(256, 4) k_batch_grad(const BatchGradItem* __restrict__ items,
                                                       const long long* __restrict__ start, int count) {
  int lo = 0, hi = count - 1;
  const long long b = blockIdx.x;
  while (lo < hi) {
    const int mid = (lo + hi + 1) >> 1;
    if (__ldg(start + mid) <= b) lo = mid;
    else hi = mid - 1;
  }
  const BatchGradItem& it = items[lo];
  const long long local = b - __ldg(start + lo);
  const int gx = it.gx;
  rows_grad_body(it.g, (int)(local % gx), (int)(local / gx));
}

ur_status ur_batch_launch_sigma(const BatchSigmaItem* items, int count, int maxnb, cudaStream_t s) {
  if (count <= 0) return UR_OK;
  k_batch_sigma<<<dim3((unsigned)((maxnb + 255) / 256), (unsigned)count), 256, 0, s>>>(items);
  UR_LAUNCH_CHECK("k_batch_sigma");
  return UR_OK;
}

ur_status ur_batch_launch_grad(const BatchGradItem* items, const long long* start, int count, long long nblocks,
                               size_t smem, cudaStream_t s) {
  if (nblocks <= 0) return UR_OK;
  UR_REQUIRE(nblocks < (1ll << 31), "batched adjoint rows: too many blocks");
  if (smem > UR_DYN_SMEM_FREE)
    UR_CUDA_CHECK(cudaFuncSetAttribute(k_batch_grad, cudaFuncAttributeMaxDynamicSharedMemorySize, (int)smem));
  k_batch_grad<<<(unsigned)nblocks, 256, smem, s>>>(items, start, count);
  UR_LAUNCH_CHECK("k_batch_grad");
  return UR_OK;
}

// ---------------------------------------------------------------------------
// Out-of-core adjoint (the per-slab adjoint of the streamed forward): the inverse
// intermediate of all N planes does not fit when the grid is large, so the output planes
// are produced slab by slab.  For every slab the z pass is recomputed over all spectrum
// columns from the forward intermediate (F~ along z, times sigma(bin), inverse along z)
// and only the slab's planes are kept; the slab then goes through the y inverse and the
// row pass (dL/du accumulated, dL/dm written to a device staging buffer and copied to
// pinned host memory on a copy stream, double-buffered).
// ---------------------------------------------------------------------------
extern "C" ur_status ur_plan_set_adj_slab_planes(ur_plan* p, int32_t planes) {
  UR_REQUIRE(p && planes >= 1, "ur_plan_set_adj_slab_planes: bad argument");
  p->adj_slab_planes = planes > p->n ? p->n : planes;
  return UR_OK;
}

extern "C" ur_status ur_backward_slabs(const ur_plan* p, const double* dl_dmean, const double* fwd_bins,
                                       const float* cell, int32_t ucell, const int32_t* origin, const ur_shape* shape,
                                       const float* weights, float* dl_dcell, float* dl_dmask_host, void* ws,
                                       size_t ws_bytes, void* stream) {
  UR_REQUIRE(p && dl_dmean && fwd_bins && cell && shape && dl_dcell && ws, "ur_backward_slabs: null argument");
  UR_REQUIRE(p->fast, "ur_backward_slabs: power-of-two grids only (edge %d)", p->n);
  UR_REQUIRE(ucell >= 1, "ur_backward_slabs: empty cell");
  UR_REQUIRE(!origin || (origin[0] >= 0 && origin[1] >= 0 && origin[2] >= 0), "ur_backward_slabs: origin must be >= 0");
  UR_REQUIRE(shape->kind >= UR_SHAPE_SPHERE && shape->kind <= UR_SHAPE_WEIGHTS, "ur_backward_slabs: bad shape kind");
  UR_REQUIRE(shape->kind != UR_SHAPE_WEIGHTS || weights, "ur_backward_slabs: weights required for UR_SHAPE_WEIGHTS");
  UR_REQUIRE(!weights || ((uintptr_t)weights % 8) == 0, "ur_backward_slabs: weights must be 8-byte aligned");
  const size_t need = ur_workspace_size(p, UR_WS_FORWARD | UR_WS_ADJ_SLABS);
  UR_REQUIRE(ws_bytes >= need, "ur_backward_slabs: workspace %zu < %zu bytes", ws_bytes, need);
  UR_REQUIRE(((uintptr_t)ws % 256) == 0, "ur_backward_slabs: misaligned ws");
  if (p->vsinc) {
    ur_set_error("ur_backward_slabs: the adjoint of the voxel-sinc corrected binning is not built");
    return UR_ERR_UNSUPPORTED;
  }
  if (dl_dmask_host) {
    cudaPointerAttributes at;
    const cudaError_t e = cudaPointerGetAttributes(&at, dl_dmask_host);
    UR_REQUIRE(e == cudaSuccess && at.type == cudaMemoryTypeHost,
               "ur_backward_slabs: dl_dmask_host must be page-locked host memory");
  }
  UR_TRY(ur_fault_point("backward"));
  cudaStream_t s = (cudaStream_t)stream;
  const int n = p->n, H = p->H, nb = p->nbins, S = p->adj_slab_planes;
  const double n3 = (double)n * n * n;
  // workspace: [X][two host staging slabs][Y slab][sigma][two dL/dm staging slabs of SM planes]
  const int SM = ur_adj_dm_planes(p);
  float2* X = (float2*)ws;
  char* o = (char*)ws + ur_align_up(p->ws_inter, 256) + 2 * ur_align_up(p->ws_slab, 256);
  float2* Ys = (float2*)o;
  o += ur_align_up((size_t)S * n * p->xp * sizeof(float2), 256);
  float* sigma = (float*)o;
  o += ur_align_up(p->ws_sigma, 256);
  float* dm[2];
  const size_t dm_bytes = (size_t)SM * n * n * sizeof(float);
  dm[0] = (float*)o;
  dm[1] = (float*)(o + ur_align_up(dm_bytes, 256));

  k_sigma<<<(nb + 255) / 256, 256, 0, s>>>(dl_dmean, fwd_bins, nb, n3, 0, sigma);
  UR_LAUNCH_CHECK("k_sigma");
  UR_CUDA_CHECK(cudaMemsetAsync(dl_dcell, 0, sizeof(float) * (size_t)ucell * ucell * ucell, s));
  const int k2_zero = ur_k2_zero(p);
  const AdjRange rg = ur_adj_range(p, ur_shape_args(shape), dl_dmask_host != nullptr);

  GradArgs g;
  memset(&g, 0, sizeof g);
  g.tw = p->tw;
  g.stw = p->stw + p->stw_m_off;
  g.cell = cell;
  g.ucell = ucell;
  if (origin) {
    g.ox = origin[0] % ucell;
    g.oy = origin[1] % ucell;
    g.oz = origin[2] % ucell;
  }
  g.sh = ur_shape_args(shape);
  g.weights = shape->kind == UR_SHAPE_WEIGHTS ? weights : nullptr;
  g.inv_n3 = (float)(1.0 / n3);
  g.dl_dcell = dl_dcell;

  cudaStream_t cs = nullptr;
  cudaEvent_t done[2] = {nullptr, nullptr}, freed[2] = {nullptr, nullptr};
  ur_status st = UR_OK;
  if (dl_dmask_host) {
    bool ok = cudaStreamCreateWithFlags(&cs, cudaStreamNonBlocking) == cudaSuccess;
    for (int b = 0; b < 2 && ok; ++b)
      ok = cudaEventCreateWithFlags(&done[b], cudaEventDisableTiming) == cudaSuccess &&
           cudaEventCreateWithFlags(&freed[b], cudaEventDisableTiming) == cudaSuccess;
    if (!ok) {
      ur_set_error("ur_backward_slabs: cannot create the copy stream or its events");
      st = UR_ERR_CUDA;
    }
  }
  int sub = 0;  // running index of the dL/dm staging sub-slabs (double-buffered)
  for (int za = rg.zlo; za < rg.zhi && st == UR_OK; za += S) {
    const int cnt = za + S <= rg.zhi ? S : rg.zhi - za;
    // z pass over every column, keeping planes [za, za + cnt)
    ColArgs a = ur_col_args(p);
    a.ncols = (long long)n * H;
    a.A = p->xp;
    a.S = (long long)n * p->xp;
    a.Ad = p->xp;
    a.Sd = (long long)n * p->xp;
    a.src = X;
    a.nload = p->nz;
    a.zoff = p->z0;
    a.dst = Ys;
    a.sigma = sigma;
    a.k2_zero = k2_zero;
    a.out_lo = za;
    a.out_cnt = cnt;
    ur_timing_begin("adj_cols_z", s);
    st = ur_fast_cols(n, 3 /* z adjoint */, a, s);
    ur_timing_end(s);
    if (st != UR_OK) break;
    // y inverse of the slab, in place
    ColArgs c = ur_col_args(p);
    c.src = Ys;
    c.dst = Ys;
    c.ncols = (long long)cnt * H;
    c.A = (long long)n * p->xp;
    c.S = p->xp;
    c.Ad = c.A;
    c.Sd = c.S;
    c.nload = n;
    c.zoff = 0;
    c.nbins = 0;
    c.k2_zero = k2_zero;
    c.row_skip = rg.row_skip;
    c.gen_z0 = za;
    c.sh = g.sh;
    ur_timing_begin("adj_cols_y", s);
    st = ur_fast_cols(n, 1 /* y inverse */, c, s);
    ur_timing_end(s);
    if (st != UR_OK) break;
    // rows of the slab in sub-slabs of SM planes: dL/du accumulated, dL/dm into staging buffer b
    for (int zb = za; zb < za + cnt && st == UR_OK; zb += (dl_dmask_host ? SM : cnt), ++sub) {
      const int cz = dl_dmask_host ? (zb + SM <= za + cnt ? SM : za + cnt - zb) : cnt;
      const int b = sub & 1;
      if (dl_dmask_host && sub >= 2) cudaStreamWaitEvent(s, freed[b], 0);
      g.Y = Ys;
      g.yp = p->xp;
      g.ybase_z = za;
      g.z0 = zb;
      g.dl_dmask = dl_dmask_host ? dm[b] : nullptr;
      g.mbase_z = zb;
      ur_timing_begin("adj_rows_grad", s);
      st = ur_fast_rows_grad(n, g, cz, s);
      ur_timing_end(s);
      if (st != UR_OK) break;
      if (dl_dmask_host) {
        cudaEventRecord(done[b], s);
        cudaStreamWaitEvent(cs, done[b], 0);
        const cudaError_t ce = cudaMemcpyAsync(dl_dmask_host + (size_t)zb * n * n, dm[b], (size_t)cz * n * n * sizeof(float),
                                               cudaMemcpyDeviceToHost, cs);
        if (ce != cudaSuccess) {
          ur_set_error("ur_backward_slabs: dL/dm copy failed: %s", cudaGetErrorString(ce));
          st = UR_ERR_CUDA;
          break;
        }
        cudaEventRecord(freed[b], cs);
      }
    }
  }
  if (cs) {
    // the caller's stream waits for the copies still queued
    cudaEvent_t end;
    if (cudaEventCreateWithFlags(&end, cudaEventDisableTiming) == cudaSuccess) {
      cudaEventRecord(end, cs);
      cudaStreamWaitEvent(s, end, 0);
      cudaEventDestroy(end);
    }
    cudaStreamDestroy(cs);
  }
  for (int b = 0; b < 2; ++b) {
    if (done[b]) cudaEventDestroy(done[b]);
    if (freed[b]) cudaEventDestroy(freed[b]);
  }
  return st;
}
