// Argument blocks and host entry points of the power-of-two kernels.
#pragma once

#include "ur_forward.cuh"
#include "ur_density.cuh"

// Values per column and thread of the column transforms: 8 up to 512 (pairs of columns, ur_pair.cu), 16
// from 1024 on (single columns, ur_fast.cu: three radix-16 stages at 4096 instead of four radix-8
// ones; measured 22-23 % faster steps), 32 in the adjoint's y pass at 1024 (ColCfg)
#define UR_FAST_COL_E(n, mode) ((n) == 1024 && ((mode) == P2_Y_INV || (mode) == P2_Y_INV_ROWS) ? 32 : 16)
// ... and of the transforms of stored rows of n reals (generated rows and the adjoint rows: 8)
#define UR_FAST_STORED_ROW_E(n) ((n) == 1024 ? 16 : 8)

// P2_Y_INV_ROWS: P2_Y_INV that writes only the rows inside the particle (ColArgs::row_skip); the
// launchers choose it, since the test costs the full inverse 6 % (512^3: 203 -> 215 us)
enum { P2_Y_FWD = 0, P2_Y_INV = 1, P2_Z_BIN = 2, P2_Z_ADJ = 3, P2_Y_INV_ROWS = 4 };

struct RowArgs {
  const void* ed;          // density rows (GEN = 0), plane-major, nrows x N
  float2* X;               // output half-spectrum rows, nrows x (N/2+1), xp apart
  int xp;
  long long nrows;
  int z0;                  // absolute plane index of row 0 / N (GEN = 1)
  const float* cell;       // GEN = 1: unit cell U^3
  int ucell, ox, oy, oz;   // origin >= 0
  FastDiv fu;              // division by ucell
  ShapeArgs sh;
  LatArgs lat;             // GEN = 2: the cell sampled on a rotated lattice
  const float* weights;    // GEN >= 1 with UR_SHAPE_WEIGHTS: full-box weights
  const float2* tw;        // table exp(-2 pi i t / N), t < N
  const float2* stw;       // stage twiddles of the N/2-point transform (power-of-two kernels)
  int skip_empty;          // GEN >= 1: rows outside the particle (row_outside) are not written
};

struct GradArgs {
  const float2* Y;         // inverse-transformed rows (along z and y), planes [ybase_z, ...)
  int yp;                  // row pitch of Y
  int ybase_z;
  int z0;                  // first absolute plane of this launch
  int rb;                  // rows per block (set by the launcher)
  const float2* tw;
  const float2* stw;       // stage twiddles of the N/2-point transform
  const float* cell;
  int ucell, ox, oy, oz;   // origin, each reduced to [0, ucell) by the host
  int cstep;               // (N/8) mod ucell (set by the launcher)
  ShapeArgs sh;
  const float* weights;
  float inv_n3;
  float* dl_dmask;         // dL/dm planes from mbase_z on (plane z at z - mbase_z)
  int mbase_z;
  float* dl_dcell;
};

// one item of a batched generic row pass
struct BatchRowsItem {
  RowArgs ra;
  int N, RB, nst;
  const StageInfo* sched;
};

bool ur_fast_supported(int n);
ur_status ur_fast_rows(int n, const RowArgs& a, int gen, int ed_f16, cudaStream_t s);
ur_status ur_fast_cols(int n, int mode, const ColArgs& a, cudaStream_t s);
bool ur_pair_supported(int n);
size_t ur_stage_twiddles(int lg, int E, float2* out);
size_t ur_pair_twiddles(int n, float4* out);
ur_status ur_pair_cols(int n, int mode, const ColArgs& a, cudaStream_t s);
ur_status ur_fast_rows_grad(int n, const GradArgs& a, int nplanes, cudaStream_t s);
