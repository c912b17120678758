// Operator apply: y = kappa .* (L phi) (or L phi), the homogeneous part of the
// flux-divergence Laplacian of Sec. 2.3.  Two passes:
//   K4  template cells: the translation-invariant cell stencil of the interior
//       (every face stencil there is the same weighted-LS template);
//   K5  irregular cells (near the EB or a domain wall): footprint-dense rows,
//       stored footprint-major so that consecutive rows load coalesced.
// Covered cells get y = 0.
#include <cuda_runtime.h>
#include <algorithm>
#include <stdint.h>
#include <string.h>
#include <vector>

#include "eb_apply.cuh"
#include "eb_internal.cuh"
#include "eb_apply_tma.cuh"
#include "eb_apply_quad.cuh"
#include "eb_apply_wall.cuh"
#include "eb_apply_brick.cuh"
#include "eb_apply_fold.cuh"

#include <cuda.h>

namespace eb {

// footprint offsets of the template stencil, staged in shared memory
template <typename T, int TILE_X>
__global__ void __launch_bounds__(256) k_apply_template(ApplyArgs<T> a) {
  extern __shared__ __align__(16) unsigned char sm_raw[];
  int32_t* off = reinterpret_cast<int32_t*>(sm_raw);
  T* coef = reinterpret_cast<T*>(sm_raw + ((a.nfoot * 4 + 15) / 16) * 16);
  for (int i = threadIdx.x; i < a.nfoot; i += blockDim.x) {
    off[i] = a.foot_off[i];
    coef[i] = a.tmpl[i];
  }
  __syncthreads();
  int64_t c = (int64_t)blockIdx.x * blockDim.x + threadIdx.x;
  if (c >= a.ncell) return;
  uint8_t kind = a.kind[c];
  if (kind == 2) return;  // written by the irregular pass
  T acc = 0;
  if (kind == 1) {
    const T* p = a.phi + c;
#pragma unroll 8
    for (int i = 0; i < a.nfoot; ++i) acc += coef[i] * __ldg(p + off[i]);
    if (!a.kappa_weighted) acc *= (T)a.inv_kappa[c];
  }
  a.y[c] = acc;
}

template <typename T>
__global__ void __launch_bounds__(256) k_apply_irregular(ApplyArgs<T> a) {
  extern __shared__ __align__(16) unsigned char sm_raw[];
  int32_t* off = reinterpret_cast<int32_t*>(sm_raw);
  for (int i = threadIdx.x; i < a.nfoot; i += blockDim.x) off[i] = a.foot_off[i];
  __syncthreads();
  int64_t t = (int64_t)blockIdx.x * blockDim.x + threadIdx.x;
  if (t >= a.n_irr) return;
  int64_t c = a.irr_cell[t];
  int64_t row = a.irr_row[t];
  const T* rows = a.rows + row;
  T acc = 0;
  const int64_t hi = a.ncell - 1;
  for (int i = 0; i < a.nfoot; ++i) {
    int64_t q = c + off[i];
    q = q < 0 ? 0 : (q > hi ? hi : q);  // out-of-domain offsets carry zero coefficients
    acc += __ldg(rows + (int64_t)i * a.n_rows) * __ldg(a.phi + q);
  }
  if (!a.kappa_weighted) acc *= (T)a.inv_kappa[c];
  a.y[c] = acc;
}

// Irregular rows for box neighbourhoods of radius R in D dimensions: the
// footprint is a union of x-contiguous segments (dz, dy, dx in [-X, X]) whose
// coefficients are consecutive in footprint order.  A lane has a row and W
// warps share out the segments of 32 rows (a rolled loop keeps the code small),
// summed in shared memory; a segment whose (y + dy, z + dz) leaves the grid has
// zero coefficients and is skipped, and only the x-ends of the first and last
// grid rows need an address clamp.  With W = 1 the chain of a row's loads is
// the kernel's time until the rows fill the chip: the 30000 wall-edge rows of a
// 100^3 grid take 56 us in FP32, and 17 us with W = 8 (FP64 at 160^3, 50000
// rows: 131 and 55 us).  From SEG_MANY rows on, where there are warps enough,
// the repeated index work costs more than it gives (FP32, 280000 rows: 91 and
// 93 us; 1.15 M rows: 306 and 370 us; FP64 within 1 % either way, whole applies of 141^3 to 201^3).
// 2-D in FP64 always takes one warp: the nine segments of a row have no chain to cut, and blocks with
// shared memory of their own, beside the template pass's larger ones on few SMs, make applies that follow
// one another wait for the SMs to change their partition: 29 us an apply at 200^2 to 300^2 with one warp, 110
// to 140 us with eight (FP32, where both passes fit one partition: 13 us either way, and 24 instead of 27 us alone).
constexpr int SEG_BLOCK_WARPS = 8;
constexpr int64_t SEG_MANY = 262144;

// footprint index of the first entry of segment (dy, dz)
template <int R, int D>
__device__ __forceinline__ int seg_first(int dy, int dz) {
  constexpr int L = R + 1;
  const int X = (dy < -R || dy > R || dz < -R || dz > R) ? R : L;
  if (D == 3) return canon_idx<R>(-X, dy, dz);
  return dy == -L ? 0 : 2 * R + 1 + (dy + R) * (2 * L + 1);
}

template <typename T, int R, int D, int W>
__global__ void __launch_bounds__(32 * SEG_BLOCK_WARPS) k_apply_irregular_seg(ApplyArgs<T> a, int nx, int ny, int nz) {
  constexpr int L = R + 1;
  constexpr int NZ = D == 3 ? 2 * L + 1 : 1;
  constexpr int NY = 2 * L + 1;
  __shared__ T part[SEG_BLOCK_WARPS][32];
  const int warp = threadIdx.x >> 5, lane = threadIdx.x & 31;
  const int64_t t = ((int64_t)blockIdx.x * (SEG_BLOCK_WARPS / W) + warp / W) * 32 + lane;
  const bool ok = t < a.n_irr;
  int64_t c = 0;
  T acc0 = 0, acc1 = 0;
  if (ok) {
    c = a.irr_cell[t];
    const int cx = (int)(c % nx);
    const int64_t cr = c / nx;
    const int cy = (int)(cr % ny), cz = (int)(cr / ny);
    const int64_t stride = a.n_rows;
    const T* row = a.rows + a.irr_row[t];
    const int64_t ncell = a.ncell;
    const T* cf = row;
#pragma unroll 1
    for (int sgi = warp % W; sgi < NZ * NY; sgi += W) {
      const int dz = D == 3 ? sgi / NY - L : 0;
      const int dy = sgi % NY - L;
      const int az = dz < 0 ? -dz : dz, ay = dy < 0 ? -dy : dy;
      if (az > R && ay > R) continue;
      const bool wide = !(az > R || ay > R);  // x extent L (wide) or R
      const int X = wide ? L : R;
      const int zz = cz + dz, yy = cy + dy;
      if (zz < 0 || zz >= nz || yy < 0 || yy >= ny) {
        cf += (int64_t)(2 * X + 1) * stride;
        continue;
      }
      if (W > 1) cf = row + (int64_t)seg_first<R, D>(dy, dz) * stride;  // one warp walks on from the last segment
      const int64_t base = (int64_t)nx * ((int64_t)yy + (int64_t)ny * zz) + cx;
      if (base - X >= 0 && base + X < ncell) {
        const T* ph = a.phi + base;
        if (wide) {
#pragma unroll
          for (int dx = -L; dx <= L; ++dx) {
            if (dx & 1) acc1 = fma(__ldg(cf), __ldg(ph + dx), acc1);
            else acc0 = fma(__ldg(cf), __ldg(ph + dx), acc0);
            cf += stride;
          }
        } else {
#pragma unroll
          for (int dx = -R; dx <= R; ++dx) {
            if (dx & 1) acc1 = fma(__ldg(cf), __ldg(ph + dx), acc1);
            else acc0 = fma(__ldg(cf), __ldg(ph + dx), acc0);
            cf += stride;
          }
        }
        continue;
      }
      for (int dx = -X; dx <= X; ++dx) {
        int64_t q = base + dx;
        q = q < 0 ? 0 : (q >= ncell ? ncell - 1 : q);
        acc0 = fma(__ldg(cf), __ldg(a.phi + q), acc0);
        cf += stride;
      }
    }
  }
  T acc = acc0 + acc1;
  if (W > 1) {
    part[warp][lane] = acc;
    __syncthreads();
  }
  if (warp % W == 0 && ok) {
#pragma unroll
    for (int w = 1; w < W; ++w) acc += part[warp + w][lane];
    if (!a.kappa_weighted) acc *= (T)a.inv_kappa[c];
    a.y[c] = acc;
  }
}

// wall-layer x-runs need 16-byte aligned phi for their vector loads
template <typename T>
static bool use_runs(const ApplyArgs<T>& a) {
  const ApplyPlan* pl = a.plan;
  return pl && pl->quad && pl->nG > 0 && ((uintptr_t)a.phi & 15u) == 0;
}

template <typename T>
static cudaError_t launch_runs(const ApplyArgs<T>& a, cudaStream_t st) {
  const ApplyPlan* pl = a.plan;
  XqArgs<T> x;
  x.nG = pl->nG;
  x.cellG = pl->cellG;
  x.classG = pl->classG;
  if constexpr (sizeof(T) == 4) x.rowsK = pl->rowsK32;
  else x.rowsK = pl->rowsK64;
  x.nfoot = a.nfoot;
  x.phi = a.phi;
  x.y = a.y;
  x.inv_kappa = a.inv_kappa;
  x.kappa_weighted = a.kappa_weighted;
  x.nx = pl->nx;
  x.ny = pl->ny;
  x.nz = pl->nz;
  const unsigned nb = (unsigned)((pl->nG + 31) / 32);
  if (pl->R == 3) k_class_xquad<T, 3><<<nb, 128, 0, st>>>(x);
  else k_class_xquad<T, 2><<<nb, 128, 0, st>>>(x);
  eb::count_launch();
  return cudaGetLastError();
}

template <typename T>
static cudaError_t launch_brick(const ApplyArgs<T>& a, cudaStream_t st) {
  const ApplyPlan* pl = a.plan;
  BrickArgs<T> b;
  b.nx = pl->nx;
  b.ny = pl->ny;
  b.nz = pl->nz;
  b.nyb = pl->nyb;
  b.nzb = pl->nzb;
  b.y_org = pl->y_org;
  b.z_org = pl->z_org;
  b.y_hi = pl->y_hi;
  b.z_hi = pl->z_hi;
  b.unit_class = pl->unit_class;
  if constexpr (sizeof(T) == 4) b.rowsK = pl->rowsK32;
  else b.rowsK = pl->rowsK64;
  b.nfoot = a.nfoot;
  b.phi = a.phi;
  b.y = a.y;
  b.inv_kappa = a.inv_kappa;
  b.kappa_weighted = a.kappa_weighted;
  const unsigned grid = (unsigned)(2 * b.nyb * b.nzb);
  cudaError_t e;
  if (pl->R == 3) {
    constexpr size_t sm = brick_smem<T, 3>();
    if ((e = cudaFuncSetAttribute(k_wall_brick<T, 3>, cudaFuncAttributeMaxDynamicSharedMemorySize, (int)sm))) return e;
    k_wall_brick<T, 3><<<grid, BR_W * 32, sm, st>>>(b);
  } else {
    constexpr size_t sm = brick_smem<T, 2>();
    if ((e = cudaFuncSetAttribute(k_wall_brick<T, 2>, cudaFuncAttributeMaxDynamicSharedMemorySize, (int)sm))) return e;
    k_wall_brick<T, 2><<<grid, BR_W * 32, sm, st>>>(b);
  }
  eb::count_launch();
  return cudaGetLastError();
}

#ifndef EB_QUAD_PER_SM
#define EB_QUAD_PER_SM 8  // CTAs per SM of the unique-row stream (0: one CTA per 128 rows)
#endif

template <typename T, int W>
static cudaError_t launch_seg_w(const ApplyArgs<T>& a, cudaStream_t st) {
  const ApplyPlan* pl = a.plan;
  constexpr int rows = 32 * SEG_BLOCK_WARPS / W, threads = 32 * SEG_BLOCK_WARPS;
  const unsigned nb = (unsigned)((a.n_irr + rows - 1) / rows);
  if (pl->dim == 3 && pl->R == 3) k_apply_irregular_seg<T, 3, 3, W><<<nb, threads, 0, st>>>(a, pl->nx, pl->ny, pl->nz);
  else if (pl->dim == 3) k_apply_irregular_seg<T, 2, 3, W><<<nb, threads, 0, st>>>(a, pl->nx, pl->ny, pl->nz);
  else if (pl->R == 3) k_apply_irregular_seg<T, 3, 2, W><<<nb, threads, 0, st>>>(a, pl->nx, pl->ny, pl->nz);
  else k_apply_irregular_seg<T, 2, 2, W><<<nb, threads, 0, st>>>(a, pl->nx, pl->ny, pl->nz);
  eb::count_launch();
  return cudaGetLastError();
}

template <typename T>
static cudaError_t launch_seg(const ApplyArgs<T>& a, cudaStream_t st) {
  const bool shared = a.n_irr < SEG_MANY && !(sizeof(T) == 8 && a.plan->dim == 2);
  return shared ? launch_seg_w<T, SEG_BLOCK_WARPS>(a, st) : launch_seg_w<T, 1>(a, st);
}

// class cells outside the runs and the slab bricks: per-cell segment walk over the canonical rows
template <typename T>
static cudaError_t launch_seg_rest(const ApplyArgs<T>& a, cudaStream_t st) {
  const ApplyPlan* pl = a.plan;
  ApplyArgs<T> c = a;
  c.n_irr = pl->nL;
  c.irr_cell = pl->cellL;
  c.irr_row = pl->classL;
  return launch_seg(c, st);
}

template <typename T>
static cudaError_t launch_irregular(const ApplyArgs<T>& a, cudaStream_t st) {
  const ApplyPlan* pl = a.plan;
  if (pl && pl->quad) {
    // unique rows (HBM stream) in the quad layout; without the x-runs (phi not 16-byte aligned) the class
    // rows (L2-resident, shared by the wall-layer cells) follow by the segment walk over the canonical rows
    const QuadArgs<T> q = quad_args<T>(*pl);
    int64_t bu = (pl->nU + 127) / 128;
    if (EB_QUAD_PER_SM > 0) bu = std::min<int64_t>(bu, (int64_t)pl->nsm * EB_QUAD_PER_SM);
    if (bu > 0) {
      if (pl->R == 3) k_irr_quad<T, 3, ApplyEpi><<<(unsigned)bu, 128, 0, st>>>(a, q, ApplyEpi());
      else k_irr_quad<T, 2, ApplyEpi><<<(unsigned)bu, 128, 0, st>>>(a, q, ApplyEpi());
      eb::count_launch();
    }
    if (use_runs(a)) return cudaGetLastError();  // the class cells go on the template pass's stream
    const int64_t nrest = pl->nC;
    if (nrest > 0) {
      ApplyArgs<T> c = a;
      c.n_irr = nrest;
      c.irr_cell = pl->cellC;
      c.irr_row = pl->classC;
      return launch_seg(c, st);
    }
    return cudaGetLastError();
  }
  if (pl && pl->seg) return launch_seg(a, st);
  const int64_t nb = (a.n_irr + 255) / 256;
  k_apply_irregular<T><<<(unsigned)nb, 256, a.nfoot * 4, st>>>(a);
  eb::count_launch();
  return cudaGetLastError();
}

typedef CUresult (*EncodeTiledFn)(CUtensorMap*, CUtensorMapDataType, cuuint32_t, void*, const cuuint64_t*,
                                   const cuuint64_t*, const cuuint32_t*, const cuuint32_t*, CUtensorMapInterleave,
                                   CUtensorMapSwizzle, CUtensorMapL2promotion, CUtensorMapFloatOOBfill);

static EncodeTiledFn encode_fn() {
  static const EncodeTiledFn fn = [] {  // looked up once (thread-safe static initialisation)
    void* p = nullptr;
    cudaDriverEntryPointQueryResult q;
    if (cudaGetDriverEntryPointByVersion("cuTensorMapEncodeTiled", &p, 12000, cudaEnableDefault, &q) == cudaSuccess &&
        q == cudaDriverEntryPointSuccess)
      return (EncodeTiledFn)p;
    return (EncodeTiledFn) nullptr;
  }();
  return fn;
}

template <typename T, int R, int D, bool ZSYM>
static cudaError_t launch_tma(const ApplyArgs<T>& a, const ApplyPlan& pl, cudaStream_t s) {
  constexpr int L = R + 1;
  constexpr int S = 2 * L + 1;
  constexpr int NP = D == 3 ? S + 1 : 1;
  constexpr int PX = TT_OX + 2 * TT_XH, PY = TT_OY + 2 * L;
  EncodeTiledFn enc = encode_fn();
  if (!enc) return cudaErrorNotSupported;
  CUtensorMap map;
  cuuint64_t gdim[3] = {(cuuint64_t)pl.nx, (cuuint64_t)pl.ny, (cuuint64_t)pl.nz};
  cuuint64_t gstr[2] = {(cuuint64_t)pl.nx * sizeof(T), (cuuint64_t)pl.nx * pl.ny * sizeof(T)};
  cuuint32_t box[3] = {PX, PY, 1};
  cuuint32_t es[3] = {1, 1, 1};
  CUresult r = enc(&map, sizeof(T) == 4 ? CU_TENSOR_MAP_DATA_TYPE_FLOAT32 : CU_TENSOR_MAP_DATA_TYPE_FLOAT64, 3,
                   (void*)a.phi, gdim, gstr, box, es, CU_TENSOR_MAP_INTERLEAVE_NONE, CU_TENSOR_MAP_SWIZZLE_NONE,
                   CU_TENSOR_MAP_L2_PROMOTION_L2_128B, CU_TENSOR_MAP_FLOAT_OOB_FILL_NONE);
  if (r != CUDA_SUCCESS) return cudaErrorInvalidValue;
  TmplCoef<T, R> cf;
  const T* cube;
  if constexpr (sizeof(T) == 4) cube = ZSYM ? pl.zcube32.data() : pl.cube32.data();
  else cube = ZSYM ? pl.zcube64.data() : pl.cube64.data();
  for (int i = 0; i < S * S * S; ++i) cf.c[i] = cube[i];
  TmplArgs<T> ta;
  ta.nx = pl.nx;
  ta.ny = pl.ny;
  ta.nz = pl.nz;
  ta.ntx = (pl.nx + TT_OX - 1) / TT_OX;
  ta.nty = (pl.ny + TT_OY - 1) / TT_OY;
  ta.zchunk = D == 3 ? 8 : 1;
  ta.nzc = (pl.nz + ta.zchunk - 1) / ta.zchunk;
  ta.items = (int64_t)ta.ntx * ta.nty * ta.nzc;
  ta.kind = a.kind;
  ta.inv_kappa = a.inv_kappa;
  ta.y = a.y;
  ta.kappa_weighted = a.kappa_weighted;
  ta.err = pl.err;
  constexpr size_t SLOT = ((PX * PY * sizeof(T) + 127) / 128) * 128;  // ring slot bytes (128-byte aligned TMA writes)
  size_t smem = (size_t)NP * SLOT + NP * 8;
  auto kern = k_apply_tma<T, R, D, ZSYM>;
  // attribute and occupancy are per device; kept for the last device seen
  static int cached_dev = -1, cached_per_sm = 0;
  int dev = 0;
  cudaError_t e = cudaGetDevice(&dev);
  if (e != cudaSuccess) return e;
  if (dev != cached_dev) {
    e = cudaFuncSetAttribute(kern, cudaFuncAttributeMaxDynamicSharedMemorySize, (int)smem);
    if (e != cudaSuccess) return e;
    e = cudaOccupancyMaxActiveBlocksPerMultiprocessor(&cached_per_sm, kern, TT_THREADS, smem);
    if (e != cudaSuccess) return e;
    cached_dev = dev;
  }
  int per_sm = cached_per_sm;
  int64_t grid = (int64_t)pl.nsm * (per_sm > 0 ? per_sm : 1);
  if (grid > ta.items) grid = ta.items;
  kern<<<(unsigned)grid, TT_THREADS, smem, s>>>(map, cf, ta); eb::count_launch();
  return cudaGetLastError();
}

// tensor map of phi for the staged planes (TT_OX + 2 TT_XH) x (TT_OY + 2L) of the template passes
template <typename T, int L>
static cudaError_t phi_map(const ApplyArgs<T>& a, const ApplyPlan& pl, CUtensorMap* map) {
  constexpr int PX = TT_OX + 2 * TT_XH, PY = TT_OY + 2 * L;
  EncodeTiledFn enc = encode_fn();
  if (!enc) return cudaErrorNotSupported;
  cuuint64_t gdim[3] = {(cuuint64_t)pl.nx, (cuuint64_t)pl.ny, (cuuint64_t)pl.nz};
  cuuint64_t gstr[2] = {(cuuint64_t)pl.nx * sizeof(T), (cuuint64_t)pl.nx * pl.ny * sizeof(T)};
  cuuint32_t box[3] = {PX, PY, 1};
  cuuint32_t es[3] = {1, 1, 1};
  CUresult r = enc(map, sizeof(T) == 4 ? CU_TENSOR_MAP_DATA_TYPE_FLOAT32 : CU_TENSOR_MAP_DATA_TYPE_FLOAT64, 3,
                   (void*)a.phi, gdim, gstr, box, es, CU_TENSOR_MAP_INTERLEAVE_NONE, CU_TENSOR_MAP_SWIZZLE_NONE,
                   CU_TENSOR_MAP_L2_PROMOTION_L2_128B, CU_TENSOR_MAP_FLOAT_OOB_FILL_NONE);
  return r == CUDA_SUCCESS ? cudaSuccess : cudaErrorInvalidValue;
}

#ifndef EB_FOLD_PER_SM
#define EB_FOLD_PER_SM 1  // persistent CTAs per SM of the folded template pass (0: as many as fit)
#endif

template <typename T, int R, bool TMA>
static cudaError_t launch_fold(const ApplyArgs<T>& a, const ApplyPlan& pl, cudaStream_t s) {
  constexpr int L = R + 1, F = L + 1;
  static_assert(FD_OX == TT_OX && FD_PX == TT_OX + 2 * TT_XH, "staged plane of the tensor map");
  CUtensorMap map;
  cudaError_t e = cudaSuccess;
  if constexpr (TMA) e = phi_map<T, L>(a, pl, &map);
  else memset(&map, 0, sizeof(map));
  if (e != cudaSuccess) return e;
  FoldCoef<T, R> cf;
  for (int i = 0; i < F * F * F; ++i) cf.c[i] = sizeof(T) == 4 ? (T)pl.fold32[i] : (T)pl.fold64[i];
  TmplArgs<T> ta;
  ta.nx = pl.nx;
  ta.ny = pl.ny;
  ta.nz = pl.nz;
  ta.ntx = (pl.nx + FD_OX - 1) / FD_OX;
  ta.nty = (pl.ny + FD_OY - 1) / FD_OY;
  ta.zchunk = TMA ? 8 : pl.fold_zchunk[sizeof(T) == 8];
  ta.nzc = (pl.nz + ta.zchunk - 1) / ta.zchunk;
  ta.items = (int64_t)ta.ntx * ta.nty * ta.nzc;
  ta.kind = a.kind;
  ta.inv_kappa = a.inv_kappa;
  ta.y = a.y;
  ta.kappa_weighted = a.kappa_weighted;
  ta.err = pl.err;
  constexpr size_t smem = fold_smem<T, R>();
  auto kern = k_apply_fold<T, R, TMA>;
  static int cached_dev = -1, cached_per_sm = 0;  // per device: attribute set, occupancy
  int dev = 0;
  if ((e = cudaGetDevice(&dev)) != cudaSuccess) return e;
  if (dev != cached_dev) {
    if ((e = cudaFuncSetAttribute(kern, cudaFuncAttributeMaxDynamicSharedMemorySize, (int)smem))) return e;
    if ((e = cudaOccupancyMaxActiveBlocksPerMultiprocessor(&cached_per_sm, kern, FD_THREADS, smem))) return e;
    cached_dev = dev;
  }
  int per_sm = cached_per_sm > 0 ? cached_per_sm : 1;
  if (EB_FOLD_PER_SM > 0 && per_sm > EB_FOLD_PER_SM) per_sm = EB_FOLD_PER_SM;
  int64_t grid = (int64_t)pl.nsm * per_sm;
  if (grid > ta.items) grid = ta.items;
  kern<<<(unsigned)grid, FD_THREADS, smem, s>>>(map, cf, ta, a.phi, pl.fold_act);
  eb::count_launch();
  return cudaGetLastError();
}

template <typename T>
static cudaError_t launch_template_pass(const ApplyArgs<T>& a, cudaStream_t s) {
  const ApplyPlan* pl = a.plan;
  // a tensor map needs rows of phi that start and end at 16 bytes: the plan looks at their length, the address is the call's
  const bool tma = pl && (sizeof(T) == 4 ? pl->tma32 : pl->tma64) && ((uintptr_t)a.phi & 15u) == 0;
  if (pl && pl->fold_act && (tma || pl->fold_copies[sizeof(T) == 8])) {
    if (pl->R == 3) return tma ? launch_fold<T, 3, true>(a, *pl, s) : launch_fold<T, 3, false>(a, *pl, s);
    return tma ? launch_fold<T, 2, true>(a, *pl, s) : launch_fold<T, 2, false>(a, *pl, s);
  }
  if (tma) {
    if (pl->dim == 3 && pl->R == 3)
      return pl->zsym ? launch_tma<T, 3, 3, true>(a, *pl, s) : launch_tma<T, 3, 3, false>(a, *pl, s);
    if (pl->dim == 3 && pl->R == 2)
      return pl->zsym ? launch_tma<T, 2, 3, true>(a, *pl, s) : launch_tma<T, 2, 3, false>(a, *pl, s);
    if (pl->dim == 2 && pl->R == 3) return launch_tma<T, 3, 2, false>(a, *pl, s);
    if (pl->dim == 2 && pl->R == 2) return launch_tma<T, 2, 2, false>(a, *pl, s);
  }
  size_t sm = ((a.nfoot * 4 + 15) / 16) * 16 + a.nfoot * sizeof(T);
  int64_t nb = (a.ncell + 255) / 256;
  k_apply_template<T, 32><<<(unsigned)nb, 256, sm, s>>>(a); eb::count_launch();
  return cudaGetLastError();
}

// y_j = sum_i M_ij phi_i over the cells i whose footprint holds j (M = kappa L, or L when not
// kappa-weighted: phi_i / kappa_i): the rows read in transposed order, one thread per output cell, no
// atomics.  Covered cells get 0.
template <typename T>
__global__ void __launch_bounds__(256) k_apply_transpose(ApplyArgs<T> a) {
  const int64_t j = (int64_t)blockIdx.x * blockDim.x + threadIdx.x;
  if (j >= a.ncell) return;
  if (a.kind[j] == 0) {
    a.y[j] = (T)0;
    return;
  }
  const int jx = (int)(j % a.nx), jy = (int)((j / a.nx) % a.ny), jz = (int)(j / ((int64_t)a.nx * a.ny));
  T acc = 0;
  for (int k = 0; k < a.nfoot; ++k) {
    const int ix = jx - a.foot_d[3 * k], iy = jy - a.foot_d[3 * k + 1], iz = jz - a.foot_d[3 * k + 2];
    if ((unsigned)ix >= (unsigned)a.nx || (unsigned)iy >= (unsigned)a.ny || (unsigned)iz >= (unsigned)a.nz) continue;
    const int64_t i = ix + (int64_t)a.nx * (iy + (int64_t)a.ny * iz);
    const uint8_t ki = a.kind[i];
    if (ki == 0) continue;
    const T m = ki == 1 ? a.tmpl[k] : a.rows[(int64_t)k * a.n_rows + a.row_of_cell[i]];
    const T p = a.kappa_weighted ? a.phi[i] : a.phi[i] * (T)a.inv_kappa[i];
    acc = fma(m, p, acc);
  }
  a.y[j] = acc;
}

// act[(z * 4 nty + g) * ntx + tx]: 1 when one of the cells (64 of x, FD_YB rows of y) of group g in tile column tx
// of plane z has the template row; ncells: how many (up to 255); a warp per entry
__global__ void k_fold_active(const uint8_t* __restrict__ kind, int nx, int ny, int nz, int ntx, int ngy,
                              uint8_t* __restrict__ act, uint8_t* __restrict__ ncells) {
  const int64_t t = (int64_t)blockIdx.x * (blockDim.x >> 5) + (threadIdx.x >> 5);
  if (t >= (int64_t)nz * ngy * ntx) return;
  const int lane = threadIdx.x & 31;
  const int tx = (int)(t % ntx), g = (int)(t / ntx % ngy), z = (int)(t / ((int64_t)ntx * ngy));
  int cells = 0;
  for (int r = 0; r < FD_YB; ++r) {
    const int y = g * FD_YB + r;
    for (int x = tx * FD_OX + lane; y < ny && x < nx && x < (tx + 1) * FD_OX; x += 32)
      cells += kind[x + (int64_t)nx * (y + (int64_t)ny * z)] == 1;
  }
  cells = __reduce_add_sync(0xffffffffu, cells);
  if (lane == 0) {
    act[t] = cells > 0;
    ncells[t] = (uint8_t)min(cells, 255);
  }
}
int64_t fold_act_size(int nx, int ny, int nz) {
  return (int64_t)nz * ((ny + FD_OY - 1) / FD_OY * (FD_OY / FD_YB)) * ((nx + FD_OX - 1) / FD_OX);
}
cudaError_t fold_active(const uint8_t* kind, int nx, int ny, int nz, uint8_t* act, uint8_t* cells, cudaStream_t s) {
  const int64_t n = fold_act_size(nx, ny, nz);
  k_fold_active<<<(unsigned)((n + 7) / 8), 256, 0, s>>>(kind, nx, ny, nz, (nx + FD_OX - 1) / FD_OX,
                                                       (ny + FD_OY - 1) / FD_OY * (FD_OY / FD_YB), act, cells);
  eb::count_launch();
  return cudaGetLastError();
}

// The folded pass with plain copies against the general template pass, for rows of phi that do not suit TMA.  The
// general pass spreads its cells over the whole chip; the folded one does a quarter of the arithmetic, but a CTA per SM
// works through pieces of tiles, and a small grid has few of them.  In FP64, where a plane of a tile takes 50 us
// (R = 3; R = 2: 27 us), pieces of 8 planes left most SMs idle on grids up to 120^3 (inside a sphere at 41^3, R = 3: 328 us
// an apply, 112 us with the general pass), so the pieces are as thin as it takes for the busiest CTA to have the
// least to do, by the tiles' active row groups (0.2 of a plane for a piece's first planes, 0.05 for a plane's barriers);
// with two rounds of CTAs or more the pieces stay at 8, where the sum is even enough (141^3: 1679 us, 1697 us with it).
// The folded pass pays from FOLD_CELLS template cells for each plane of the busiest CTA's on (applies in us, general
// and folded pass: R = 3, box minus a sphere, 45^3 with 6000 cells a plane 206 and 190, 53^3 with 15600 286 and 199, inside a sphere 47^3
// with 13700 162 and 172, 53^3 with 20900 206 and 128; R = 2, box, 45^3 with 16600 99 and 96, alone 84 and 115, inside,
// 47^3 with 18500 66 and 71, 65^3 with 24600 136 and 113).  In FP32 a plane takes 3 us and pieces of 8 are no
// loss; the folded pass pays from 2^14 template cells on for R = 3 (inside, 47^3 with 14000 cells 35 and 56 us, 53^3 with
// 23000 64 and 57; box, 45^3 with 6000 54 and 49) and from 2^16 on for R = 2 (inside, 47^3 with 19000 18 and 36, 59^3 with
// 44000 24 and 28, 65^3 with 62000 31 and 28; box, 61^3 with 76000 42 and 40).
constexpr double FOLD_CELLS[2] = {22000.0, 15000.0};  // R = 2, 3
void fold_plan(ApplyPlan* pl, const uint8_t* ncells) {
  constexpr int NG = FD_OY / FD_YB;
  const int ntx = (pl->nx + FD_OX - 1) / FD_OX, nty = (pl->ny + FD_OY - 1) / FD_OY, nz = pl->nz;
  // per tile: the work of the planes below z, in planes of four active groups and FD_PX columns
  std::vector<double> below((size_t)ntx * nty * (nz + 1));
  int64_t cells = 0;
  for (int tx = 0; tx < ntx; ++tx)
    for (int ty = 0; ty < nty; ++ty) {
      double* w = below.data() + (size_t)(tx * nty + ty) * (nz + 1);
      const double group = std::min(FD_PX, pl->nx - tx * FD_OX + 2 * TT_XH) / (double)(NG * FD_PX);
      for (int z = 0; z < nz; ++z) {
        w[z + 1] = w[z] + 0.05;
        for (int g = 0; g < NG; ++g) {
          const int n = ncells[((int64_t)z * nty * NG + ty * NG + g) * ntx + tx];
          cells += n;
          if (n > 0) w[z + 1] += group;
        }
      }
    }
  pl->fold_copies[0] = cells >= (pl->R == 3 ? 1 << 14 : 1 << 16);
  double best = 0.0;  // planes of the busiest CTA
  for (int zc = 8; zc >= 1; --zc) {
    const int nzc = (nz + zc - 1) / zc;
    const int64_t items = (int64_t)ntx * nty * nzc;
    std::vector<double> load(pl->nsm, 0.0);  // CTA i takes the items i, i + nsm, ...
    for (int64_t i = 0; i < items; ++i) {
      const double* w = below.data() + (size_t)(i / nzc) * (nz + 1);
      const int z0 = (int)(i % nzc) * zc;
      load[i % pl->nsm] += 0.2 + w[std::min(z0 + zc, nz)] - w[z0];
    }
    const double most = *std::max_element(load.begin(), load.end());
    if (zc == 8 || most < 0.95 * best) {
      best = most;
      pl->fold_zchunk[1] = zc;
    }
    if (zc == 8 && items >= 2 * pl->nsm) break;
  }
  pl->fold_copies[1] = cells >= FOLD_CELLS[pl->R == 3] * best;
}

template <typename T>
cudaError_t launch_apply(const ApplyArgs<T>& a, cudaStream_t s) {
  if (a.transpose) {
    k_apply_transpose<T><<<(unsigned)((a.ncell + 255) / 256), 256, 0, s>>>(a);
    eb::count_launch();
    return cudaGetLastError();
  }
  const ApplyPlan* pl = a.plan;
  cudaError_t e;
  bool fork = pl && pl->side && a.n_irr > 0;
  if (fork) {
    // the irregular rows run on the side stream, overlapped with the template pass (disjoint cells).
    // The template pass is launched first: its persistent grid takes a few CTAs per SM and the
    // HBM-bound row stream fills the rest of each SM, so the two run at the same time.
    if ((e = cudaEventRecord(pl->fork, s))) return e;
    if ((e = cudaStreamWaitEvent(pl->side, pl->fork, 0))) return e;
  }
  if ((e = launch_template_pass<T>(a, s))) return e;
  if (a.n_irr > 0) {
    if ((e = launch_irregular<T>(a, fork ? pl->side : s))) return e;
  }
  if (a.n_irr > 0 && use_runs(a)) {
    // The wall-layer class cells (FMA-bound, rows L2-resident) follow the template pass on the main stream while the
    // HBM-bound unique-row stream runs on the side stream.  In FP64 all but that stream is bound by the FP64 pipe,
    // and each pass alone leaves it idle in its last wave and its barriers: the slab bricks and the rest go behind
    // the row stream, beside the template pass (750 -> 496 us at 64^3, 2640 -> 2296 us at 160^3, 5809 -> 5168 us at
    // 220^3).  In FP32 the row stream is the longer side already: the same move takes 164 -> 202 us at 128^3 and gains
    // 1 % at 256^3, the runs alone 164 -> 176 us and 2 %.
    const cudaStream_t wall = sizeof(T) == 8 && fork ? pl->side : s;
    if ((e = launch_runs<T>(a, s))) return e;
    if (pl->brick && (e = launch_brick<T>(a, wall))) return e;
    if (pl->nL > 0 && (e = launch_seg_rest<T>(a, wall))) return e;
  }
  if (fork) {
    if ((e = cudaEventRecord(pl->join, pl->side))) return e;
    if ((e = cudaStreamWaitEvent(s, pl->join, 0))) return e;
  }
  return cudaSuccess;
}

template cudaError_t launch_apply<float>(const ApplyArgs<float>&, cudaStream_t);
template cudaError_t launch_apply<double>(const ApplyArgs<double>&, cudaStream_t);

}  // namespace eb
