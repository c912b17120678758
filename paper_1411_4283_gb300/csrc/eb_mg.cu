// Geometric multigrid preconditioner for the Krylov solve of kappa L phi = f.
//
// The paper preconditions GMRES with algebraic multigrid (PETSc GAMG, Sec.
// 3.2).  Here a cell-centred geometric V-cycle approximates the inverse of a
// second-order, kappa-weighted, 7-point (5-point in 2-D) operator on the same
// cut-cell grid:
//   (M phi)_v = (1/h^2) [ sum_faces alpha_f (phi_nb - phi_v) - 2 sum_walls alpha_f phi_v ] - e_v phi_v
// with alpha_f the face area fractions (Dirichlet walls half a cell away) and,
// at cut cells, e_v >= 0 chosen so that M's diagonal equals the diagonal of
// the high-order operator (the small-cell stiffness the Krylov method must
// see).  Coarse levels average kappa and the face fractions of their
// children and sum the EB terms (Galerkin scaling for piecewise-constant
// transfers); smoothing is weighted Jacobi; restriction averages the children;
// prolongation is piecewise constant.
//
// A few cut cells have a high-order diagonal that is weak (below half of the
// 7-point one), zero or positive: the row is dominated by its neighbours, the
// 7-point model is wrong there, and BiCGStab preconditioned by the V-cycle
// alone goes through long near-breakdown phases (at 256^3, 169 FP64
// iterations instead of 17).  After the V-cycle the preconditioner therefore
// solves the high-order operator exactly on the 3x3(x3) block of cells around
// each such cell (a multiplicative Schwarz step: z += A_BB^-1 (r - A z)_B,
// blocks precomputed by Gauss-Jordan in FP64).  The whole map is fixed and
// linear, so it serves as a right preconditioner of BiCGStab.
#include <cuda_runtime.h>
#include <math.h>
#include <stdint.h>

#include <algorithm>
#include <vector>

#include "eb_internal.cuh"
#include "eb_mg.cuh"
#include "eb_tables.cuh"

namespace eb {

__device__ __forceinline__ void xyz_of(int64_t c, int nx, int ny, int* x) {
  x[0] = (int)(c % nx);
  int64_t r = c / nx;
  x[1] = (int)(r % ny);
  x[2] = (int)(r / ny);
}

// Fine-level coefficients.  cpl[d][c]: coupling (1/h^2) alpha of the face between c and c + e_d;
// diag[c]: diagonal (negative on volumes, 0 on covered cells).
__global__ void k_mg_fine(int dim, int nx, int ny, int nz, double h, const uint8_t* __restrict__ flag,
                          const uint8_t* ff0, const uint8_t* ff1, const uint8_t* ff2, const int32_t* cf0,
                          const int32_t* cf1, const int32_t* cf2, const double* fm0, const double* fm1,
                          const double* fm2, int KFS, const double* __restrict__ dinv_high, float* cp0, float* cp1,
                          float* cp2, float* diag, int32_t* weak, int32_t* nweak, int cap) {
  int64_t c = (int64_t)blockIdx.x * blockDim.x + threadIdx.x;
  int64_t ncell = (int64_t)nx * ny * nz;
  if (c >= ncell) return;
  int x[3];
  xyz_of(c, nx, ny, x);
  const uint8_t* ff[3] = {ff0, ff1, ff2};
  const int32_t* cfm[3] = {cf0, cf1, cf2};
  const double* fm[3] = {fm0, fm1, fm2};
  float* cp[3] = {cp0, cp1, cp2};
  int n[3] = {nx, ny, nz};
  double ih2 = 1.0 / (h * h);
  double sum = 0.0;
  for (int d = 0; d < dim; ++d) {
    for (int side = 0; side < 2; ++side) {
      int fx[3] = {x[0], x[1], x[2]};
      if (side) fx[d] += 1;
      int64_t m0 = nx + (d == 0), m1 = ny + (d == 1);
      int64_t fl = (int64_t)fx[0] + m0 * ((int64_t)fx[1] + m1 * fx[2]);
      double a = 0.0;
      if (flag[c] > 0 && ff[d][fl] > 0) a = ff[d][fl] == 1 ? 1.0 : fm[d][(int64_t)cfm[d][fl] * KFS];
      bool wall = side ? x[d] == n[d] - 1 : x[d] == 0;
      if (wall) sum += 2.0 * a;
      else sum += a;
      if (side) cp[d][c] = (float)(wall ? 0.0 : a * ih2);
    }
  }
  if (flag[c] == 0) { diag[c] = 0.0f; return; }
  double dg = -sum * ih2;
  if (flag[c] == 2) {
    const double dh = dinv_high[c] != 0.0 ? 1.0 / dinv_high[c] : 0.0;  // diagonal of the high-order operator
    if (dh > 0.5 * dg) {             // weaker than half the 7-point diagonal, zero or positive
      const int q = atomicAdd(nweak, 1);
      if (q < cap) weak[q] = (int32_t)c;
    }
    if (dh < dg) dg = dh;            // add a non-negative EB term e_v
  }
  diag[c] = (float)dg;
}

// Coarse level from the fine level (factor 2 per dimension).  The coarse
// coupling of a face averages its 2^(D-1) fine faces and is rescaled by
// (h/H)^2; walls likewise; the EB part of the diagonal sums the children's
// with the Galerkin factor 4 / 2^D.
__global__ void k_mg_coarsen(int dim, int nxf, int nyf, int nzf, int nxc, int nyc, int nzc, const float* __restrict__ cpf0,
                             const float* __restrict__ cpf1, const float* __restrict__ cpf2,
                             const float* __restrict__ dgf, float* cpc0, float* cpc1, float* cpc2, float* dgc) {
  int64_t c = (int64_t)blockIdx.x * blockDim.x + threadIdx.x;
  int64_t ncc = (int64_t)nxc * nyc * nzc;
  if (c >= ncc) return;
  int X[3];
  xyz_of(c, nxc, nyc, X);
  int nf[3] = {nxf, nyf, nzf};
  int nc[3] = {nxc, nyc, nzc};
  const float* cpf[3] = {cpf0, cpf1, cpf2};
  float* cpc[3] = {cpc0, cpc1, cpc2};
  const int nch = 1 << dim;
  const float nfaces = (float)(1 << (dim - 1));
  // per child: couplings to in-block neighbours are internal; external ones form the coarse faces
  float ext[3][2] = {{0, 0}, {0, 0}, {0, 0}};
  float offd_f = 0.0f, dsum = 0.0f;
  int live = 0;
  for (int k = 0; k < nch; ++k) {
    int o[3] = {k & 1, (k >> 1) & 1, (k >> 2) & 1};
    int f[3];
    bool in = true;
    for (int d = 0; d < 3; ++d) {
      f[d] = d < dim ? 2 * X[d] + o[d] : 0;
      if (f[d] >= nf[d]) in = false;
    }
    if (!in) continue;
    int64_t fc = (int64_t)f[0] + (int64_t)nxf * ((int64_t)f[1] + (int64_t)nyf * f[2]);
    float dg = dgf[fc];
    if (dg == 0.0f) continue;  // covered child
    ++live;
    float offsum = 0.0f;
    for (int d = 0; d < dim; ++d) {
      // + face of the child
      float up = cpf[d][fc];
      // - face: the coupling stored on the lower neighbour
      float dn = 0.0f;
      if (f[d] > 0) {
        int g[3] = {f[0], f[1], f[2]};
        g[d] -= 1;
        dn = cpf[d][(int64_t)g[0] + (int64_t)nxf * ((int64_t)g[1] + (int64_t)nyf * g[2])];
      }
      offsum += up + dn;
      if (o[d] == 1) ext[d][1] += up;
      if (o[d] == 0) ext[d][0] += dn;
    }
    offd_f += offsum;
    dsum += dg;
  }
  if (!live) {
    dgc[c] = 0.0f;
    for (int d = 0; d < dim; ++d) cpc[d][c] = 0.0f;
    return;
  }
  // fine diagonal = -(sum of couplings + walls + EB) ; the part beyond the couplings is walls + EB
  float extra = -dsum - offd_f;       // >= 0: wall and EB terms of the children (1/h^2 units)
  const float r2 = 0.25f;             // (h/H)^2
  float cpl_sum = 0.0f;
  for (int d = 0; d < dim; ++d) {
    float up = X[d] + 1 < nc[d] ? ext[d][1] / nfaces * r2 : 0.0f;
    cpc[d][c] = up;
    float dn = X[d] > 0 ? ext[d][0] / nfaces * r2 : 0.0f;
    cpl_sum += up + dn;
    // faces on the domain boundary keep their Dirichlet weight inside `extra`
  }
  float eb = extra * 4.0f / (float)nch * r2;
  dgc[c] = -(cpl_sum + eb);
}

// sum of the couplings times the neighbours' values at cell c = p of a level; val(c, p) is a cell's value
template <typename T, int D, typename Val>
__device__ __forceinline__ T mg_offdiag(const int* n, int64_t c, const int* p, const float* cp0, const float* cp1,
                                        const float* cp2, const Val& val) {
  const float* cp[3] = {cp0, cp1, cp2};
  const int64_t st[3] = {1, n[0], (int64_t)n[0] * n[1]};
  T s = (T)0;
#pragma unroll
  for (int d = 0; d < D; ++d) {
    int q[3] = {p[0], p[1], p[2]};
    if (p[d] + 1 < n[d]) {
      q[d] = p[d] + 1;
      s += (T)__ldg(cp[d] + c) * val(c + st[d], q);
    }
    if (p[d] > 0) {
      q[d] = p[d] - 1;
      s += (T)__ldg(cp[d] + c - st[d]) * val(c - st[d], q);
    }
  }
  return s;
}

// Level kernels run on a 3-D grid of (32 x 4)-thread blocks over (x, y) rows and z planes, so that a
// thread's cell coordinates need no integer division.  The dimension is a template argument: with it at run time
// the per-direction pointers and coordinates lived in local memory.
constexpr int MG_BX = 32, MG_BY = 4;

__device__ __forceinline__ bool mg_cell(int nx, int ny, int* p, int64_t* c) {
  p[0] = blockIdx.x * MG_BX + threadIdx.x;
  p[1] = blockIdx.y * MG_BY + threadIdx.y;
  p[2] = blockIdx.z;
  if (p[0] >= nx || p[1] >= ny) return false;
  *c = (int64_t)p[0] + (int64_t)nx * ((int64_t)p[1] + (int64_t)ny * p[2]);
  return true;
}

template <typename T>
struct MgSweep {
  int n[3], nc[2];        // cells of the level; of the coarser one in x and y (MG_POST)
  const float* cp[3];
  const float* dg;
  const T* b;
  const T* x;
  const T* xc;            // the coarser level's correction (MG_POST)
  T* out;
  float w;
};

// Weighted Jacobi: out = x + w (b - M x) / diag.  A level's arrays mostly stay in L2 (128^3 in FP32: 14 us a sweep,
// the loads of seven cells' values through L1), and on the coarser levels the launch bounds a pass, so there the
// values that another pass would have written for the sweep are made on the fly:
//   MG_FIRST, MG_PROLONG   no sweep: the first one from x = 0, out = w b / diag; x + x_c (piecewise constant on volumes)
//   MG_PRE, MG_POST        those values and the sweep that follows, in one pass
// The fused passes repeat a division or two more loads for each neighbour: 6.9 and 7.1 us at 64^3 in FP32 (4.8
// for the sweep alone, before another pass and its launch), but 29 and 30 us at 128^3 (two passes: 25 and 26 us), hence the line between them.  In FP64
// the divide is a sequence on a pipe 64 times slower: an iteration of an FP64 solve takes 734 us in two passes and 741 us
// fused at 30^3, 1071 and 1090 at 40^3, 1271 and 1304 at 48^3, 2093 and 2243 at 80^3, 4201 and 4734 at 128^3, so the line lies
// where the two are within 2 %.  The level passes of a cycle at 128^3 in FP32 took 225 us in 18 launches before and
// take 133 us in 14 now, k_mg_coarse 85 and 32 us.
enum { MG_PLAIN, MG_FIRST, MG_PROLONG, MG_PRE, MG_POST };
template <typename T>
constexpr int64_t MG_FUSE_CELLS = sizeof(T) == 4 ? 1 << 20 : 1 << 16;
template <typename T, int D, int MODE>
__global__ void __launch_bounds__(MG_BX * MG_BY) k_mg_jacobi(const __grid_constant__ MgSweep<T> a) {
  int p[3];
  int64_t c;
  if (!mg_cell(a.n[0], a.n[1], p, &c)) return;
  const float d = __ldg(a.dg + c);
  if (d == 0.0f) {
    a.out[c] = (T)0;
    return;
  }
  const auto val = [&](int64_t i, const int* q) -> T {
    if (MODE == MG_PLAIN) return __ldg(a.x + i);
    const float di = __ldg(a.dg + i);
    if (MODE == MG_POST || MODE == MG_PROLONG) {
      const T v = __ldg(a.x + i);
      return di == 0.0f ? v : v + __ldg(a.xc + (q[0] >> 1) + (int64_t)a.nc[0] * ((q[1] >> 1) + (int64_t)a.nc[1] * (D == 3 ? q[2] >> 1 : 0)));
    }
    return di == 0.0f ? (T)0 : (T)a.w * __ldg(a.b + i) / (T)di;
  };
  const T v = val(c, p);
  if (MODE == MG_FIRST || MODE == MG_PROLONG) {
    a.out[c] = v;
    return;
  }
  const T r = __ldg(a.b + c) - ((T)d * v + mg_offdiag<T, D>(a.n, c, p, a.cp[0], a.cp[1], a.cp[2], val));
  a.out[c] = v + (T)a.w * r / (T)d;
}

// coarse right-hand side: average of the children's residuals b - M x.  A lane takes the children of one fine x (two
// or four, a warp thereby reads whole rows) and adds its neighbour's: with a thread per coarse cell the chain of its
// eight children's loads was the time on the coarser levels (10 us from 32^3 cells and 20 us from 128^3, 9 and 16 us now).
template <typename T, int D>
__global__ void __launch_bounds__(MG_BX * MG_BY) k_mg_restrict(const __grid_constant__ MgSweep<T> a) {
  const int fx = blockIdx.x * MG_BX + threadIdx.x, Y = blockIdx.y * MG_BY + threadIdx.y, Z = blockIdx.z;
  if (Y >= a.nc[1]) return;  // a whole warp
  const auto val = [&](int64_t i, const int*) { return __ldg(a.x + i); };
  T acc = (T)0;
#pragma unroll
  for (int k = 0; k < (1 << (D - 1)); ++k) {
    const int f[3] = {fx, 2 * Y + (k & 1), D == 3 ? 2 * Z + (k >> 1) : 0};
    if (f[0] >= a.n[0] || f[1] >= a.n[1] || (D == 3 && f[2] >= a.n[2])) continue;
    const int64_t fc = (int64_t)f[0] + (int64_t)a.n[0] * ((int64_t)f[1] + (int64_t)a.n[1] * f[2]);
    const float d = __ldg(a.dg + fc);
    if (d == 0.0f) continue;
    acc += __ldg(a.b + fc) - ((T)d * __ldg(a.x + fc) + mg_offdiag<T, D>(a.n, fc, f, a.cp[0], a.cp[1], a.cp[2], val));
  }
  acc += __shfl_down_sync(0xffffffffu, acc, 1);
  if (!(fx & 1) && fx < a.n[0])
    a.out[(fx >> 1) + (int64_t)a.nc[0] * ((int64_t)Y + (int64_t)a.nc[1] * Z)] = acc / (T)(1 << D);
}

// The levels from `l0` down, when small, in one CTA: the same V-cycle with block-wide barriers instead of kernel
// boundaries.  What bounds it is the latency of some forty dependent phases, so all levels lie in shared memory:
// right-hand side, iterate and its copy, w / diag, couplings, which neighbours exist and the parent's index; a
// level's phases are run by as many warps as it has cells for.  From global memory a phase took 2 us (16^3 in FP32:
// 85 us a cycle, 33 now).
template <typename T>
struct MgDev {
  int n[3];
  const float* cp[3];
  const float* dg;
  T* b;
  T* x;
  T* w;
};
constexpr int MG_CTA_THREADS = 1024;
template <typename T, int D>
__host__ __device__ constexpr int64_t mg_cta_bytes(int64_t cells) {  // of one level (16-byte multiple)
  return (cells * (4 * (int64_t)sizeof(T) + 4 * D + 3) + 15) / 16 * 16;
}
template <typename T, int D>
struct MgShared {
  int n[3], cells, threads;
  T *b, *x, *w, *id;
  float* cp;        // [D][cells]
  uint16_t* parent;
  uint8_t* nb;      // bit 2 d: a neighbour above in direction d, bit 2 d + 1: below
  __device__ MgShared(const MgDev<T>& L, unsigned char* at) {
    for (int d = 0; d < 3; ++d) n[d] = L.n[d];
    cells = n[0] * n[1] * n[2];
    threads = min(MG_CTA_THREADS, (cells + 31) / 32 * 32);
    b = reinterpret_cast<T*>(at);
    x = b + cells;
    w = x + cells;
    id = w + cells;
    cp = reinterpret_cast<float*>(id + cells);
    parent = reinterpret_cast<uint16_t*>(cp + D * cells);
    nb = reinterpret_cast<uint8_t*>(parent + cells);
  }
  __device__ __forceinline__ T offdiag(int c, const T* v) const {
    const int m = nb[c], st[3] = {1, n[0], n[0] * n[1]};
    T s = (T)0;
#pragma unroll
    for (int d = 0; d < D; ++d) {
      if (m >> (2 * d) & 1) s += (T)cp[d * cells + c] * v[c + st[d]];
      if (m >> (2 * d + 1) & 1) s += (T)cp[d * cells + c - st[d]] * v[c - st[d]];
    }
    return s;
  }
  __device__ __forceinline__ void sync() const {  // the level's warps
    asm volatile("bar.sync 1, %0;" ::"r"(threads) : "memory");
  }
  // x + w (b - M x) / diag = (1 - w) x + (w / diag) (b - couplings)
  __device__ void sweeps(int count, float om) {
    for (int it = 0; it < count; ++it) {
      for (int c = threadIdx.x; c < cells; c += threads)
        w[c] = id[c] == (T)0 ? (T)0 : ((T)1 - (T)om) * x[c] + id[c] * (b[c] - offdiag(c, x));
      sync();
      T* t = x;
      x = w;
      w = t;
    }
  }
};

template <typename T, int D>
__global__ void __launch_bounds__(MG_CTA_THREADS) k_mg_coarse(int nlev, const MgDev<T>* __restrict__ lev, float om, int nu,
                                                              int ncoarse) {
  extern __shared__ __align__(16) unsigned char mg_smem[];
  const int tid = threadIdx.x;
  int64_t at = 0;
  for (int l = 0; l < nlev; ++l) {
    const MgDev<T> L = lev[l];
    const MgShared<T, D> S(L, mg_smem + at);
    at += mg_cta_bytes<T, D>(S.cells);
    const int mx = (S.n[0] + 1) / 2, my = (S.n[1] + 1) / 2;
    for (int c = tid; c < S.cells; c += MG_CTA_THREADS) {
      const float d = L.dg[c];
      S.id[c] = d == 0.0f ? (T)0 : (T)om / (T)d;
      if (l == 0) S.b[c] = L.b[c];
      const int p[3] = {c % S.n[0], c / S.n[0] % S.n[1], c / (S.n[0] * S.n[1])};
      int m = 0;
#pragma unroll
      for (int k = 0; k < D; ++k) {
        S.cp[k * S.cells + c] = L.cp[k][c];
        m |= (p[k] + 1 < S.n[k]) << (2 * k) | (p[k] > 0) << (2 * k + 1);
      }
      S.nb[c] = (uint8_t)m;
      S.parent[c] = (uint16_t)((p[0] >> 1) + mx * ((p[1] >> 1) + my * (D == 3 ? p[2] >> 1 : 0)));
    }
  }
  __syncthreads();
  // descend; odd sweep counts leave a level's iterate in its other buffer (bit l of odd)
  unsigned odd = 0;
  at = 0;
  for (int l = 0; l < nlev; ++l) {
    MgShared<T, D> S(lev[l], mg_smem + at);
    const int64_t here = at;
    at += mg_cta_bytes<T, D>(S.cells);
    const bool last = l == nlev - 1;
    const int more = (last ? ncoarse : nu) - 1;
    if (tid < S.threads) {
      for (int c = tid; c < S.cells; c += S.threads) S.x[c] = S.id[c] * S.b[c];
      S.sync();
      S.sweeps(more, om);
    }
    odd |= (unsigned)(more & 1) << l;
    __syncthreads();
    if (last) break;
    const MgShared<T, D> F(lev[l], mg_smem + here), C(lev[l + 1], mg_smem + at);
    const T* x = (more & 1) ? F.w : F.x;
    const float* dg = lev[l].dg;
    for (int c = tid; c < C.cells; c += MG_CTA_THREADS) {
      const int X[3] = {c % C.n[0], c / C.n[0] % C.n[1], c / (C.n[0] * C.n[1])};
      T acc = (T)0;
#pragma unroll
      for (int k = 0; k < (1 << D); ++k) {
        const int f0 = 2 * X[0] + (k & 1), f1 = 2 * X[1] + ((k >> 1) & 1), f2 = D == 3 ? 2 * X[2] + (k >> 2) : 0;
        if (f0 >= F.n[0] || f1 >= F.n[1] || (D == 3 && f2 >= F.n[2])) continue;
        const int fc = f0 + F.n[0] * (f1 + F.n[1] * f2);
        const float d = __ldg(dg + fc);
        if (d != 0.0f) acc += F.b[fc] - ((T)d * x[fc] + F.offdiag(fc, x));
      }
      C.b[c] = acc / (T)(1 << D);
    }
    __syncthreads();
  }
  for (int l = nlev - 2; l >= 0; --l) {  // ascend
    at = 0;
    for (int k = 0; k < l; ++k) at += mg_cta_bytes<T, D>((int64_t)lev[k].n[0] * lev[k].n[1] * lev[k].n[2]);
    MgShared<T, D> S(lev[l], mg_smem + at);
    const MgShared<T, D> C(lev[l + 1], mg_smem + at + mg_cta_bytes<T, D>(S.cells));
    const T* xc = (odd >> (l + 1) & 1) ? C.w : C.x;
    if (odd >> l & 1) {
      T* t = S.x;
      S.x = S.w;
      S.w = t;
    }
    if (tid < S.threads) {
      for (int c = tid; c < S.cells; c += S.threads)
        if (S.id[c] != (T)0) S.x[c] += xc[S.parent[c]];
      S.sync();
      S.sweeps(nu, om);
    }
    odd ^= (unsigned)(nu & 1) << l;
    __syncthreads();
  }
  const MgShared<T, D> S(lev[0], mg_smem);
  const T* x = (odd & 1) ? S.w : S.x;
  for (int c = tid; c < S.cells; c += MG_CTA_THREADS) lev[0].x[c] = x[c];
}

static unsigned nb256(int64_t n) { return (unsigned)((n + 255) / 256); }

// ---------------------------------------------------------------- local block solves
constexpr int BLK = 27;  // 3 x 3 x 3 cells around a weak-diagonal cut cell
constexpr int MAX_BLOCKS = 8192;

struct RowSrc {
  const int32_t* irr_cell;
  const int32_t* irr_row;
  int64_t n_irr;
  const uint8_t* kind;
  const double* tmpl64;
  const double* rows64;
  const float* tmpl32;
  const float* rows32;
  int64_t n_rows;
  int nfoot;
  const int32_t* foot_off;
  const int16_t* lut;
  int L, S, nx, ny, nz;
  int64_t ncell;
};

// canonical row of cell c (-1: the template row, -2: covered)
__device__ int64_t row_of_cell(const RowSrc& a, int64_t c) {
  if (a.kind[c] == 0) return -2;
  if (a.kind[c] == 1) return -1;
  int64_t lo = 0, hi = a.n_irr - 1;
  while (lo < hi) {
    int64_t mid = (lo + hi) >> 1;
    if (a.irr_cell[mid] < c) lo = mid + 1;
    else hi = mid;
  }
  return a.irr_row[lo];
}

template <typename T>
__device__ __forceinline__ T coef_at(const RowSrc& a, int64_t row, int f);
template <>
__device__ __forceinline__ double coef_at<double>(const RowSrc& a, int64_t row, int f) {
  return row == -1 ? a.tmpl64[f] : a.rows64[(int64_t)f * a.n_rows + row];
}
template <>
__device__ __forceinline__ float coef_at<float>(const RowSrc& a, int64_t row, int f) {
  return row == -1 ? a.tmpl32[f] : a.rows32[(int64_t)f * a.n_rows + row];
}

// A_BB of every block (FP64); padding entries get the identity
__global__ void k_blk_assemble(RowSrc a, int nblk, const int32_t* __restrict__ cells, double* __restrict__ M) {
  const int64_t t = (int64_t)blockIdx.x * blockDim.x + threadIdx.x;
  if (t >= (int64_t)nblk * BLK * BLK) return;
  const int b = (int)(t / (BLK * BLK)), i = (int)(t / BLK % BLK), j = (int)(t % BLK);
  const int32_t ci = cells[b * BLK + i], cj = cells[b * BLK + j];
  double v = 0.0;
  if (ci < 0 || cj < 0) {
    v = i == j ? 1.0 : 0.0;
  } else {
    int xi[3], xj[3];
    xyz_of(ci, a.nx, a.ny, xi);
    xyz_of(cj, a.nx, a.ny, xj);
    const int dx = xj[0] - xi[0], dy = xj[1] - xi[1], dz = xj[2] - xi[2];
    const int f = a.lut[(dx + a.L) + a.S * ((dy + a.L) + a.S * (dz + a.L))];
    const int64_t row = row_of_cell(a, ci);
    if (f >= 0 && row != -2) v = coef_at<double>(a, row, f);
  }
  M[t] = v;
}

// in-place Gauss-Jordan inverse with partial pivoting, one thread per block
__global__ void k_blk_invert(int nblk, double* __restrict__ M, float* __restrict__ M32, int32_t* __restrict__ fail) {
  const int b = blockIdx.x * blockDim.x + threadIdx.x;
  if (b >= nblk) return;
  double a[BLK][2 * BLK];
  const double* src = M + (int64_t)b * BLK * BLK;
  for (int i = 0; i < BLK; ++i)
    for (int j = 0; j < BLK; ++j) {
      a[i][j] = src[i * BLK + j];
      a[i][BLK + j] = i == j ? 1.0 : 0.0;
    }
  for (int k = 0; k < BLK; ++k) {
    int p = k;
    for (int i = k + 1; i < BLK; ++i)
      if (fabs(a[i][k]) > fabs(a[p][k])) p = i;
    if (a[p][k] == 0.0) { atomicExch(fail, 1); return; }
    if (p != k)
      for (int j = 0; j < 2 * BLK; ++j) { double t = a[k][j]; a[k][j] = a[p][j]; a[p][j] = t; }
    const double inv = 1.0 / a[k][k];
    for (int j = 0; j < 2 * BLK; ++j) a[k][j] *= inv;
    for (int i = 0; i < BLK; ++i) {
      if (i == k) continue;
      const double m = a[i][k];
      if (m == 0.0) continue;
      for (int j = 0; j < 2 * BLK; ++j) a[i][j] -= m * a[k][j];
    }
  }
  double* dst = M + (int64_t)b * BLK * BLK;
  for (int i = 0; i < BLK; ++i)
    for (int j = 0; j < BLK; ++j) {
      dst[i * BLK + j] = a[i][BLK + j];
      M32[(int64_t)b * BLK * BLK + i * BLK + j] = (float)a[i][BLK + j];
    }
}

// res_i = r_ci - (A z)_ci for the cells of every block; one warp per cell, the lanes splitting the
// footprint (few cells, long rows: a thread per cell leaves the GPU idle behind 637 dependent loads).
// TR: the transposed operator, (A^T z)_c = sum_f A(c - off_f, f) z_(c - off_f) (the rows that reach c;
// a linear offset that wraps across a grid line lands on a row whose entry there is zero)
template <typename T, bool TR>
__global__ void k_blk_res(RowSrc a, int nblk, const int32_t* __restrict__ cells, const T* __restrict__ r,
                          const T* __restrict__ z, T* __restrict__ res) {
  const int64_t t = ((int64_t)blockIdx.x * blockDim.x + threadIdx.x) >> 5;  // warp-uniform
  const int lane = threadIdx.x & 31;
  if (t >= (int64_t)nblk * BLK) return;
  const int32_t c = cells[t];
  if (c < 0) {
    if (lane == 0) res[t] = (T)0;
    return;
  }
  const int64_t row = row_of_cell(a, c);
  if (row == -2) {
    if (lane == 0) res[t] = (T)0;
    return;
  }
  T acc = (T)0;
  const int64_t hi = a.ncell - 1;
  if (TR) {
    for (int f = lane; f < a.nfoot; f += 32) {
      const int64_t q = c - a.foot_off[f];
      if (q < 0 || q > hi) continue;
      const int64_t rq = row_of_cell(a, q);
      if (rq == -2) continue;
      acc = fma(coef_at<T>(a, rq, f), z[q], acc);
    }
  } else {
    for (int f = lane; f < a.nfoot; f += 32) {
      int64_t q = c + a.foot_off[f];
      q = q < 0 ? 0 : (q > hi ? hi : q);  // out-of-domain entries have zero coefficients
      acc = fma(coef_at<T>(a, row, f), z[q], acc);
    }
  }
#pragma unroll
  for (int o = 16; o > 0; o >>= 1) acc += __shfl_xor_sync(0xffffffffu, acc, o);
  if (lane == 0) res[t] = r[c] - acc;
}

// z_ci += sum_j inv(A_BB)_ij res_j (blocks may overlap: additive); TR: inv(A_BB^T) = inv(A_BB)^T
template <typename T, bool TR>
__global__ void k_blk_corr(int nblk, const int32_t* __restrict__ cells, const T* __restrict__ inv,
                           const T* __restrict__ res, T* z) {
  const int64_t t = (int64_t)blockIdx.x * blockDim.x + threadIdx.x;
  if (t >= (int64_t)nblk * BLK) return;
  const int32_t c = cells[t];
  if (c < 0) return;
  const int64_t b = t / BLK, i = t % BLK;
  const T* rr = res + b * BLK;
  T d = (T)0;
  if (TR) {
    const T* m = inv + b * BLK * BLK + i;
    for (int j = 0; j < BLK; ++j) d = fma(m[j * BLK], rr[j], d);
  } else {
    const T* m = inv + (b * BLK + i) * BLK;
    for (int j = 0; j < BLK; ++j) d = fma(m[j], rr[j], d);
  }
  atomicAdd(z + c, d);
}

static RowSrc row_src(const Multigrid& mg) {
  RowSrc a;
  a.irr_cell = mg.irr_cell;
  a.irr_row = mg.irr_row;
  a.n_irr = mg.n_irr;
  a.kind = mg.kind;
  a.tmpl64 = mg.tmpl64;
  a.rows64 = mg.rows64;
  a.tmpl32 = mg.tmpl32;
  a.rows32 = mg.rows32;
  a.n_rows = mg.n_rows;
  a.nfoot = mg.nfoot;
  a.foot_off = mg.foot_off;
  a.lut = mg.foot_lut;
  a.L = mg.R + 1;
  a.S = 2 * mg.R + 3;
  a.nx = mg.lev[0].n[0];
  a.ny = mg.lev[0].n[1];
  a.nz = mg.lev[0].n[2];
  a.ncell = mg.lev[0].ncell;
  return a;
}

// blocks around the weak-diagonal cut cells (3 x 3 x 3, or 3 x 3 in 2-D with the other entries padding):
// cell lists on the host, A_BB and its inverse on the device
// cells of the block around weak cell list[b]: the 3x3x3 box (in the domain, not covered), -1 elsewhere
__global__ void k_blk_cells(const int32_t* __restrict__ list, int nb, int nx, int ny, int nz,
                            const uint8_t* __restrict__ flag, int32_t* __restrict__ cells) {
  const int64_t t = (int64_t)blockIdx.x * blockDim.x + threadIdx.x;
  if (t >= (int64_t)nb * BLK) return;
  const int b = (int)(t / BLK), k = (int)(t % BLK);
  int p[3];
  xyz_of(list[b], nx, ny, p);
  const int X = p[0] + k % 3 - 1, Y = p[1] + k / 3 % 3 - 1, Z = p[2] + k / 9 - 1;
  int32_t v = -1;
  if (X >= 0 && X < nx && Y >= 0 && Y < ny && Z >= 0 && Z < nz) {
    const int64_t q = X + (int64_t)nx * (Y + (int64_t)ny * Z);
    if (flag[q]) v = (int32_t)q;
  }
  cells[t] = v;
}

static cudaError_t blocks_setup(const MgFineInput& in, Multigrid* mg, const int32_t* weak_d, const int32_t* nweak_d,
                                cudaStream_t s) {
  if (!in.irr_cell || in.n_irr == 0) return cudaSuccess;
  const int nx = in.n[0], ny = in.n[1], nz = in.n[2];
  cudaError_t e;
  int32_t nw = 0;
  if ((e = cudaMemcpyAsync(&nw, nweak_d, 4, cudaMemcpyDeviceToHost, s))) return e;
  if ((e = cudaStreamSynchronize(s))) return e;
  const int nb = nw < MAX_BLOCKS ? nw : MAX_BLOCKS;
  std::vector<int32_t> list(nb > 0 ? nb : 1);
  if (nb > 0) {
    if ((e = cudaMemcpyAsync(list.data(), weak_d, (size_t)nb * 4, cudaMemcpyDeviceToHost, s))) return e;
    if ((e = cudaStreamSynchronize(s))) return e;
    std::sort(list.begin(), list.begin() + nb);  // appended in any order: make the blocks deterministic
  }
  // row lookup data
  mg->irr_cell = in.irr_cell;
  mg->irr_row = in.irr_row;
  mg->n_irr = in.n_irr;
  mg->kind = in.kind;
  mg->tmpl64 = in.tmpl64;
  mg->tmpl32 = in.tmpl32;
  mg->rows64 = in.rows64;
  mg->rows32 = in.rows32;
  mg->n_rows = in.n_rows;
  mg->nfoot = in.nfoot;
  mg->foot_off = in.foot_off;
  mg->R = in.R;
  if (nb == 0) return cudaSuccess;
  const int L = in.R + 1, S = 2 * L + 1;
  std::vector<int16_t> lut(S * S * S, -1);
  int nf = 0;
  const int zr = in.dim == 3 ? L : 0;
  for (int z = -zr; z <= zr; ++z)
    for (int y = -L; y <= L; ++y)
      for (int x = -L; x <= L; ++x)
        if (in_footprint(x, y, z, in.R, in.box)) lut[(x + L) + S * ((y + L) + S * (z + L))] = (int16_t)nf++;
  if (nf != in.nfoot) return cudaErrorInvalidValue;
  if ((e = cudaMalloc(&mg->foot_lut, lut.size() * 2))) return e;
  if ((e = cudaMalloc(&mg->blk_cells, (size_t)nb * BLK * 4))) return e;
  if ((e = cudaMalloc(&mg->blk_inv64, (size_t)nb * BLK * BLK * 8))) return e;
  if ((e = cudaMalloc(&mg->blk_inv32, (size_t)nb * BLK * BLK * 4))) return e;
  if ((e = cudaMalloc(&mg->blk_res, (size_t)nb * BLK * 8))) return e;
  if ((e = cudaMemcpyAsync(mg->foot_lut, lut.data(), lut.size() * 2, cudaMemcpyHostToDevice, s))) return e;
  int32_t* dl;
  if ((e = cudaMalloc(&dl, (size_t)nb * 4))) return e;
  if ((e = cudaMemcpyAsync(dl, list.data(), (size_t)nb * 4, cudaMemcpyHostToDevice, s))) { cudaFree(dl); return e; }
  k_blk_cells<<<nb256((int64_t)nb * BLK), 256, 0, s>>>(dl, nb, nx, ny, nz, in.flag, mg->blk_cells);
  eb::count_launch();
  mg->nblk = nb;
  RowSrc a = row_src(*mg);
  const int64_t nm = (int64_t)nb * BLK * BLK;
  k_blk_assemble<<<nb256(nm), 256, 0, s>>>(a, nb, mg->blk_cells, mg->blk_inv64);
  int32_t* fail;
  if ((e = cudaMalloc(&fail, 4))) return e;
  cudaMemsetAsync(fail, 0, 4, s);
  k_blk_invert<<<(nb + 31) / 32, 32, 0, s>>>(nb, mg->blk_inv64, mg->blk_inv32, fail);
  eb::count_launches(2);
  int32_t hf = 0;
  cudaMemcpyAsync(&hf, fail, 4, cudaMemcpyDeviceToHost, s);
  e = cudaStreamSynchronize(s);
  cudaFree(fail);
  cudaFree(dl);
  if (e) return e;
  if (hf) mg->nblk = 0;  // a singular block: no local solves
  return cudaGetLastError();
}

static cudaError_t mg_cta_attributes() {
  const auto attr = cudaFuncAttributeMaxDynamicSharedMemorySize;
  const int bytes = 227 * 1024;
  cudaError_t e = cudaFuncSetAttribute(k_mg_coarse<float, 2>, attr, bytes);
  if (!e) e = cudaFuncSetAttribute(k_mg_coarse<float, 3>, attr, bytes);
  if (!e) e = cudaFuncSetAttribute(k_mg_coarse<double, 2>, attr, bytes);
  return e ? e : cudaFuncSetAttribute(k_mg_coarse<double, 3>, attr, bytes);
}

cudaError_t mg_setup(const MgFineInput& in, Multigrid* mg, cudaStream_t s) {
  mg->dim = in.dim;
  mg->nlev = 0;
  int32_t* weak = nullptr;  // fine-level cut cells with a weak high-order diagonal (list, count after it)
  int n[3] = {in.n[0], in.n[1], in.n[2]};
  cudaError_t e;
  for (int l = 0; l < MG_MAXLEV; ++l) {
    MgLevel& L = mg->lev[l];
    for (int d = 0; d < 3; ++d) L.n[d] = n[d];
    int64_t nc = (int64_t)n[0] * n[1] * n[2];
    L.ncell = nc;
    for (int d = 0; d < 3; ++d) {
      if ((e = cudaMalloc(&L.cp[d], nc * 4))) return e;
      if ((e = cudaMemsetAsync(L.cp[d], 0, nc * 4, s))) return e;
    }
    if ((e = cudaMalloc(&L.dg, nc * 4))) return e;
    for (int k = 0; k < 3; ++k)
      if ((e = cudaMalloc(&L.v32[k], nc * 4))) return e;
    for (int k = 0; k < 3; ++k)
      if ((e = cudaMalloc(&L.v64[k], nc * 8))) return e;
    mg->nlev = l + 1;
    if (l == 0) {
      if ((e = cudaMalloc(&weak, (MAX_BLOCKS + 1) * 4))) return e;
      if ((e = cudaMemsetAsync(weak + MAX_BLOCKS, 0, 4, s))) return e;
      k_mg_fine<<<nb256(nc), 256, 0, s>>>(in.dim, n[0], n[1], n[2], in.h, in.flag, in.ff[0], in.ff[1], in.ff[2],
                                          in.cf[0], in.cf[1], in.cf[2], in.fm[0], in.fm[1], in.fm[2], in.KFS,
                                          in.dinv_high, L.cp[0], L.cp[1], L.cp[2], L.dg, weak, weak + MAX_BLOCKS,
                                          MAX_BLOCKS);
      eb::count_launch();
    } else {
      MgLevel& F = mg->lev[l - 1];
      k_mg_coarsen<<<nb256(nc), 256, 0, s>>>(in.dim, F.n[0], F.n[1], F.n[2], n[0], n[1], n[2], F.cp[0], F.cp[1], F.cp[2],
                                             F.dg, L.cp[0], L.cp[1], L.cp[2], L.dg);
      eb::count_launch();
    }
    if ((e = cudaGetLastError())) return e;
    int mn = n[0] < n[1] ? n[0] : n[1];
    if (in.dim == 3 && n[2] < mn) mn = n[2];
    if (mn <= 4) break;
    for (int d = 0; d < in.dim; ++d) n[d] = (n[d] + 1) / 2;
  }
  if (weak) {
    e = blocks_setup(in, mg, weak, weak + MAX_BLOCKS, s);
    cudaFree(weak);
    if (e) return e;
  }
  // device descriptors of every level for the single-CTA coarse cycle
  MgDev<float> h32[MG_MAXLEV];
  MgDev<double> h64[MG_MAXLEV];
  for (int l = 0; l < mg->nlev; ++l) {
    MgLevel& L = mg->lev[l];
    for (int d = 0; d < 3; ++d) { h32[l].n[d] = L.n[d]; h64[l].n[d] = L.n[d]; h32[l].cp[d] = L.cp[d]; h64[l].cp[d] = L.cp[d]; }
    h32[l].dg = L.dg; h64[l].dg = L.dg;
    h32[l].b = L.v32[0]; h32[l].x = L.v32[1]; h32[l].w = L.v32[2];
    h64[l].b = L.v64[0]; h64[l].x = L.v64[1]; h64[l].w = L.v64[2];
  }
  if ((e = mg_cta_attributes())) return e;
  if ((e = cudaMalloc(&mg->dev32, sizeof(h32)))) return e;
  if ((e = cudaMalloc(&mg->dev64, sizeof(h64)))) return e;
  if ((e = cudaMemcpyAsync(mg->dev32, h32, sizeof(h32), cudaMemcpyHostToDevice, s))) return e;
  if ((e = cudaMemcpyAsync(mg->dev64, h64, sizeof(h64), cudaMemcpyHostToDevice, s))) return e;
  return cudaStreamSynchronize(s);
}

void mg_free(Multigrid* mg) {
  cudaFree(mg->blk_cells);
  cudaFree(mg->blk_inv64);
  cudaFree(mg->blk_inv32);
  cudaFree(mg->blk_res);
  cudaFree(mg->foot_lut);
  mg->blk_cells = nullptr;
  mg->blk_inv64 = nullptr;
  mg->blk_inv32 = nullptr;
  mg->blk_res = nullptr;
  mg->foot_lut = nullptr;
  mg->nblk = 0;
  if (mg->dev32) cudaFree(mg->dev32);
  if (mg->dev64) cudaFree(mg->dev64);
  mg->dev32 = mg->dev64 = nullptr;
  for (int k = 0; k < 2; ++k)
    if (mg->exec[k]) { cudaGraphExecDestroy(mg->exec[k]); mg->exec[k] = nullptr; }
  for (int l = 0; l < mg->nlev; ++l) {
    MgLevel& L = mg->lev[l];
    for (int d = 0; d < 3; ++d) cudaFree(L.cp[d]);
    cudaFree(L.dg);
    for (int k = 0; k < 3; ++k) {
      cudaFree(L.v32[k]);
      cudaFree(L.v64[k]);
    }
  }
  mg->nlev = 0;
}

template <typename T>
static T* vbuf(MgLevel& L, int k);
template <>
float* vbuf<float>(MgLevel& L, int k) { return L.v32[k]; }
template <>
double* vbuf<double>(MgLevel& L, int k) { return L.v64[k]; }

// z = V(b) on level l; b and z live in the level's buffers (0: b, 1: x, 2: work)
constexpr int64_t MG_CTA_CELLS = 4096;            // levels at most this large run inside one CTA ...
constexpr int64_t MG_CTA_SMEM = 227 * 1024;       // ... if they and the coarser ones fit its shared memory

// shared memory of the levels from l down (MG_CTA_SMEM + 1: not in one CTA)
template <typename T, int D>
static int64_t mg_cta_smem(const Multigrid& mg, int l) {
  if (mg.lev[l].ncell > MG_CTA_CELLS) return MG_CTA_SMEM + 1;
  int64_t bytes = 0;
  for (int k = l; k < mg.nlev; ++k) bytes += mg_cta_bytes<T, D>(mg.lev[k].ncell);
  return bytes;
}

static dim3 mg_grid(const int* n) {
  return dim3((unsigned)((n[0] + MG_BX - 1) / MG_BX), (unsigned)((n[1] + MG_BY - 1) / MG_BY), (unsigned)n[2]);
}

template <typename T, int D>
static cudaError_t vcycle(const Multigrid& mgc, int l, cudaStream_t s) {
  Multigrid& mg = const_cast<Multigrid&>(mgc);
  MgLevel& L = mg.lev[l];
  const float om = 0.8f;
  const int64_t smem = mg_cta_smem<T, D>(mg, l);
  if (smem <= MG_CTA_SMEM) {
    MgDev<T>* dev = sizeof(T) == 4 ? (MgDev<T>*)mg.dev32 : (MgDev<T>*)mg.dev64;
    k_mg_coarse<T, D><<<1, MG_CTA_THREADS, smem, s>>>(mg.nlev - l, dev + l, om, MG_NU, 24);
    eb::count_launch();
    return cudaGetLastError();
  }
  static_assert(MG_NU >= 2, "MG_PRE makes two sweeps");
  const bool coarsest = l == mg.nlev - 1;
  const int pre = coarsest ? 24 : MG_NU, post = coarsest ? 0 : MG_NU;
  const bool fuse = L.ncell <= MG_FUSE_CELLS<T>;
  const int first = fuse ? 2 : 1;  // sweeps of the first kernel
  // the level's result ends in buffer 1: the first kernel writes buffer 1 or 2 by the parity of the passes that
  // follow it
  const bool even = (pre - first + post + (coarsest || fuse ? 0 : 1)) % 2 == 0;
  T* x = vbuf<T>(L, even ? 1 : 2);
  T* w = vbuf<T>(L, even ? 2 : 1);
  const dim3 blk(MG_BX, MG_BY), grd = mg_grid(L.n);
  MgSweep<T> a;
  for (int d = 0; d < 3; ++d) {
    a.n[d] = L.n[d];
    a.cp[d] = L.cp[d];
  }
  a.nc[0] = a.nc[1] = 0;
  a.dg = L.dg;
  a.b = vbuf<T>(L, 0);
  a.x = a.xc = nullptr;
  a.out = x;
  a.w = om;
  if (fuse) k_mg_jacobi<T, D, MG_PRE><<<grd, blk, 0, s>>>(a);
  else k_mg_jacobi<T, D, MG_FIRST><<<grd, blk, 0, s>>>(a);
  eb::count_launch();
  const auto pass = [&](int mode) {
    a.x = x;
    a.out = w;
    if (mode == MG_POST) k_mg_jacobi<T, D, MG_POST><<<grd, blk, 0, s>>>(a);
    else if (mode == MG_PROLONG) k_mg_jacobi<T, D, MG_PROLONG><<<grd, blk, 0, s>>>(a);
    else k_mg_jacobi<T, D, MG_PLAIN><<<grd, blk, 0, s>>>(a);
    eb::count_launch();
    T* t = x;
    x = w;
    w = t;
  };
  for (int it = first; it < pre; ++it) pass(MG_PLAIN);
  if (!coarsest) {
    MgLevel& C = mg.lev[l + 1];
    a.nc[0] = C.n[0];
    a.nc[1] = C.n[1];
    a.x = x;
    a.out = vbuf<T>(C, 0);
    const int rows[3] = {L.n[0], C.n[1], C.n[2]};
    k_mg_restrict<T, D><<<mg_grid(rows), blk, 0, s>>>(a);
    eb::count_launch();
    const cudaError_t e = vcycle<T, D>(mg, l + 1, s);
    if (e) return e;
    a.xc = vbuf<T>(C, 1);
    pass(fuse ? MG_POST : MG_PROLONG);
    for (int it = fuse ? 1 : 0; it < post; ++it) pass(MG_PLAIN);
  }
  if (x != vbuf<T>(L, 1)) return cudaErrorUnknown;  // parity bookkeeping above
  return cudaGetLastError();
}

template <typename T>
static cudaError_t vcycle(const Multigrid& mg, cudaStream_t s) {
  return mg.dim == 3 ? vcycle<T, 3>(mg, 0, s) : vcycle<T, 2>(mg, 0, s);
}

// The V-cycle works on the levels' fixed buffers, so it is captured once per
// precision as a CUDA graph (on a private stream) and replayed; the input and
// output copies stay outside the graph.
template <typename T>
cudaError_t mg_precond(const Multigrid& mgc, const T* r, T* z, cudaStream_t s) {
  Multigrid& mg = const_cast<Multigrid&>(mgc);
  MgLevel& L = mg.lev[0];
  const int k = sizeof(T) == 4 ? 0 : 1;
  cudaError_t e;
  cudaStreamCaptureStatus cst = cudaStreamCaptureStatusNone;
  if ((e = cudaStreamIsCapturing(s, &cst))) return e;
  const bool capturing = cst == cudaStreamCaptureStatusActive;  // inside a graph being captured: the cycle's kernels
  if (!capturing && !mg.exec[k]) {
    cudaStream_t cap;
    if ((e = cudaStreamCreateWithFlags(&cap, cudaStreamNonBlocking))) return e;
    long long before = eb::launches_so_far();
    if ((e = cudaStreamBeginCapture(cap, cudaStreamCaptureModeThreadLocal))) { cudaStreamDestroy(cap); return e; }
    cudaError_t ev = vcycle<T>(mg, cap);
    cudaGraph_t graph = nullptr;
    e = cudaStreamEndCapture(cap, &graph);
    cudaStreamDestroy(cap);
    if (ev) return ev;
    if (e) return e;
    mg.nodes[k] = eb::launches_so_far() - before;
    eb::uncount_launches(mg.nodes[k]);  // capture issued no work
    e = cudaGraphInstantiate(&mg.exec[k], graph, 0);
    cudaGraphDestroy(graph);
    if (e) return e;
  }
  if ((e = cudaMemcpyAsync(vbuf<T>(L, 0), r, L.ncell * sizeof(T), cudaMemcpyDeviceToDevice, s))) return e;
  if (capturing) {
    if ((e = vcycle<T>(mg, s))) return e;
  } else {
    if ((e = cudaGraphLaunch(mg.exec[k], s))) return e;
    eb::count_launches(mg.nodes[k]);
  }
  if ((e = cudaMemcpyAsync(z, vbuf<T>(L, 1), L.ncell * sizeof(T), cudaMemcpyDeviceToDevice, s))) return e;
  if (mg.nblk > 0) {
    RowSrc a = row_src(mg);
    const int64_t nt = (int64_t)mg.nblk * BLK;
    const T* inv;
    if constexpr (sizeof(T) == 4) inv = mg.blk_inv32;
    else inv = mg.blk_inv64;
    if (mg.transpose) {
      k_blk_res<T, true><<<nb256(nt * 32), 256, 0, s>>>(a, mg.nblk, mg.blk_cells, r, z, (T*)mg.blk_res);
      k_blk_corr<T, true><<<nb256(nt), 256, 0, s>>>(mg.nblk, mg.blk_cells, inv, (const T*)mg.blk_res, z);
    } else {
      k_blk_res<T, false><<<nb256(nt * 32), 256, 0, s>>>(a, mg.nblk, mg.blk_cells, r, z, (T*)mg.blk_res);
      k_blk_corr<T, false><<<nb256(nt), 256, 0, s>>>(mg.nblk, mg.blk_cells, inv, (const T*)mg.blk_res, z);
    }
    eb::count_launches(2);
  }
  return cudaGetLastError();
}

template cudaError_t mg_precond<float>(const Multigrid&, const float*, float*, cudaStream_t);
template cudaError_t mg_precond<double>(const Multigrid&, const double*, double*, cudaStream_t);

}  // namespace eb
