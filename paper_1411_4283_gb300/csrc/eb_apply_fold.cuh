// Template pass of the operator apply (Sec. 2.3) for the interior cells in
// 3-D, with the template row folded by its reflection symmetry.
//
// The interior cell row is the sum of the six interior face stencils, so it is
// even in each of dx, dy, dz (to rounding in the LS solves; the plan averages
// the eight sign images and checks that they agree).  With
// T(a, b, c) = c(+-a, +-b, +-c) and the folds S_z^c f = f(z+c) + f(z-c)
// (S^0 f = f), the apply is
//     y(x, y, z) = sum_{a,b,c >= 0} T(a,b,c) S_x^a S_y^b S_z^c phi,
// evaluated in two passes per output plane z (the a-sum last):
//   stage 1: for every staged x (tile plus halo) and the tile's y,
//            U_a(x, y) = sum_{b,c} T(a,b,c) S_y^b S_z^c phi(x, ., .)
//            -- a thread owns one staged x column and four consecutive y:
//            it folds the planes z+-c (P_c), then the rows y+-b of P_c,
//            and accumulates the five U_a, which go to shared memory;
//   stage 2: y(x, y) = U_0(x) + sum_{a >= 1} (U_a(x+a) + U_a(x-a)).
// Against the z-folded pass (357 FMAs per cell for R = 3) this takes about
// 126 FMAs and 36 adds per cell: one FMA per term of the folded footprint
// (112 terms T(a, b, c) for R = 3) per staged column (72 staged columns per
// 64 cells), the fold adds, and in stage 2 nine loads and eight adds.
//
// Only the staged columns that an output of the tile needs and only the groups
// of four rows with a template cell (act, fixed with the cell kinds) are worked
// on: covered cells, wall layers, the neighbourhood of the EB and the rest of a
// ragged last tile cost no arithmetic, which in FP64 is what bounds the pass
// (1.66 ms at 160^3, 1.51 ms now; FP32 at 100^3 42 us, as before).
//
// Data movement is that of the z-folded pass: a ring of 2L+2 staged planes
// (64 + 8 by 16 + 2L) filled one plane ahead, by TMA with bounded mbarrier
// waits (every CTA leaves its item loop together when a wait gives up), or,
// where the length of a row of phi is not a multiple of 16 bytes, by
// asynchronous copies of single values (before, the general template pass ran
// there: FP32 132 us at 101^3 and 981 us at 201^3, 47 and 204 us now; FP64 779
// and 694 us at 101^3).  Which of the two such a grid takes, and in pieces of how
// many planes, is fold_plan's (eb_apply.cu).
#pragma once
#include <cuda.h>
#include <cuda_runtime.h>
#include <stdint.h>

#include "eb_apply_tma.cuh"

namespace eb {

constexpr int FD_OX = 64;                    // tile width (x)
constexpr int FD_OY = 16;                    // tile height (y)
constexpr int FD_PX = FD_OX + 2 * TT_XH;     // staged x (halo TT_XH, 16-byte aligned TMA boxes)
constexpr int FD_YB = 4;                     // outputs per thread along y in stage 1
constexpr int FD_T1 = FD_PX * (FD_OY / FD_YB);  // stage-1 tasks: one per (staged x, y group) = 288
constexpr int FD_THREADS = FD_T1;

template <typename T, int R>
struct FoldCoef {
  static constexpr int L = R + 1;
  T c[(L + 1) * (L + 1) * (L + 1)];  // T(a, b, c) at a + (L+1) (b + (L+1) c)
};

// one value of phi into shared memory, zero outside the grid
template <typename T>
__device__ __forceinline__ void copy_async(T* dst, const T* src, bool in) {
  asm volatile("cp.async.ca.shared.global [%0], [%1], %2, %3;" ::"r"(smem_u32(dst)), "l"(src), "n"(sizeof(T)),
               "r"(in ? (int)sizeof(T) : 0)
               : "memory");
}

template <typename T, int R, bool TMA>
__global__ void __launch_bounds__(FD_THREADS) k_apply_fold(const __grid_constant__ CUtensorMap tmap,
                                                          const __grid_constant__ FoldCoef<T, R> cf, TmplArgs<T> a,
                                                          const T* __restrict__ phi, const uint8_t* __restrict__ act) {
  constexpr int L = R + 1;
  constexpr int S = 2 * L + 1;
  constexpr int NP = S + 1;  // ring: planes z-L .. z+L and the one requested ahead
  constexpr int PY = FD_OY + 2 * L;
  constexpr uint32_t PBYTES = FD_PX * PY * sizeof(T);
  constexpr int PLANE = (int)(((PBYTES + 127) / 128) * 128 / sizeof(T));
  constexpr int NR = FD_YB + 2 * L;      // staged rows a stage-1 thread reads
  constexpr int UPL = FD_OY * FD_PX;     // one U_a plane
  static_assert(L <= TT_XH && FD_THREADS == 4 * FD_PX, "x halo, copies by columns");
  extern __shared__ __align__(128) unsigned char sm_fold[];
  T* ring = reinterpret_cast<T*>(sm_fold);
  T* U = ring + (size_t)NP * PLANE;      // [L+1][FD_OY][FD_PX]
  uint64_t* bars = reinterpret_cast<uint64_t*>(U + (size_t)(L + 1) * UPL);
  const int tid = threadIdx.x;
  if (TMA && tid == 0) {
    for (int p = 0; p < NP; ++p) mbar_init(&bars[p], 1);
    asm volatile("fence.mbarrier_init.release.cluster;" ::: "memory");
  }
  __syncthreads();
  uint32_t parity = 0, pending = 0;
  bool failed = false;
  for (int64_t item = blockIdx.x; item < a.items; item += gridDim.x) {
    const int zc = (int)(item % a.nzc);
    const int64_t t2 = item / a.nzc;
    const int tyl = (int)(t2 % a.nty), txl = (int)(t2 / a.nty);
    const int x0 = txl * FD_OX, y0 = tyl * FD_OY;
    const int z0 = zc * a.zchunk;
    const int z1 = min(z0 + a.zchunk, a.nz);
    const int ncol = min(FD_PX, a.nx - x0 + 2 * TT_XH);  // staged columns an output of this tile needs
    // the tile's row groups with template cells, per plane: bit g of the nibble
    const int64_t zstride = (int64_t)a.nty * (FD_OY / FD_YB) * a.ntx;
    const uint8_t* ap = act + (int64_t)tyl * (FD_OY / FD_YB) * a.ntx + txl;
    auto groups = [&](int z) {
      uint32_t m = 0;
#pragma unroll
      for (int g = 0; g < FD_OY / FD_YB; ++g) m |= (uint32_t)ap[z * zstride + g * a.ntx] << g;
      return m;
    };
    // plane zz by copies: the thread's column tid % FD_PX, every fourth row
    auto copy_plane = [&](int zz) {
      const int slot = ((zz % NP) + NP) % NP;
      const int gx = x0 - TT_XH + tid % FD_PX;
      const bool inxz = (unsigned)gx < (unsigned)a.nx && (unsigned)zz < (unsigned)a.nz;
      T* dst = ring + (size_t)slot * PLANE + tid;
#pragma unroll
      for (int k = 0; k < (PY + 3) / 4; ++k) {  // FD_THREADS / FD_PX = 4 rows at a time
        const int row = tid / FD_PX + 4 * k, gy = y0 - L + row;
        if (row >= PY) break;
        const bool in = inxz && (unsigned)gy < (unsigned)a.ny;
        copy_async(dst + k * FD_THREADS, in ? phi + (gx + (int64_t)a.nx * (gy + (int64_t)a.ny * zz)) : phi, in);
      }
    };
    if constexpr (TMA) {
      if (tid == 0) {
        asm volatile("fence.proxy.async.shared::cta;" ::: "memory");
        for (int q = 0; q < S; ++q) {
          const int zz = z0 - L + q, slot = ((zz % NP) + NP) % NP;
          mbar_expect_tx(&bars[slot], PBYTES);
          tma_load_3d(ring + (size_t)slot * PLANE, &tmap, &bars[slot], x0 - TT_XH, y0 - L, zz);
        }
      }
      for (int q = 0; q < S; ++q) pending |= 1u << (((z0 - L + q) % NP + NP) % NP);
      for (int q = 0; q < S; ++q) {
        const int slot = (((z0 - L + q) % NP) + NP) % NP;
        if (!mbar_wait(&bars[slot], (parity >> slot) & 1u)) { failed = true; break; }
        parity ^= 1u << slot;
        pending &= ~(1u << slot);
      }
    } else {
      for (int q = 0; q < S; ++q) copy_plane(z0 - L + q);
      asm volatile("cp.async.wait_all;" ::: "memory");
    }
    if (__syncthreads_or(failed)) { failed = true; break; }
    uint32_t gm = groups(z0), gm_next = 0;
    for (int z = z0; z < z1; ++z, gm = gm_next) {
      if (z + 1 < z1) gm_next = groups(z + 1);
      if (!TMA && z + 1 < z1) copy_plane(z + L + 1);
      if (TMA && z + 1 < z1) {
        const int zz = z + L + 1, slot = (zz % NP + NP) % NP;
        if (tid == 0) {
          asm volatile("fence.proxy.async.shared::cta;" ::: "memory");
          mbar_expect_tx(&bars[slot], PBYTES);
          tma_load_3d(ring + (size_t)slot * PLANE, &tmap, &bars[slot], x0 - TT_XH, y0 - L, zz);
        }
        pending |= 1u << slot;
      }
      if (TMA && z > z0) {
        const int slot = ((z + L) % NP + NP) % NP;
        if (mbar_wait(&bars[slot], (parity >> slot) & 1u)) {
          parity ^= 1u << slot;
          pending &= ~(1u << slot);
        } else {
          failed = true;  // acted on at the barrier that ends this step, uniformly
        }
      }
      // kinds of this thread's stage-2 cells, loaded now so that their latency hides behind stage 1
      uint8_t kd[FD_OY / 4];
      if (tid < FD_OX * 4) {
        const int xg = x0 + tid % FD_OX;
#pragma unroll
        for (int m = 0; m < FD_OY / 4; ++m) {
          const int yg2 = y0 + tid / FD_OX + 4 * m;
          kd[m] = (xg < a.nx && yg2 < a.ny) ? a.kind[xg + (int64_t)a.nx * ((int64_t)yg2 + (int64_t)a.ny * z)] : 2;
        }
      }
      // ring slot of plane z - L (one modulo per step; the others follow by a wrapped increment)
      const int s0 = ((z - L) % NP + NP) % NP;
      // ---- stage 1: U_a(xs, yg + j) for j < FD_YB, one thread per needed column of each active group
      const int gi = (tid >= ncol) + (tid >= 2 * ncol) + (tid >= 3 * ncol);
      if (tid < __popc(gm) * ncol) {
        const int xs = tid - gi * ncol;
        uint32_t m = gm;  // the gi-th active group
        for (int g = 0; g < gi; ++g) m &= m - 1;
        const int yg = (__ffs(m) - 1) * FD_YB;
        T u[L + 1][FD_YB];
#pragma unroll
        for (int q = 0; q <= L; ++q)
#pragma unroll
          for (int j = 0; j < FD_YB; ++j) u[q][j] = (T)0;
#pragma unroll
        for (int c = 0; c <= L; ++c) {
          int sp = s0 + L + c, sm = s0 + L - c;
          sp -= sp >= NP ? NP : 0;
          sm -= sm >= NP ? NP : 0;
          const T* pp = ring + (size_t)sp * PLANE + yg * FD_PX + xs;
          const T* pm = ring + (size_t)sm * PLANE + yg * FD_PX + xs;
          T p[NR];
#pragma unroll
          for (int r = 0; r < NR; ++r) p[r] = c == 0 ? pp[r * FD_PX] : pp[r * FD_PX] + pm[r * FD_PX];
#pragma unroll
          for (int b = 0; b <= L; ++b) {
#pragma unroll
            for (int j = 0; j < FD_YB; ++j) {
              const T q = b == 0 ? p[j + L] : p[j + L + b] + p[j + L - b];
#pragma unroll
              for (int aa = 0; aa <= L; ++aa) {
                if (!fp_box(aa, b, c, R)) continue;
                u[aa][j] = fma(cf.c[aa + (L + 1) * (b + (L + 1) * c)], q, u[aa][j]);
              }
            }
          }
        }
#pragma unroll
        for (int aa = 0; aa <= L; ++aa)
#pragma unroll
          for (int j = 0; j < FD_YB; ++j) U[aa * UPL + (yg + j) * FD_PX + xs] = u[aa][j];
      }
      __syncthreads();
      // ---- stage 2: x fold and the epilogue; thread: x = tid % FD_OX, rows (tid / FD_OX) + 4 m
      if (tid < FD_OX * 4) {
        const int ox = tid % FD_OX, oy0 = tid / FD_OX;
        const int xg = x0 + ox;
#pragma unroll
        for (int m = 0; m < FD_OY / 4; ++m) {
          const int oy = oy0 + 4 * m;
          const int yg2 = y0 + oy;
          const uint8_t k = kd[m];  // 2 (leave alone) outside the grid
          const int64_t c = xg + (int64_t)a.nx * ((int64_t)yg2 + (int64_t)a.ny * z);
          if (k == 1) {
            const T* ur = U + oy * FD_PX + ox + TT_XH;
            T acc = ur[0];
#pragma unroll
            for (int aa = 1; aa <= L; ++aa) acc += ur[aa * UPL + aa] + ur[aa * UPL - aa];
            a.y[c] = a.kappa_weighted ? acc : acc * (T)a.inv_kappa[c];
          } else if (k == 0) {
            a.y[c] = (T)0;
          }
        }
      }
      if (!TMA) asm volatile("cp.async.wait_all;" ::: "memory");
      // every thread is done with plane z - L and with U; a wait that gave up on any thread ends the CTA's work
      if (__syncthreads_or(failed)) { failed = true; break; }
    }
    if (failed) break;
  }
  if (TMA && failed) {
    for (int p = 0; p < NP; ++p)
      if ((pending >> p) & 1u) mbar_wait(&bars[p], (parity >> p) & 1u);
    if (tid == 0) atomicExch(a.err, 1);
  }
}

template <typename T, int R>
constexpr size_t fold_smem() {
  constexpr int L = R + 1;
  constexpr int NP = 2 * L + 2;
  constexpr size_t SLOT = ((FD_PX * (FD_OY + 2 * L) * sizeof(T) + 127) / 128) * 128;
  return NP * SLOT + (size_t)(L + 1) * FD_OY * FD_PX * sizeof(T) + NP * 8;
}

}  // namespace eb
