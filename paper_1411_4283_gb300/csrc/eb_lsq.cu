// The weighted least squares of Sec. 2.2.1, mixed path (EB_LS_MIXED): s = W t with t the least-||t|| solution
// of B^T t = F, B = W A, for every system of a build or of a batch of builds.
//
// Per system (n rows, K unknowns), by a group of W warps:
//   rows    a row of a full cell depends on its offset only and is read from a table; the rows of cut cells,
//           EB faces and walls are shifted to x0 in FP64 (registers, Horner's scheme) into a scratch array;
//   factor  R of B = Q R in FP32 by modified Gram-Schmidt, B held in registers (warp h of the group owns the
//           columns j = h mod W, a lane the rows = lane mod 32): per step the owner posts its column, every
//           warp dots it with its later columns and with itself and updates them, so that neither a square
//           root nor a division is on the way to the next step; then M = R^-1 explicitly, so that a solve
//           with R^T R is two small products instead of 2 K dependent steps;
//   t       z = M M^T F, then t = B z and r = F - B^T t in FP64: the only two FP64 passes over the rows;
//   refine  z = M M^T r, dt = B z, t += dt, r -= B^T dt, with B as the sum of two FP32 numbers and
//           compensated FP32 sums (about 2^-45), until dt is at rounding level.  The first correction is about
//           cond(B) 2^-24 of t, so an error of 2^-45 of it is far below the error 2^-53 cond(B) that the FP64
//           passes leave; where the first one is larger than MIX_DF_MAX the pass is repeated in FP64 instead.
//           The size of a correction is known before it is made (||M^T r||), and with the last one's size the
//           rate: a correction after which none is needed skips r, and is plain FP32 if it is below MIX_F32_MAX.
// A system whose factor is too ill-conditioned, or whose corrections do not settle, gets status 3 and is
// solved by the FP64 kernel (k_lsq), which also makes the rank test.
//
// What bounds it: in the end FP64 issue (two DFMA a clock and SM), so the FP64 work is cut to 4 n K flops and
// the shifts of the rows that need one; FP32 products are 64 times cheaper on this part, which pays for 11 of
// them in place of one DFMA.  As it stands the FP64 pipe is 40 % busy and the rest is the latency of the serial
// parts (factor 27 %, row lists and shifts 25 % of a block's time) that two blocks per SM do not hide: the matrix
// in registers takes all 255 of them and spills 528 bytes a thread as it is (the batch form 600), and three blocks, with
// more spills, measured the same.  90,201 systems of the 48^3 box minus a sphere (n = 396 on average, K = 35): 22.4 ms;
// the kernel before it (FP32 Householder with the chunk in shared memory, FP64 corrections: 4 n K (1 + 3.1) FP64 flops,
// 35 lanes of 64 in B^T t) 71.3 ms.
// Error against 64 bits on the same moment tables (2-norm of operator and boundary part on rough data), in brackets
// of the kernel before and of the FP64 kernel: 63^3 box minus a sphere 4.1e-15 and 1.2e-14 (6.4e-15 and 2.6e-14; 3.2e-15
// and 1.1e-14), Neumann data inside a sphere at 60^3 1.35e-15 and 1.17e-13 (1.32e-15 and 1.16e-13; 1.44e-15 and
// 1.17e-13), second order at 97^3 6.2e-16 and 2.9e-15 (1.0e-15 and 5.5e-15; 7.0e-16 and 2.9e-15).
#include <cuda_runtime.h>
#include <math.h>
#include <stdint.h>

#include <algorithm>

#include "eb_build.cuh"
#include "eb_grid.cuh"
#include "eb_internal.cuh"
#include "eb_tables.cuh"

namespace eb {

constexpr int MIX_MAX_CORR = 8;             // corrections
constexpr float MIX_TOL = 1e-14f;           // converged: the correction moved t by at most this (2-norm, relative)
constexpr float MIX_NEXT = 1e-16f;          // ... or the next one, by the rate of the last two, would by at most this
// a correction above this is made in FP64 (2^-45 of it would show: of quartics' Neumann systems, whose first correction is
// often larger than 1e-4, 5e-4 took the operator's error at 60^3 inside a sphere from 1.35e-15 to 1.43e-15)
template <int Q>
constexpr float MIX_DF_MAX = Q == 4 ? 1e-4f : 5e-4f;
constexpr float MIX_F32_MAX = 1e-10f;       // the last correction is made in plain FP32 below this
constexpr float MIX_MIN_DIAG = 2e-5f;       // min |R_kk| below this times the largest: the FP64 kernel

// f(integral constants 0 .. N-1): a loop whose body's array indices are constants whatever its size
template <int I>
struct Int {
  static constexpr int value = I;
};
template <int N, int I = 0, typename F>
__device__ __forceinline__ void static_for(F&& f) {
  if constexpr (I < N) {
    f(Int<I>{});
    static_for<N, I + 1>(f);
  }
}

// ---------------------------------------------------------------- monomials and the shift, in registers
template <int DIM, int Q>
struct Mono {
  static constexpr int K = DIM == 2 ? (Q + 1) * (Q + 2) / 2 : (Q + 1) * (Q + 2) * (Q + 3) / 6;
  // graded index of the monomial with exponent p along d and (a, b) along the others (ascending)
  __device__ static constexpr int at(int d, int p, int a, int b) {
    const int p0 = d == 0 ? p : a, p1 = d == 1 ? p : (d == 0 ? a : b), p2 = d == 2 ? p : b;
    const int g = DIM == 2 ? p0 + p1 : p0 + p1 + p2, l = g - p0;
    return DIM == 2 ? g * (g + 1) / 2 + p1 : g * (g + 1) * (g + 2) / 6 + l * (l + 1) / 2 + p2;
  }
};

// moments of (x + delta)^p from those of x^p, one dimension at a time (see shift_moments)
template <int DIM, int Q>
__device__ __forceinline__ void shift_regs(double (&m)[Mono<DIM, Q>::K], const double (&delta)[3]) {
  static_for<DIM>([&](auto dim) {
    constexpr int d = decltype(dim)::value;
    const double dl = delta[d];
    if (dl != 0.0) {
      static_for<Q + 1>([&](auto first) {
        static_for<DIM == 2 ? 1 : Q + 1 - decltype(first)::value>([&](auto second) {
          constexpr int a = decltype(first)::value, b = decltype(second)::value;
#pragma unroll
          for (int i = 1; i <= Q - a - b; ++i)
#pragma unroll
            for (int j = Q - a - b; j >= i; --j)
              m[Mono<DIM, Q>::at(d, j, a, b)] =
                  fma(dl, m[Mono<DIM, Q>::at(d, j - 1, a, b)], m[Mono<DIM, Q>::at(d, j, a, b)]);
        });
      });
    }
  });
}

// v = h + l up to 2^-46 |v| on the integer pipe (a conversion costs as much as an FP64 operation): h takes the
// leading 24 bits, l the next 23; below FP32's range both are zero
__device__ __forceinline__ void split_bits(double v, float* h, float* l) {
  const uint32_t H = (uint32_t)__double2hiint(v), L = (uint32_t)__double2loint(v);
  const uint32_t e = H & 0x7ff00000u, sg = H & 0x80000000u;
  const uint32_t t = (H & 0x7fffffffu) - 0x38000000u;  // exponent rebased from 1023 to 127
  *h = e > 0x38000000u ? __uint_as_float(sg | __funnelshift_l(L, t, 3)) : 0.0f;
  const uint32_t base = ((e - 0x38000000u) << 3) - (23u << 23);  // 2^(exponent - 23)
  const float lo = __uint_as_float(sg | base | ((L & 0x1fffffffu) >> 6)) - __uint_as_float(sg | base);
  *l = e > 0x38000000u + (24u << 20) ? lo : 0.0f;
}

// ---------------------------------------------------------------- sums over a warp
__host__ __device__ constexpr int pow2_above(int n) { return n <= 1 ? 1 : 2 * pow2_above((n + 1) / 2); }

struct PairF {  // unevaluated sum of two FP32 numbers
  float s, c;
};
// (the _rn forms: a product contracted into one of these sums would void them)
__device__ __forceinline__ void two_sum(float& s, float& c, float p) {
  const float t = __fadd_rn(s, p), b = __fsub_rn(t, s);
  c = __fadd_rn(c, __fadd_rn(__fsub_rn(s, __fsub_rn(t, b)), __fsub_rn(p, b)));
  s = t;
}
__device__ __forceinline__ double add(double a, double b) { return a + b; }
__device__ __forceinline__ float add(float a, float b) { return a + b; }
__device__ __forceinline__ PairF add(PairF a, PairF b) {
  two_sum(a.s, a.c, b.s);
  a.c += b.c;
  return a;
}
__device__ __forceinline__ double xchg(double v, int o) { return __shfl_xor_sync(0xffffffffu, v, o); }
__device__ __forceinline__ float xchg(float v, int o) { return __shfl_xor_sync(0xffffffffu, v, o); }
__device__ __forceinline__ PairF xchg(PairF v, int o) {
  return {__shfl_xor_sync(0xffffffffu, v.s, o), __shfl_xor_sync(0xffffffffu, v.c, o)};
}

// Sums over the warp of N <= 32 values a lane, by exchanging halves (N - 1 exchanges in place of 5 N): the
// lanes with (lane >> SH) == i are left with the i-th sum, where 32 >> SH = the power of two above N
template <int N, typename T>
__device__ __forceinline__ T spread_sums(const T* v, int lane) {
  constexpr int P = pow2_above(N);
  T a[P];
#pragma unroll
  for (int i = 0; i < P; ++i) a[i] = i < N ? v[i] : T{};
  int o = 16;
#pragma unroll
  for (int p = P; p > 1; p >>= 1, o >>= 1) {
    const bool up = lane & o;
#pragma unroll
    for (int i = 0; i < p / 2; ++i) {
      const T keep = up ? a[i + p / 2] : a[i], send = up ? a[i] : a[i + p / 2];
      a[i] = add(keep, xchg(send, o));
    }
  }
  for (; o > 0; o >>= 1) a[0] = add(a[0], xchg(a[0], o));
  return a[0];
}
template <int N>
__host__ __device__ constexpr int spread_shift() {
  int s = 5;
  for (int p = pow2_above(N); p > 1; p >>= 1) --s;
  return s;
}

// Sums over the warp of K values a lane into out[0..K)
template <int K, typename T, typename Out>
__device__ __forceinline__ void sums_to(const T* v, int lane, Out&& out) {
  constexpr int N0 = K < 32 ? K : 32, N1 = K - N0;
  {
    const T s = spread_sums<N0>(v, lane);
    constexpr int SH = spread_shift<N0>();
    if ((lane & ((1 << SH) - 1)) == 0 && (lane >> SH) < N0) out(lane >> SH, s);
  }
  if constexpr (N1 > 0) {
    const T s = spread_sums<N1>(v + N0, lane);
    constexpr int SH = spread_shift<N1>();
    if ((lane & ((1 << SH) - 1)) == 0 && (lane >> SH) < N1) out(N0 + (lane >> SH), s);
  }
}

// ---------------------------------------------------------------- one group's shared memory
template <int K, int W, int R>
struct __align__(16) MixSmem {
  static constexpr int NR = 32 * R;
  static constexpr int KR = (K + 3) / 4 * 4;  // row stride of R (vector loads along a row)
  static constexpr int KM = K | 1;            // row stride of M (odd: loads down a column)
  static constexpr int CPW = (K + W - 1) / W;
  float Rm[K * KR];
  float gb[W][(CPW + 4) / 4 * 4];  // a step's dots, per warp
  float v[W > 1 ? 2 : 1][W > 1 ? NR : 4];
  double t[NR], wt[NR];
  double F[K], zd[K], r[K], part[W][K];
  float rinv[K], rf[K], y[K], z[K];
  float M[K * KM];
  int32_t src[NR];      // row in processing order: its offset in the table, or its place in the scratch
  int32_t cnt[W][2];
  uint16_t orig[NR];    // its place in the row list
  int32_t slot;
  double down;          // undoes the scale of F
};

template <int K, int W, int R>
struct Rows {  // where a row's entries are: entry k at p[k * stride]
  const double* tab;
  const float *tab_h, *tab_l;
  const double* scr;
  const float *scr_h, *scr_l;
  int nf;
};

template <int W>
__device__ __forceinline__ void group_sync() {
  if constexpr (W == 1) __syncwarp();
  else __syncthreads();  // a block is one group
}

// R and 1 / R_kk of the system's rows, by modified Gram-Schmidt in FP32
template <int K, int W, int R, int RR>
__device__ __forceinline__ void factor(MixSmem<K, W, R>& S, const Rows<K, W, R>& rows, int n, int h, int lane) {
  constexpr int CPW = MixSmem<K, W, R>::CPW, KR = MixSmem<K, W, R>::KR;
  float a[CPW][RR];
  static_for<RR>([&](auto row) {
    constexpr int r = decltype(row)::value;
    const int i = r * 32 + lane;
    const bool ok = i < n, tb = i < rows.nf;
    const int32_t sr = ok ? S.src[i] : 0;
    const int stride = tb ? TAB_N : 32 * R;
    const float* p = (tb ? rows.tab_h : rows.scr_h) + sr + h * stride;
#pragma unroll
    for (int c = 0; c < CPW; ++c, p += W * stride) a[c][r] = ok && c * W + h < K ? *p : 0.0f;
  });
  // Columns in three blocks: a block's steps run one piece of code over the columns from its first one on
  // (the finished ones among them are updated too, to no effect).  One piece per step would be cheaper by a
  // quarter of the products, but the instruction cache does not hold it: with nine blocks and four lengths of
  // rows (460 KB of code) a third of all stalls were missing instructions.
  static_for<3>([&](auto block) {
    constexpr int C0 = decltype(block)::value * CPW / 3, C1 = (decltype(block)::value + 1) * CPW / 3;
    constexpr int NC = CPW - C0;
    const int k1 = C1 * W < K ? C1 * W : K;
#pragma unroll 1
    for (int k = C0 * W; k < k1; ++k) {
      const int kk = k / W, w = k - kk * W;  // column k is the local column kk of warp w
      float v[RR];
      if constexpr (W > 1) {
        float* vb = S.v[k & 1];
        if (h == w) {
#pragma unroll
          for (int c = C0; c < C1; ++c)
            if (kk == c) {
#pragma unroll
              for (int r = 0; r < RR; ++r) vb[r * 32 + lane] = a[c][r];
            }
        }
        group_sync<W>();
#pragma unroll
        for (int r = 0; r < RR; ++r) v[r] = vb[r * 32 + lane];
      } else {
        __syncwarp();
#pragma unroll
        for (int c = C0; c < C1; ++c)
          if (kk == c) {
#pragma unroll
            for (int r = 0; r < RR; ++r) v[r] = a[c][r];
          }
      }
      float d[NC + 1];  // d[0]: the column with itself; d[1 + i]: with the own column C0 + i
      {
        float s0 = 0.0f, s1 = 0.0f;
#pragma unroll
        for (int r = 0; r < RR; ++r) {
          if (r & 1) s1 = fmaf(v[r], v[r], s1);
          else s0 = fmaf(v[r], v[r], s0);
        }
        d[0] = s0 + s1;
      }
#pragma unroll
      for (int c = 0; c < NC; ++c) {
        float s0 = 0.0f;
#pragma unroll
        for (int r = 0; r < RR; ++r) s0 = fmaf(v[r], a[C0 + c][r], s0);
        d[1 + c] = s0;
      }
      // sums over the warp, back to every lane through shared memory
      sums_to<NC + 1>(d, lane, [&](int i, float v1) { S.gb[h][i] = v1; });
      __syncwarp();
      const float ss = S.gb[h][0];
      const float inv = ss > 0.0f ? __fdividef(1.0f, ss) : 0.0f;
#pragma unroll
      for (int c = 0; c < NC; ++c) {
        const float g = S.gb[h][1 + c] * inv;
#pragma unroll
        for (int r = 0; r < RR; ++r) a[C0 + c][r] = fmaf(-g, v[r], a[C0 + c][r]);
      }
      {  // R_kj, the lanes' own columns; the owner of column k its diagonal
        const float rs = ss > 0.0f ? rsqrtf(ss) : 0.0f;
        const int j = (C0 + lane) * W + h;
        if (lane < NC && j > k && j < K) S.Rm[k * KR + j] = S.gb[h][1 + lane] * rs;
        if (h == w && lane == 0) {
          S.Rm[k * KR + k] = ss * rs;
          S.rinv[k] = rs;
        }
      }
    }
  });
}

template <bool BATCH, int DIM, int Q, int W, int R, int MINB>
__global__ void __launch_bounds__(W > 1 ? 32 * W : 128, MINB)
    k_lsq_mixed(const __grid_constant__ LsArgs a0, const __grid_constant__ Tables T, const LsArgs* __restrict__ batch,
                const int64_t* __restrict__ slot_base, int n_geom) {
  constexpr int K = Mono<DIM, Q>::K, G = 32 * W, GROUPS = W > 1 ? 1 : 4;
  using Smem = MixSmem<K, W, R>;
  extern __shared__ __align__(16) unsigned char smem_raw[];
  const int warp = threadIdx.x >> 5, lane = threadIdx.x & 31;
  const int grp = warp / W, h = warp % W, tid = h * 32 + lane;
  Smem& S = reinterpret_cast<Smem*>(smem_raw)[grp];
  constexpr int NR = Smem::NR;
  // the rows that are made here: entry k of row q at [k * NR + q], FP64 and as two FP32 numbers
  double* scr = a0.scratch + ((int64_t)blockIdx.x * GROUPS + grp) * (2 * NR * K);
  float* scr_h = reinterpret_cast<float*>(scr + NR * K);
  float* scr_l = scr_h + NR * K;
  int next = 0;  // thread 0: the system after this one, asked for a system ahead
  if (tid == 0) next = atomicAdd(a0.next, 1);
  while (true) {
    group_sync<W>();  // the previous system is done with
    if (tid == 0) S.slot = next;
    group_sync<W>();
    int s = S.slot;
    if (s >= a0.n_slots) break;
    if (tid == 0) next = atomicAdd(a0.next, 1);
    int g = 0;
    if constexpr (BATCH) {  // the geometry of system s: last g with slot_base[g] <= s
      int lo = 0, hi = n_geom - 1;
      while (lo < hi) {
        const int mid = (lo + hi + 1) >> 1;
        if (slot_base[mid] <= s) lo = mid;
        else hi = mid - 1;
      }
      g = lo;
      s -= (int)slot_base[g];
    }
    const LsArgs& a = BATCH ? batch[g] : a0;
    const Dims& dm = a.dm;
    const int64_t p0 = a.row_ptr[s];
    const int n = (int)(a.row_ptr[s + 1] - p0);
    const int64_t gf = a.slot_face[s];
    // base cell and x0 (Sec. 2.4: face centre for grid faces, cell centre for EB faces)
    int base[3] = {0, 0, 0};
    int dface = -1;
    int64_t cut_self = -1, flocal = -1;
    if (gf >= dm.n_grid_faces) {
      cut_self = gf - dm.n_grid_faces;
      cell_xyz(dm, a.cut_cell[cut_self], base);
    } else {
      for (int d = 0; d < DIM; ++d)
        if (gf >= dm.face_base[d]) dface = d;
      flocal = gf - dm.face_base[dface];
      face_xyz(dm, dface, flocal, base);
    }
    // ---- rows in processing order: full cells (table) first, then the rest (scratch)
    constexpr int RT = (R + W - 1) / W;  // rows per lane
    {
      uint32_t desc[RT];
      int code[RT], below[RT];  // table offset or -1; rows of the same sort before it in this warp's share
      int nfull = 0, ncut = 0;
#pragma unroll
      for (int q = 0; q < RT; ++q) {
        const int i = (h * RT + q) * 32 + lane;
        code[q] = -2;
        if (i < n) {
          desc[q] = a.row_desc[p0 + i];
          code[q] = -1;
          if (rd_kind(desc[q]) == 0) {
            int c[3], x2[3];
#pragma unroll
            for (int d = 0; d < 3; ++d) {
              const int dl = d < DIM ? rd_off(desc[q], d) : 0;
              c[d] = base[d] + dl;
              x2[d] = 2 * dl + (d == dface) + 11;  // offset from x0 in units of h / 2
            }
            if (a.cut_of_cell[cell_id(dm, c)] < 0) code[q] = tab_place(x2);  // radius <= 3: inside the table
          }
        }
        const unsigned mf = __ballot_sync(0xffffffffu, code[q] >= 0), mc = __ballot_sync(0xffffffffu, code[q] == -1);
        const unsigned lt = (1u << lane) - 1u;
        below[q] = code[q] >= 0 ? nfull + __popc(mf & lt) : ncut + __popc(mc & lt);
        nfull += __popc(mf);
        ncut += __popc(mc);
      }
      if constexpr (W > 1) {
        if (lane == 0) {
          S.cnt[h][0] = nfull;
          S.cnt[h][1] = ncut;
        }
        group_sync<W>();
      } else {
        if (lane == 0) S.cnt[0][0] = nfull;
        __syncwarp();
      }
      int f0 = 0, c0 = 0, nf = 0;
      for (int w = 0; w < W; ++w) {
        if (w < h) {
          f0 += S.cnt[w][0];
          c0 += S.cnt[w][1];
        }
        nf += S.cnt[w][0];
      }
#pragma unroll
      for (int q = 0; q < RT; ++q) {
        const int i = (h * RT + q) * 32 + lane;
        if (code[q] >= 0) {
          const int at = f0 + below[q];
          S.src[at] = code[q];
          S.orig[at] = (uint16_t)i;
          S.wt[at] = a.wtab[code[q]];
        } else if (code[q] == -1) {
          const int at = nf + c0 + below[q];
          S.src[at] = (int32_t)desc[q];  // replaced by its place when the row is made
          S.orig[at] = (uint16_t)i;
        }
      }
      group_sync<W>();
    }
    int nf = 0;
    for (int w = 0; w < W; ++w) nf += S.cnt[w][0];
    Rows<K, W, R> rows{a.ftab, a.ftab_h, a.ftab_l, scr, scr_h, scr_l, nf};
    // ---- the rows that need a shift to x0, 32 at a time
#pragma unroll 1
    for (int b0 = nf + 32 * h; b0 < n; b0 += G) {
      const int at = b0 + lane;
      if (at < n) {
        const uint32_t ds = (uint32_t)S.src[at];
        const int kind = rd_kind(ds);
        int c[3], x2[3];
        double delta[3];
#pragma unroll
        for (int d = 0; d < 3; ++d) {
          const int dl = d < DIM ? rd_off(ds, d) : 0;
          c[d] = base[d] + dl;
          x2[d] = 2 * dl + (d == dface);
        }
        double m[K];
        const double* from = nullptr;
        bool neumann = false;
        int32_t cut = -1;
        if (kind == 2) {
          const int wd = rd_wdir(ds), ws = rd_wside(ds);
          x2[wd] += ws ? 1 : -1;
          int fx[3] = {c[0], c[1], c[2]};
          if (ws) fx[wd] += 1;
          const int32_t cf = a.cutface_of[wd][face_local(dm, wd, fx)];
          if (cf >= 0) {
            const double* fm = a.face_mom[wd] + (int64_t)cf * dm.KFS;
#pragma unroll
            for (int i = 0; i < K; ++i) m[i] = T.tang[wd][i] >= 0 ? fm[T.tang[wd][i]] : 0.0;
          } else {
            from = T.full_face[wd];
          }
        } else {
          cut = a.cut_of_cell[cell_id(dm, c)];
          neumann = kind == 1 && a.eb_bc && a.eb_bc[cut] != 0;
          if (kind == 1) from = a.eb_mom + (int64_t)cut * dm.KS;
          else from = cut >= 0 ? a.vol_mom + (int64_t)cut * dm.KS : T.full_vol;
        }
#pragma unroll
        for (int d = 0; d < 3; ++d) delta[d] = 0.5 * x2[d];
        const int y[3] = {x2[0] + 11, x2[1] + 11, x2[2] + 11};
        double w = a.wtab[tab_place(y)];
        double sc;
        if (!neumann) {
          if (from) {
#pragma unroll
            for (int i = 0; i < K; ++i) m[i] = from[i];
          }
          shift_regs<DIM, Q>(m, delta);
          sc = w / m[0];
        } else {
          // Neumann row (Sec. 2.2.1): (1/m^0) sum_d p_d m^{p - e_d}_d, from the EB moments weighted by
          // the normal components, shifted to x0.  It is a derivative in xi = (x - x0)/h, so its
          // coefficient is h^(D-1) s_hat and the physical minimum-norm problem weighs it with W_ii / h.
          w = w / dm.h;
#pragma unroll
          for (int i = 0; i < K; ++i) m[i] = 0.0;
          static_for<DIM>([&](auto dim) {
            constexpr int d = decltype(dim)::value;
            double q[K];
            const double* nm = a.eb_nmom + ((int64_t)cut * DIM + d) * dm.KS;
#pragma unroll
            for (int i = 0; i < K; ++i) q[i] = nm[i];
            shift_regs<DIM, Q>(q, delta);
            static_for<Q>([&](auto u_) {
              static_for<DIM == 2 ? 1 : Q - decltype(u_)::value>([&](auto v_) {
                constexpr int u = decltype(u_)::value, v = decltype(v_)::value;
#pragma unroll
                for (int p = 1; p <= Q - u - v; ++p)
                  m[Mono<DIM, Q>::at(d, p, u, v)] =
                      fma((double)p, q[Mono<DIM, Q>::at(d, p - 1, u, v)], m[Mono<DIM, Q>::at(d, p, u, v)]);
              });
            });
          });
          sc = w / a.eb_mom[(int64_t)cut * dm.KS];
        }
        S.wt[at] = w;
        const int place = at - nf;
        S.src[at] = place;
#pragma unroll
        for (int i = 0; i < K; ++i) {
          const double v = m[i] * sc;
          scr[i * NR + place] = v;
          float vh, vl;
          split_bits(v, &vh, &vl);
          scr_h[i * NR + place] = vh;
          scr_l[i * NR + place] = vl;
        }
      }
    }
    // ---- F_hat (Sec. 2.2.1): grid face: p_d m_f^{p-e_d}; EB face: sum_d p_d m_{d,f}^{p-e_d}
    for (int i = tid; i < K; i += G) {
      double f = 0.0;
      if (cut_self >= 0) {
        for (int d = 0; d < DIM; ++d) {
          const double* nm = a.eb_nmom + ((int64_t)cut_self * DIM + d) * dm.KS;
          if (T.lower[d][i] >= 0) f += (double)T.mon[i][d] * nm[T.lower[d][i]];
        }
      } else {
        const int q = T.lower[dface][i];
        if (q >= 0) {
          const int32_t cf = a.cutface_of[dface][flocal];
          double mq;
          if (cf >= 0) mq = T.tang[dface][q] >= 0 ? a.face_mom[dface][(int64_t)cf * dm.KFS + T.tang[dface][q]] : 0.0;
          else mq = T.full_face[dface][q];
          f = (double)T.mon[i][dface] * mq;
        }
      }
      S.r[i] = f;
    }
    group_sync<W>();
    // F scaled to size one by a power of two, which passes every rounding, so that the coefficients scale with the
    // face's moments: the solves' FP32 numbers, and the squares in the size of a correction, do not hold every scale
    // (F at 1e-18: the corrections' squares were zero, the system passed for settled and t was 1e-8 off; at 1e21
    // their overflow did the same).  F that is zero, subnormal or not finite stays, for the FP64 kernel.
    {
      uint32_t top = 0;  // high words of non-negative numbers compare like the numbers
      for (int i = lane; i < K; i += 32) top = max(top, (uint32_t)__double2hiint(S.r[i]) & 0x7fffffffu);
      const uint32_t e = __reduce_max_sync(0xffffffffu, top) >> 20;
      const bool normal = e > 0 && e < 2046;
      const double up = normal ? __hiloint2double((int)((2046 - e) << 20), 0) : 1.0;
      for (int i = tid; i < K; i += G) {
        const double f = S.r[i] * up;
        S.F[i] = f;
        S.rf[i] = (float)f;
      }
      if (tid == 0) S.down = normal ? __hiloint2double((int)(e << 20), 0) : 1.0;
    }
    // ---- R, then M = R^-1 (a lane per column)
    if constexpr (W > 1 && K > 15) {  // most systems have fewer than 14 rows a lane
      if (n <= 32 * 14) factor<K, W, R, 14>(S, rows, n, h, lane);
      else factor<K, W, R, R>(S, rows, n, h, lane);
    } else {
      factor<K, W, R, R>(S, rows, n, h, lane);
    }
    group_sync<W>();
    {
      // non-negative numbers compare like their bits
      const int k0 = lane < K ? lane : K - 1, k1 = lane + 32 < K ? lane + 32 : K - 1;
      const unsigned u0 = __float_as_uint(S.Rm[k0 * Smem::KR + k0]), u1 = __float_as_uint(S.Rm[k1 * Smem::KR + k1]);
      const float dmin = __uint_as_float(__reduce_min_sync(0xffffffffu, min(u0, u1)));
      const float dmax = __uint_as_float(__reduce_max_sync(0xffffffffu, max(u0, u1)));
      if (!(dmin > MIX_MIN_DIAG * dmax)) {  // also when there are fewer rows than unknowns
        if (tid == 0) a.status[s] = 3;
        continue;
      }
    }
    for (int j = tid; j < K; j += G) {
      float x[K];
      static_for<K>([&](auto row) {
        constexpr int i = K - 1 - decltype(row)::value;
        float acc0 = i == j ? 1.0f : 0.0f, acc1 = 0.0f;
#pragma unroll
        for (int l = i + 1; l < K; ++l) {
          if ((l - i) & 1) acc0 = fmaf(-S.Rm[i * Smem::KR + l], x[l], acc0);
          else acc1 = fmaf(-S.Rm[i * Smem::KR + l], x[l], acc1);
        }
        x[i] = (acc0 + acc1) * S.rinv[i];
        S.M[i * Smem::KM + j] = x[i];
      });
    }
    group_sync<W>();
    // z = M M^T rf; returns ||M^T rf||, the 2-norm of B z up to rounding
    auto solve = [&]() -> float {
      if constexpr (W > 1) {
        const int o = tid >> 1;
        float acc = 0.0f;
        if (o < K) {  // M is zero below its diagonal
#pragma unroll
          for (int i = 0; i < K; i += 2)
            if (i + (tid & 1) < K) acc = fmaf(S.M[(i + (tid & 1)) * Smem::KM + o], S.rf[i + (tid & 1)], acc);
        }
        acc += __shfl_xor_sync(0xffffffffu, acc, 1);
        if (o < K && !(tid & 1)) S.y[o] = acc;
        group_sync<W>();
        acc = 0.0f;
        if (o < K) {
#pragma unroll
          for (int j = 0; j < K; j += 2)
            if (j + (tid & 1) < K) acc = fmaf(S.M[o * Smem::KM + j + (tid & 1)], S.y[j + (tid & 1)], acc);
        }
        acc += __shfl_xor_sync(0xffffffffu, acc, 1);
        if (o < K && !(tid & 1)) {
          S.z[o] = acc;
          S.zd[o] = (double)acc;
        }
      } else {
        float acc = 0.0f;
        if (lane < K) {
#pragma unroll
          for (int i = 0; i < K; ++i) acc = fmaf(S.M[i * Smem::KM + lane], S.rf[i], acc);
        }
        if (lane < K) S.y[lane] = acc;
        __syncwarp();
        acc = 0.0f;
        if (lane < K) {
#pragma unroll
          for (int j = 0; j < K; ++j) acc = fmaf(S.M[lane * Smem::KM + j], S.y[j], acc);
          S.z[lane] = acc;
          S.zd[lane] = (double)acc;
        }
      }
      float q = 0.0f;
      for (int k = lane; k < K; k += 32) q = fmaf(S.y[k], S.y[k], q);
      for (int o = 16; o > 0; o >>= 1) q += __shfl_xor_sync(0xffffffffu, q, o);
      group_sync<W>();
      return sqrtf(q);
    };
    // t (+)= B z and r = F - B^T t, FP64
    auto pass64 = [&](bool first) {
      double acc[K];
#pragma unroll
      for (int k = 0; k < K; ++k) acc[k] = 0.0;
#pragma unroll 1
      for (int i0 = 32 * h; i0 < n; i0 += G) {
        const int i = i0 + lane;
        const bool ok = i < n, tb = i < nf;
        const double* p = (tb ? rows.tab : rows.scr) + (ok ? S.src[i] : 0);
        const int stride = tb ? TAB_N : 32 * R;
        double row[K];
#pragma unroll
        for (int k = 0; k < K; ++k, p += stride) row[k] = ok ? *p : 0.0;
        // one chain in the order of the degrees, its partial sums smaller than those of two chains with every other entry
        // (the terms cancel: Neumann systems came out 10 % further off), and not slower
        double t0 = 0.0;
#pragma unroll
        for (int k = 0; k < K; ++k) t0 = fma(row[k], S.zd[k], t0);
        if (!first && ok) t0 += S.t[i];
        if (ok) S.t[i] = t0;
#pragma unroll
        for (int k = 0; k < K; ++k) acc[k] = fma(row[k], t0, acc[k]);
      }
      sums_to<K>(acc, lane, [&](int k, double v) { S.part[h][k] = v; });
      group_sync<W>();
      for (int k = tid; k < K; k += G) {
        double v = S.F[k];
        for (int w = 0; w < W; ++w) v -= S.part[w][k];
        S.r[k] = v;
        S.rf[k] = (float)v;
      }
      group_sync<W>();
    };
    // t += B z in FP32
    auto pass32 = [&]() {
#pragma unroll 1
      for (int i0 = 32 * h; i0 < n; i0 += G) {
        const int i = i0 + lane;
        const bool ok = i < n, tb = i < nf;
        const float* ph = (tb ? rows.tab_h : rows.scr_h) + (ok ? S.src[i] : 0);
        const int stride = tb ? TAB_N : 32 * R;
        float q[4] = {};
#pragma unroll
        for (int k = 0; k < K; ++k, ph += stride) q[k & 3] = fmaf(ok ? *ph : 0.0f, S.z[k], q[k & 3]);
        if (ok) S.t[i] += (double)((q[0] + q[1]) + (q[2] + q[3]));
      }
      group_sync<W>();
    };
    // dt = B z, t += dt and (unless it is the last) r -= B^T dt, with compensated FP32 sums
    auto pass_df = [&](bool last) {
      PairF acc[K];
#pragma unroll
      for (int k = 0; k < K; ++k) acc[k] = {0.0f, 0.0f};
#pragma unroll 1
      for (int i0 = 32 * h; i0 < n; i0 += G) {
        const int i = i0 + lane;
        const bool ok = i < n, tb = i < nf;
        const int32_t sr = ok ? S.src[i] : 0;
        const float *ph = (tb ? rows.tab_h : rows.scr_h) + sr, *pl = (tb ? rows.tab_l : rows.scr_l) + sr;
        const int stride = tb ? TAB_N : 32 * R;
        float bh[K], bl[K];
#pragma unroll
        for (int k = 0; k < K; ++k, ph += stride, pl += stride) {
          bh[k] = ok ? *ph : 0.0f;
          bl[k] = ok ? *pl : 0.0f;
        }
        PairF q[4] = {};  // four chains: a compensated sum is six dependent operations long
#pragma unroll
        for (int k = 0; k < K; ++k) {
          const float z = S.z[k], p = __fmul_rn(bh[k], z);
          two_sum(q[k & 3].s, q[k & 3].c, p);
          q[k & 3].c += fmaf(bl[k], z, fmaf(bh[k], z, -p));
        }
        const PairF d = add(add(q[0], q[1]), add(q[2], q[3]));
        const float dh = d.s + d.c, dl = d.c - (dh - d.s);
        if (ok) S.t[i] += (double)dh + (double)dl;
        if (last) continue;
#pragma unroll
        for (int k = 0; k < K; ++k) {
          const float p = __fmul_rn(bh[k], dh);
          const float e = fmaf(bl[k], dh, fmaf(bh[k], dl, fmaf(bh[k], dh, -p)));
          two_sum(acc[k].s, acc[k].c, p);
          acc[k].c += e;
        }
      }
      if (last) {
        group_sync<W>();
        return;
      }
      sums_to<K>(acc, lane, [&](int k, PairF v) { S.part[h][k] = (double)v.s + (double)v.c; });
      group_sync<W>();
      for (int k = tid; k < K; k += G) {
        double v = S.r[k];
        for (int w = 0; w < W; ++w) v -= S.part[w][k];
        S.r[k] = v;
        S.rf[k] = (float)v;
      }
      group_sync<W>();
    };
    bool settled = false;
    float norm0 = 0.0f, prev = 1.0f;
    int n64 = 0, ndf = 0;
    for (int corr = 0; corr <= MIX_MAX_CORR && !settled; ++corr) {
      const float d = solve() / (corr ? norm0 : 1.0f);  // the correction's size, relative to t
      if (corr == 0) {
        norm0 = d;
        pass64(true);
        ++n64;
        continue;
      }
      if (!(d <= prev)) break;  // not a number, or growing
      settled = d <= MIX_TOL || (d <= 0.1f * prev && d * (d / prev) <= MIX_NEXT);
      if (d > MIX_DF_MAX<Q>) {
        pass64(false);
        ++n64;
      } else if (settled && d <= MIX_F32_MAX) {
        pass32();
      } else {
        pass_df(settled);
        ++ndf;
      }
      prev = d;
    }
    if (tid == 0 && a0.flops) {  // executed flops of this system (the row construction not counted)
      const double nk = (double)n * K;
      atomicAdd(a0.flops + 0, 4.0 * nk * n64);
      atomicAdd(a0.flops + 1, 2.0 * nk * K - 2.0 / 3.0 * K * K * K + 22.0 * 2.0 * nk * ndf);
    }
    if (!settled) {  // the FP64 kernel takes the system
      if (tid == 0) a.status[s] = 3;
      continue;
    }
    const double down = S.down;
    for (int i = tid; i < n; i += G) a.row_val[p0 + S.orig[i]] = S.wt[i] * S.t[i] * down;  // s_hat = W t
    if (tid == 0) a.status[s] = 0;
  }
}

// ---------------------------------------------------------------- dispatch
// A warp per system while 32 R rows hold the largest one (2-D and second order: 4 systems a block, no block
// barriers), else a block of four warps per system, whose lanes hold any system's rows (MAXROWS / 32 = 20).
// Both on the same systems: 3-D second order at 80^3 4.64 ms by warps and 7.19 ms by blocks, 2-D fourth order at
// 512^2 (9328 faces) 0.21 and 0.52 ms.  One large system takes a whole build, or batch, to the block shape, which is
// still well below the kernel before: second order with R_n = 3, 2-D at 512^2 (71 rows) 0.29 ms (before 0.76), 3-D at
// 80^3 (468 rows) 16.3 ms (87.8).  Fourth order in 3-D needs the registers of four warps for one system's rows;
// at 128^3 two blocks an SM take 133.7 ms, three (with more spills) 132.0 ms, seven warps a system 140.7 ms.
namespace {

struct MixShape {
  int systems;  // in flight per block
  int64_t scratch;  // doubles of one of them
  int per_sm;   // resident blocks per SM
  cudaError_t (*launch)(unsigned blocks, cudaStream_t s, const LsArgs& a0, const Tables& T, const LsArgs* batch,
                        const int64_t* slot_base, int n_geom);
};

template <int DIM, int Q, int W, int R, int MINB>
cudaError_t mix_launch(unsigned blocks, cudaStream_t s, const LsArgs& a0, const Tables& T, const LsArgs* batch,
                       const int64_t* slot_base, int n_geom) {
  const int smem = (W > 1 ? 1 : 4) * (int)sizeof(MixSmem<Mono<DIM, Q>::K, W, R>), threads = W > 1 ? 32 * W : 128;
  cudaError_t e;
  if (batch) {
    e = cudaFuncSetAttribute(k_lsq_mixed<true, DIM, Q, W, R, MINB>, cudaFuncAttributeMaxDynamicSharedMemorySize, smem);
    if (e != cudaSuccess) return e;
    k_lsq_mixed<true, DIM, Q, W, R, MINB><<<blocks, threads, smem, s>>>(a0, T, batch, slot_base, n_geom);
  } else {
    e = cudaFuncSetAttribute(k_lsq_mixed<false, DIM, Q, W, R, MINB>, cudaFuncAttributeMaxDynamicSharedMemorySize, smem);
    if (e != cudaSuccess) return e;
    k_lsq_mixed<false, DIM, Q, W, R, MINB><<<blocks, threads, smem, s>>>(a0, T, nullptr, nullptr, 1);
  }
  return cudaGetLastError();
}

template <int DIM, int Q, int R1, int MINB1, int WL, int MINBL>
MixShape shape_for(int max_rows) {
  if constexpr (R1 > 0)
    if (max_rows <= 32 * R1) return {4, 2 * 32 * R1 * Mono<DIM, Q>::K, MINB1, mix_launch<DIM, Q, 1, R1, MINB1>};
  return {1, 2 * 640 * Mono<DIM, Q>::K, MINBL, mix_launch<DIM, Q, WL, 20, MINBL>};
}

MixShape mix_shape(const Tables& T, int max_rows) {
  if (T.dim == 3) return T.K == 35 ? shape_for<3, 4, 0, 1, EB_LS_W, EB_LS_CTAS>(max_rows) : shape_for<3, 2, 8, 3, 4, 4>(max_rows);
  return T.K == 15 ? shape_for<2, 4, 4, 4, 4, 4>(max_rows) : shape_for<2, 2, 2, 6, 4, 4>(max_rows);
}

}  // namespace

int64_t lsq_mixed_blocks(const Tables& T, int max_rows, int64_t systems, int nsm, int64_t* scratch_doubles) {
  const MixShape m = mix_shape(T, max_rows);
  const int64_t nb = std::max<int64_t>(1, std::min<int64_t>((int64_t)nsm * m.per_sm, (systems + m.systems - 1) / m.systems));
  *scratch_doubles = nb * m.systems * m.scratch;
  return nb;
}

cudaError_t lsq_mixed_launch(int64_t blocks, int max_rows, cudaStream_t s, const LsArgs& a0, const Tables& T,
                             const LsArgs* batch, const int64_t* slot_base, int n_geom) {
  return mix_shape(T, max_rows).launch((unsigned)blocks, s, a0, T, batch, slot_base, n_geom);
}

}  // namespace eb
