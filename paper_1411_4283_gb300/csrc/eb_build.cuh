// Argument structures of the build kernels (eb_build.cu), shared with the host code.
#pragma once
#include <stdint.h>

#include "eb_internal.cuh"
#include "eb_tables.cuh"

namespace eb {

constexpr int RW = 6;  // 64-bit words of a (2R+1)^3 <= 343-bit mask

struct Mask {
  uint64_t w[RW];
};

struct GatherArgs {
  Dims dm;
  const uint8_t* flag;
  const uint8_t* ff[3];
  const int32_t* reach_idx;  // [ncell] index into masks or -1 (clean: whole box / ball)
  const Mask* masks;
  const int32_t* cut_of_cell;
  const int64_t* slot_face;
  const int64_t* row_ptr;    // null in the counting pass
  uint32_t* row_desc;
  int64_t* count;            // [n_slots] counting pass output
  int32_t* max_rows;         // counting pass: most rows of a slot
};

// LS kernel shapes (compile-time; EB_LS_W / EB_LS_CTAS / EB_LS_SYS / EB_LS_RPL override them for tuning builds)
#ifndef EB_LS_W
#define EB_LS_W 4
#endif
#ifndef EB_LS_CTAS
#define EB_LS_CTAS 2
#endif
#ifndef EB_LS_SYS
#define EB_LS_SYS 4
#endif
#ifndef EB_LS_RPL
#define EB_LS_RPL 4
#endif
constexpr int LS_SYS = EB_LS_SYS;  // systems in flight per CTA, FP64 factorisation (shared memory bound)
constexpr int LS_NW = 2;           // warps per system (each owns the columns j with j % LS_NW == its rank)
constexpr int RPL = EB_LS_RPL;     // rows per lane per chunk
constexpr int CH = 32 * RPL;       // rows per chunk
constexpr int KST = MAXK;          // row stride in shared memory (odd: conflict-free 64-bit access)

// Per-system shared memory of the FP64 factorisation
struct __align__(16) LsSysSmem {
  double R[MAXK * MAXK + 1];  // triangular factor, row-major
  double C[CH * KST];         // current chunk of weighted rows
  double P[32 * KST];         // partial dot products, column j in P[lane][j] (each column owned by one warp)
  double vec[5 * MAXK];       // F, y, z, tau, 1/R_kk
  double xch[LS_NW * MAXK];   // the warps' partial sums (corrected semi-normal equations)
  double hs[2][4];            // Householder scalars (beta, v0, gamma, reflect) of step k in hs[k % 2]
  unsigned long long bar;     // barrier of the system's warps (mbarrier, 32 * LS_NW arrivals per phase)
  int32_t slot;               // system being solved
  int32_t hs_seq[2];          // step number whose scalars hs[k % 2] holds (posted after the values)
};
static_assert(sizeof(LsSysSmem) % 16 == 0, "per-system blocks stay 16-byte aligned");
static_assert(LS_SYS * sizeof(LsSysSmem) <= 232448, "the systems of a CTA fit in 227 KB of shared memory");
// per-system global scratch (doubles) of the FP64 factorisation: the rows column-major (MAXROWS x MAXK),
// the weights and t (MAXROWS each)
constexpr int64_t LS_SCRATCH = (int64_t)MAXROWS * (MAXK + 2);

// offsets in units of h/2 span [-11, 11] on each axis (volume, EB and wall rows)
constexpr int TAB_S = 23;
constexpr int TAB_N = TAB_S * TAB_S * TAB_S;
// Place of the offset with indices x (0..TAB_S-1 each): even x first, then odd ones, so that the rows of
// neighbouring cells (two half-cells apart) are next to each other
__host__ __device__ inline int tab_place(const int* x) {
  return (x[0] & 1) * ((TAB_S + 1) / 2) + (x[0] >> 1) + TAB_S * (x[1] + TAB_S * x[2]);
}

struct LsArgs {
  Dims dm;
  const Tables* T;
  const uint8_t* flag;
  const int32_t* cut_of_cell;
  const int32_t* cut_cell;
  const double* vol_mom;
  const double* eb_mom;
  const double* eb_nmom;
  const uint8_t* eb_bc;
  const int32_t* cutface_of[3];
  const double* face_mom[3];
  const int64_t* slot_face;
  const int64_t* row_ptr;
  const uint32_t* row_desc;
  double* row_val;
  int64_t n_slots;
  const int32_t* slot_list;  // [n_slots] systems to solve (null: 0 .. n_slots-1)
  int32_t* next;       // work counter
  int32_t* status;     // [n_slots]: 0 ok, 1 rank deficient, 3 left to the FP64 path, 4 solved there
  double* scratch;     // per system in flight: LS_SCRATCH doubles (FP64), see k_lsq_mixed (mixed)
  int32_t* err;        // set when a bounded wait between the two warps of a system gives up
  double* flops;       // [2] executed flops, accumulated: FP64, FP32
  // weighted rows of full cells by offset (tab_place): entry k at [k * TAB_N + place], FP64 and as the sum of
  // two FP32 numbers, and the weights [TAB_N]
  const double* ftab;
  const float* ftab_h;
  const float* ftab_l;
  const double* wtab;
};

struct AsmArgs {
  Dims dm;
  const uint8_t* flag;
  const int32_t* cut_of_cell;
  const int32_t* face_slot[3];
  const int32_t* eb_slot;
  const int64_t* slot_face;
  const int64_t* row_ptr;
  const uint32_t* row_desc;
  const double* row_val;
  const uint8_t* ff[3];
  int nfoot;
  const int16_t* foot_lut;  // [(2R+3)^3] footprint index of an offset, -1 outside
  int64_t n_rows;
  double* rows64;
  float* rows32;
  double inv_h2;
  const uint8_t* eb_bc;   // [n_cut] 0 Dirichlet, 1 Neumann
  const double* eb_mom;   // [n_cut][KS] (the EB area fraction is entry 0)
};

__global__ void k_mark(Dims dm, const uint8_t* flag, uint8_t* mark);
__global__ void k_dilate(Dims dm, int axis, int R, const uint8_t* in, uint8_t* out);
__global__ void k_classify_faces(Dims dm, int d, const uint8_t* fflag, const uint8_t* dil, int32_t* state,
                                 int64_t* class_rep, int32_t* is_unique);
__global__ void k_face_slots(Dims dm, int d, const int32_t* state, const int64_t* upos, int64_t ubase,
                             const int32_t* class_slot, int32_t* slot, int64_t* slot_face);
__global__ void k_reach(Dims dm, const int32_t* cells, int64_t ncells, const uint8_t* flag, const uint8_t* ff0,
                        const uint8_t* ff1, const uint8_t* ff2, Mask* out);
cudaError_t gather_launch(const GatherArgs& a, int64_t n_slots, const int32_t* cut_cell, cudaStream_t s);
// Adjoint of the stencil solves with respect to the moment tables (k_stencil_adjoint, eb_build.cu)
struct AdjArgs {
  const double* lam;        // [ncell] adjoint solution
  const double* phi;        // [ncell] forward solution
  // derivatives of the moment tables for parameter 0; parameter p's at + p * the stride
  const double* dvol;       // [n_cut][KS] of the volume moments (stride s_vol)
  const double* deb;        // [n_cut][KS] of the EB moments (stride s_vol)
  const double* debn;       // [n_cut][dim][KS] of the normal-weighted EB moments (stride s_ebn)
  const double* dface[3];   // [n_cutface[d]][KFS] of the face moments (stride s_face[d])
  int n_par;                // parameters
  int64_t s_vol, s_ebn, s_face[3];
  int64_t n_slots;          // systems [0, n_slots) (the individually solved ones)
  int32_t* next;            // work counter
  double* scratch;          // per warp: MAXROWS * ADJ_SCRATCH doubles
  double* dJ;               // [n_par] accumulated derivatives
};
constexpr int ADJ_WARPS = 4;
constexpr int ADJ_SCRATCH = MAXK + 10;  // doubles per row of a warp's scratch
cudaError_t stencil_adjoint_launch(unsigned blocks, cudaStream_t s, const LsArgs& a, const Tables& T,
                                   const AdjArgs& g);
// FP64 factorisation (k_lsq, eb_build.cu): shared-memory attribute, then one launch over the systems of one
// geometry (batch == null) or of several (batch[g] per geometry, slot_base prefix sums of their systems)
cudaError_t lsq_prepare();
cudaError_t lsq_launch(unsigned blocks, cudaStream_t s, const LsArgs& a0, const Tables& T, const LsArgs* batch,
                       const int64_t* slot_base, int n_geom);
// Mixed path (k_lsq_mixed, eb_lsq.cu), systems of at most max_rows rows: its blocks and the scratch they need,
// and the launch; the systems it cannot finish get status 3
int64_t lsq_mixed_blocks(const Tables& T, int max_rows, int64_t systems, int nsm, int64_t* scratch_doubles);
cudaError_t lsq_mixed_launch(int64_t blocks, int max_rows, cudaStream_t s, const LsArgs& a0, const Tables& T,
                             const LsArgs* batch, const int64_t* slot_base, int n_geom);
// the systems with status 3 (global numbers: + base) appended to list[*count]
cudaError_t lsq_fallback_list(const int32_t* status, int64_t n, int64_t base, int32_t* list, int32_t* count,
                              cudaStream_t s);
__global__ void k_full_rows(Dims dm, const Tables* T, double* ftab, float* ftab_h, float* ftab_l, double* wtab);
__global__ void k_assemble_rows(AsmArgs a, const int32_t* rep_cell, int64_t nrep, int64_t row0, int32_t* err);
// boundary entries of the irregular cells' rows: counted into cnt (bptr null) or written
cudaError_t assemble_b_launch(const AsmArgs& a, const int32_t* cells, int64_t ncells, int64_t* cnt, const int64_t* bptr,
                              int64_t* bcol, double* bval, cudaStream_t s);
// counts[0, 1] += the faces of one direction with a slot and with a class slot; counts[2, 3] += the systems of
// status 1 (rank deficient) and 4 (solved by the FP64 pass)
cudaError_t count_faces(const int32_t* slot, int64_t n, int64_t n_unique, unsigned long long* counts, cudaStream_t s);
cudaError_t count_status(const int32_t* status, int64_t n, unsigned long long* counts, cudaStream_t s);

}  // namespace eb
