// Launch wrappers of the solver's CUDA kernels (definitions in assembly.cu,
// sparse.cu, krylov.cu). All take raw device pointers and a stream.
#pragma once
#include <cstdint>
#include <cuda_runtime.h>

#include "element.cuh"

namespace fsi {

// per-problem inflow data: center[3], normal[3], radius, peak, amp, freq, phase
constexpr int INLET_STRIDE = 11;

struct MeshDev {
  int64_t N, T, Tf;          // nodes, tets, fluid tets (tets [0, Tf) fluid, [Tf, T) wall)
  const double* X;           // [N*3]
  const int32_t* tets;       // [T*4]
  const uint32_t* nflag;     // [N]
  const int32_t* nprob;      // [N]
  const double* inlet;       // [nprob*INLET_STRIDE]
  const double* geo;         // [GEO][T] reference geometry of every tet (element.cuh)
};

// ---- wall shear stress (wss.cu): face = 4 * fluid tet + local index of the
// vertex opposite the face; fb = [P+1] face offsets of the problems
void launch_wss(const MeshDev& m, double mu, int64_t nf, const int64_t* face, const int64_t* fb, int32_t P,
                const double* y, double* wss, double* marea, double* area, double* sawss, cudaStream_t s);

// ---- assembly (assembly.cu)
void launch_elem_residual(const MeshDev& m, const MatConst& mc, const double* y, const double* y1,
                          const double* y2, double* Fe, cudaStream_t s);
// the node rows' sums, constrained rows replaced (t: the step's end time)
void launch_gather_residual(const MeshDev& m, const MatConst& mc, double t, const int64_t* nptr, const int32_t* nsrc,
                            const double* Fe, const double* y, const double* y1, double* F, cudaStream_t s);
// reference geometry of every tet into geo ([GEO][T])
void launch_geometry(const MeshDev& m, double* geo, cudaStream_t s);
// element Jacobians of the tets [t0, t1) into Ke (784 values per tet, from tet t0).
// Mixed form: Xl per-tet reference coordinates relative to vertex 0 (12 per tet), all
// inputs FP32
void launch_elem_jacobian(const MeshDev& m, const MatConst& mc, const float* Xl, const float* y, const float* y1,
                          const float* y2, float* Ke, int64_t t0, int64_t t1, cudaStream_t s);
// FP64: val holds JAC_VALUES values per tet of the chunk
constexpr int JAC_VALUES = 140;
void launch_elem_jacobian(const MeshDev& m, const MatConst& mc, const double* y, const double* y1, double* val,
                          double* Ke, int64_t t0, int64_t t1, cudaStream_t s);
// out = [a | b | c] converted to FP32 (3 n floats)
void launch_states_to_float(int64_t n, const double* a, const double* b, const double* c, float* out,
                            cudaStream_t s);
// add the element blocks of the tets [t0, t1) (Ke as above) into the BSR values;
// t0 = 0 starts the sums
template <class T>
void launch_gather_jacobian(int64_t nnzb, const int64_t* bptr, const int32_t* bsrc, const T* Ke, T* vals,
                            int64_t t0, int64_t t1, cudaStream_t s);
template <class T>
void launch_constraint_jacobian(const MeshDev& m, const MatConst& mc, const int32_t* diag, T* vals,
                                cudaStream_t s);

// ---- sparse (sparse.cu)
// y = J x; threads_per_row 32 (one warp per block row) or 16 (two rows per
// warp); guard: optional device flag, the kernel does nothing while *guard == 0
template <class TV>
void launch_bsr_spmv(int64_t n, const int64_t* row_ptr, const int32_t* col, const TV* vals, const TV* x,
                     double* y, int threads_per_row, const int* guard, cudaStream_t s);
void launch_to_float(int64_t n, const double* x, float* y, const int* guard, cudaStream_t s);

struct RasDev {
  int32_t np;
  const int64_t* sd_row;
  const int32_t* gnode;
  const uint8_t* owned;
  const int64_t* row_ptr;
  const int32_t* col;
  const int64_t* gblk;
  const int64_t* diag;
  const int64_t* lent_ptr;
  const int64_t* lent_pos;
  const int64_t* lent_kdiag;
  const int64_t* upd_ptr;
  const int64_t* upd_tgt;
  const int64_t* upd_src;
  const int64_t* sd_lvlL;
  const int64_t* sd_lvlU;
  const int64_t* lvlL_ptr;
  const int64_t* lvlU_ptr;
  const int32_t* lvlL_rows;
  const int32_t* lvlU_rows;
  int64_t nblocks;
  int32_t max_row_blocks;  // most blocks in one factor row
  int32_t max_row_lent;    // most L blocks in one row
  int32_t max_row_upd;     // most elimination updates in one row
  int32_t max_entry_upd;   // most updates of one L block
  int32_t factor_mode;     // factorisation kernel: 0..2 rows in order (shared-memory modes), 3 nested-dissection groups,
                           // 4 rows in order, pipelined
  // pipelined factorisation (setup.h, FactorPipe)
  const int32_t* ent_k;
  const int32_t* ent_len;
  const int64_t* meta_off;
  const uint32_t* meta;
  int32_t pipe_slots;      // L blocks in flight
  int32_t pipe_meta;       // bytes of a slot's word list
  int32_t pipe_data;       // bytes of a slot's blocks
  uint32_t pipe_tries;     // looks after which a wait gives up
  int32_t pipe_stall;      // tests only: 1 the producer issues nothing, 2 the eliminating threads give up at
                           // once (the other roles' waits run out)
  const int32_t* sd_depth; // [np] nested-dissection depth of each subdomain (0: one item)
  const int64_t* sd_item;  // [np+1] first item of each subdomain
  const int64_t* item_row; // [items] end row of each item (subdomain-relative)
  int32_t max_depth;       // deepest dissection (the nested-dissection factorisation uses 2^max_depth groups)
};
template <class TF, class TJ>
void launch_ras_extract(const RasDev& r, const TJ* vals, TF* fac, cudaStream_t s);
template <class TF>
void launch_ras_factor(const RasDev& r, TF* fac, int32_t* err, cudaStream_t s);
template <class TF>
bool ras_factor_fits(const RasDev& r, int mode);  // mode 0..4 fits one CTA
// shared memory of the factorisation CTA
template <class TF>
size_t ras_factor_smem(const RasDev& r, int mode);
// shared-memory limit of the factorisation CTA (the opt-in maximum)
constexpr size_t FACTOR_SMEM_MAX = 227 * 1024;
template <class TF>
void launch_ras_apply(const RasDev& r, const TF* fac, const double* rin, TF* work, double* z, float* z32,
                      const int* guard, cudaStream_t s);

// ---- streamed RAS apply (ras_stream.cu)
struct RasStreamDev {
  int32_t np;
  const int64_t* sd_row;
  const int32_t* gnode;
  const uint8_t* owned;
  const int64_t* L_cnt;   // [rows] L blocks of each row
  const int64_t* U_cnt;   // [rows] 1 (inverted pivot) + U blocks of each row
  const int64_t* L_off;   // [np+1] first packed L block of each subdomain
  const int64_t* U_off;   // [np+1] first packed U block of each subdomain (its U part follows its L part)
  void* pack;
  int64_t nblk;           // packed blocks
  const int64_t* src;     // [nblk] factor block copied into each packed block
  const int32_t* col;     // [nblk] subdomain-relative column row
  const int64_t* piv;     // [nblk] factor block of the row's inverted pivot; -1: copied as it is
  const uint32_t* code;   // entry codes of the chain apply (setup.h, StreamPlan)
  const int64_t* code_off;// [np+1] first code word of each subdomain
  const uint8_t* stage;   // blocks of each stage of the chain apply
  const int64_t* stage_off;// [np+1] first stage of each subdomain
  int32_t stage_blocks;   // blocks per ring stage (one bulk copy; rows may straddle stages)
  int32_t chain_blocks;   // chain and team apply: most blocks of a stage
  int32_t team;           // the team apply runs (four warps per subdomain)
  int64_t max_rows;       // rows of the largest subdomain
  int32_t nst;            // ring stages in flight per warp (2..8)
  int32_t stall;          // tests only: 1 the producer issues nothing (bounded waits run out), 2 the
                          // first wait gives up at once, 3 a wait gives up on one lane of each warp
                          // (ring: the first; team kernels: the last)
  // nested-dissection items (one item per subdomain for the other orderings)
  const int32_t* sd_depth;  // [np] depth D: 2^(D+1) - 1 items, solved by 2^D warps
  const int64_t* sd_item;   // [np+1] first item of each subdomain
  const int64_t* item_row;  // [items] end row of each item (subdomain-relative)
  const int32_t* item_blk;  // [items][4] first / end block of the item in the subdomain's L and U streams
  int32_t max_depth;        // deepest D (the CTA has 2^max_depth warps)
};
template <class TF>
size_t ras_stream_smem(const RasStreamDev& r);
template <class TF>
void launch_pack_factors(const RasStreamDev& r, const TF* fac, cudaStream_t s);
// once per context: allow the apply kernel its dynamic shared memory
template <class TF>
cudaError_t ras_stream_init(const RasStreamDev& r);
// z = B^{-1} r; z32 (optional) receives an FP32 copy; guard as for the SpMV. Takes
// the chain kernel, a team kernel where subdomains are few (r.team), or the ring
// kernel for dissected subdomains
template <class TF>
cudaError_t launch_ras_apply_stream(const RasStreamDev& r, const double* rin, double* z, float* z32, int32_t* err,
                                    const int* guard, cudaStream_t s);

// ---- batched Krylov / BLAS-1 (krylov.cu): vectors of n doubles holding P
// independent problems one after the other; reductions are segmented by
// problem over a fixed chunk table (deterministic). guard: optional device
// flag; guarded kernels do nothing while *guard == 0.
struct SegDev {
  int32_t P;                 // problems
  int64_t n_chunks;
  const int64_t* chunk_beg;  // [n_chunks+1] first dof of each chunk (chunks never straddle problems)
  const int64_t* prob_chunk; // [P+1] chunks of each problem
  const int32_t* node_prob;  // [N] problem of each node
  int* counter;              // [P][SEG_COUNTERS] blocks done per vector group, then groups done; zero between launches
};
constexpr int SEG_GROUPS = 9;  // vector groups of 8 in one multi-dot (restart <= 64 -> at most 65 vectors)
constexpr int SEG_COUNTERS = SEG_GROUPS + 1;
// out[p * ldo + k] = V_k . w for k < nv (and, with_self = 1, out[p * ldo + nv] = w . w)
void launch_seg_mdot(const SegDev& sg, int32_t nv, const double* V, int64_t ldv, const double* w, double* partial,
                     double* out, int32_t ldo, const int* guard, cudaStream_t s, int with_self = 0);
// The norm of a Gram-Schmidt step's new vector from its second pass (krylov.cu, new_norm)
struct NewNorm {
  double* hsub;       // H[p][j+1][j], ldsub apart per problem; null: no norm wanted
  int64_t ldsub;
  double* inv;        // [P] its reciprocal
  int* unsafe;        // [P] the norm is taken from the updated vector
  int* flag;          // [1] for some problem (null: no such problem)
  double* norms;      // [P] those norms
  const int* active;  // [P] the problem iterates
  int force;          // tests only: every norm from the updated vector
};
// the same with w . w, then the norm of w - V out as sqrt(w . w - ||V . w||^2) into hsub where
// that is safe, its reciprocal into inv, else unsafe[p] = 1
void launch_seg_mdot_norm(const SegDev& sg, int32_t nv, const double* V, int64_t ldv, const double* w,
                          double* partial, double* out, int32_t ldo, const NewNorm& N, const int* guard,
                          cudaStream_t s);
// selective reorthogonalisation test after one Gram-Schmidt pass (see krylov.cu)
void launch_seg_reorth_decide(int32_t P, const double* ws, const double* nrm, int32_t ldn, double* hb, int32_t lda,
                              int32_t j, const int* active, int* flag, cudaStream_t s);
void launch_seg_norm(const SegDev& sg, const double* x, double* partial, double* out, int32_t ldo,
                     const int* guard, cudaStream_t s);
// w -= V h per problem, then w *= scal[p] (scal optional). With N.flag: cleared (no scal), or the
// unsafe problems' norms formed where it is set (partial: n_chunks values)
void launch_seg_maxpy(const SegDev& sg, int64_t n, int32_t nv, const double* V, int64_t ldv, const double* h,
                      int32_t ldh, double* w, const int* guard, cudaStream_t s, const double* scal = nullptr,
                      const NewNorm& N = NewNorm{}, double* partial = nullptr);
void launch_seg_scale_inv(const SegDev& sg, int64_t n, const double* x, const double* scal, int32_t lds,
                          double* y, const int* guard, cudaStream_t s);

void launch_seg_cycle_init(int32_t P, double* g, int32_t ldg, const double* beta, const double* target, int* active,
                           int* kcols, int* any, cudaStream_t s);
// column j of each active problem's Hessenberg = a + b (the two Gram-Schmidt passes, lda apart per
// problem), then the Givens update; beside it, where N.flag (optional) is set, the unsafe problems' w_p
// divided by their norms (w: n values)
void launch_seg_givens(int32_t P, const double* a, const double* b, int32_t lda, double* H, int32_t ldh, int32_t m,
                       int32_t j, double* cs, double* sn, double* g, double* res, const double* target, int* active,
                       int* kcols, int* any, const SegDev& sg, int64_t n, double* w, const NewNorm& N,
                       const int* guard, cudaStream_t s);
void launch_seg_lsq(int32_t P, const double* H, int32_t ldh, int32_t m, const int* kcols, const double* g, double* y,
                    cudaStream_t s);
void launch_seg_update_x(const SegDev& sg, int64_t n, const double* Z, int64_t ldz, const double* y, int32_t m,
                         const int* kcols, double* x, cudaStream_t s);
void launch_seg_axpy(const SegDev& sg, int64_t n, const double* x, const double* alpha, const double* y, double* out,
                     cudaStream_t s);
void launch_seg_neg_masked(const SegDev& sg, int64_t n, const double* x, const int* mask, double* out,
                           cudaStream_t s);
void launch_axpby(int64_t n, double a, const double* x, double b, const double* y, double* out,
                  cudaStream_t s);
void launch_copy(int64_t n, const double* x, double* y, cudaStream_t s);
void launch_fill(int64_t n, double v, double* x, cudaStream_t s);

}  // namespace fsi
