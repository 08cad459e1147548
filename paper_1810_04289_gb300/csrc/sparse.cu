// Block-sparse (7x7 BSR) matrix-vector product and the restricted additive
// Schwarz preconditioner of Sec. 3, Eq. 14-16, with block ILU(k) subdomain
// solves: extraction of the overlapped submatrices J_i^delta, the batched
// factorisation (one CTA per subdomain, all subdomains in one launch), and the
// level-scheduled forward/backward solves with the restricted (owned-rows-only)
// prolongation used when the TMA-fed apply (ras_stream.cu) does not fit.
#include <cuda_runtime.h>

#include "kernels.cuh"
#include "setup.h"

namespace fsi {

namespace {

inline int grid_for(int64_t work, int block) {
  int64_t g = (work + block - 1) / block;
  const int64_t cap = 152 * 64;
  return (int)(g < 1 ? 1 : (g > cap ? cap : g));
}

// ---------------------------------------------------------------------------
// SpMV: S block slots x 8 component lanes (7 used) per row, 32 / (8 S) rows per
// warp; slot q takes every S-th block of the row, the partial sums of a component
// are combined by shuffles. FP64: values, vector and sums in FP64, one fused
// multiply-add per product (the FP64 pipe bounds this form: 4 warps of an SM issue one
// FP64 instruction per 19 cycles; a tree sum per block took 10 instructions where the
// chain takes 7: 103k-node tree 240 -> 159 us). Mixed: FP32 values and an FP32 copy
// of the vector; each block's 7-term product is formed in FP32 and the block products
// are accumulated in FP64: a conversion and an FP64 addition per block product, which
// bound the kernel about as much as memory does (174k-node tree 104 us; sums in pairs of
// floats took 98, but carry 48 bits and FP32's range).
// ---------------------------------------------------------------------------
__device__ __forceinline__ double add_product(double acc, const float* A, const float* x) {
  const float s0 = A[0] * x[0] + A[1] * x[1];
  const float s1 = A[2] * x[2] + A[3] * x[3];
  const float s2 = A[4] * x[4] + A[5] * x[5];
  return acc + (double)((s0 + s1) + (s2 + A[6] * x[6]));
}
__device__ __forceinline__ double add_product(double acc, const double* A, const double* x) {
#pragma unroll
  for (int k = 0; k < 7; ++k) acc = fma(A[k], x[k], acc);
  return acc;
}

template <class TV, int S>
__global__ void __launch_bounds__(256) k_bsr_spmv(int64_t n, const int64_t* __restrict__ row_ptr,
                                                  const int32_t* __restrict__ col, const TV* __restrict__ vals,
                                                  const TV* __restrict__ x, double* __restrict__ y,
                                                  const int* __restrict__ guard) {
  if (guard && *guard == 0) return;
  constexpr int G = 8 * S;
  const int lane = threadIdx.x & 31;
  const int gl = lane % G;
  const int r = gl / S, q = gl % S;
  const int64_t grp0 = (blockIdx.x * (int64_t)blockDim.x + threadIdx.x) / G;
  const int64_t ngrp = ((int64_t)gridDim.x * blockDim.x) / G;
  for (int64_t base = grp0 - (lane / G); base < n; base += ngrp) {
    const int64_t row = base + (lane / G);
    double acc = 0.0;
    if (r < 7 && row < n) {
      const int64_t b0 = row_ptr[row], b1 = row_ptr[row + 1];
      // four of this lane's blocks per pass: their column indices first, then
      // all their loads, so that the loads of a pass are in flight together
      for (int64_t b = b0 + q; b < b1; b += 4 * S) {
        int cl[4];
#pragma unroll
        for (int u = 0; u < 4; ++u) cl[u] = b + u * S < b1 ? col[b + u * S] : -1;
#pragma unroll
        for (int u = 0; u < 4; ++u)
          if (cl[u] >= 0) acc = add_product(acc, vals + 49 * (b + u * S) + 7 * r, x + 7 * (int64_t)cl[u]);
      }
    }
#pragma unroll
    for (int o = 1; o < S; o <<= 1) acc += __shfl_xor_sync(0xffffffffu, acc, o);
    if (r < 7 && q == 0 && row < n) y[7 * row + r] = acc;
  }
}

__global__ void k_to_float(int64_t n, const double* __restrict__ x, float* __restrict__ y,
                           const int* __restrict__ guard) {
  if (guard && *guard == 0) return;
  const int64_t i0 = blockIdx.x * (int64_t)blockDim.x + threadIdx.x, st = (int64_t)gridDim.x * blockDim.x;
  if ((reinterpret_cast<uintptr_t>(x) & 15) == 0) {  // a caller's vector may start anywhere
    for (int64_t i = i0; i < (n >> 1); i += st) {
      const double2 v = reinterpret_cast<const double2*>(x)[i];
      reinterpret_cast<float2*>(y)[i] = make_float2((float)v.x, (float)v.y);
    }
    if ((n & 1) && i0 == 0) y[n - 1] = (float)x[n - 1];
  } else {
    for (int64_t i = i0; i < n; i += st) y[i] = (float)x[i];
  }
}

// ---------------------------------------------------------------------------
// RAS: extraction of J_i^delta = R_i^delta J (R_i^delta)^T (Eq. 15)
// ---------------------------------------------------------------------------
// one warp per block (one index read per block, no division per value)
template <class TF, class TJ>
__global__ void __launch_bounds__(256) k_ras_extract(int64_t nblocks, const int64_t* __restrict__ gblk,
                                                     const TJ* __restrict__ vals, TF* __restrict__ fac) {
  const int lane = threadIdx.x & 31;
  const int64_t step = ((int64_t)gridDim.x * blockDim.x) >> 5;
#pragma unroll 2
  for (int64_t b = (blockIdx.x * (int64_t)blockDim.x + threadIdx.x) >> 5; b < nblocks; b += step) {
    const int64_t gb = gblk[b];
    const TJ* v = vals + 49 * gb;
    const TF x0 = gb >= 0 ? (TF)v[lane] : TF(0), x1 = gb >= 0 && lane < 17 ? (TF)v[lane + 32] : TF(0);
    fac[49 * b + lane] = x0;
    if (lane < 17) fac[49 * b + lane + 32] = x1;
  }
}

template <class TF> __device__ __forceinline__ TF tiny_pivot();
template <> __device__ __forceinline__ double tiny_pivot<double>() { return 1e-300; }
template <> __device__ __forceinline__ float tiny_pivot<float>() { return 1e-37f; }

// In-place inverse of the 7x7 block B (row-major) by one warp: Gauss-Jordan with
// partial pivoting on the augmented [B | I] in shared memory `aug` (7 x 14).
template <class TF>
__device__ void warp_invert7(TF* B, TF* aug, int32_t* err) {
  const int lane = threadIdx.x & 31;
  for (int e = lane; e < 98; e += 32) {
    const int r = e / 14, c = e - 14 * r;
    aug[e] = c < 7 ? B[7 * r + c] : (c - 7 == r ? TF(1) : TF(0));
  }
  __syncwarp();
  for (int k = 0; k < 7; ++k) {
    // pivot search (lane 0), row swap
    int piv = k;
    if (lane == 0) {
      TF best = fabs(aug[14 * k + k]);
      for (int r = k + 1; r < 7; ++r) {
        TF v = fabs(aug[14 * r + k]);
        if (v > best) { best = v; piv = r; }
      }
      if (!(best > tiny_pivot<TF>())) atomicExch(err, 1);
    }
    piv = __shfl_sync(0xffffffffu, piv, 0);
    if (piv != k && lane < 14) {
      TF a = aug[14 * k + lane];
      aug[14 * k + lane] = aug[14 * piv + lane];
      aug[14 * piv + lane] = a;
    }
    __syncwarp();
    const TF inv = TF(1) / aug[14 * k + k];
    __syncwarp();
    if (lane < 14) aug[14 * k + lane] *= inv;
    __syncwarp();
    // every lane reads the multipliers of its entries before any lane writes
    TF fct[4];
#pragma unroll
    for (int it = 0; it < 4; ++it) {
      const int e = lane + 32 * it;
      fct[it] = e < 98 ? aug[14 * (e / 14) + k] : TF(0);
    }
    __syncwarp();
#pragma unroll
    for (int it = 0; it < 4; ++it) {
      const int e = lane + 32 * it;
      if (e < 98) {
        const int r = e / 14, c = e - 14 * r;
        if (r != k) aug[e] -= fct[it] * aug[14 * k + c];
      }
    }
    __syncwarp();
  }
  for (int e = lane; e < 49; e += 32) {
    const int r = e / 7, c = e - 7 * r;
    B[e] = aug[14 * r + 7 + c];
  }
  __syncwarp();
}

// Batched block ILU, whole CTA on one row: one CTA per subdomain walks its rows
// in increasing order (a topological order of the elimination). At the start
// of a row the row itself is loaded into shared memory. For each L block (i,k):
// threads 0..48 form A_ik D_k^{-1} (D_k: the inverted pivot of the finished row
// k; into a separate buffer and the row), then all threads apply its updates
// A_ij -= A_ik A_kj (task = update x column) - two barriers per L block.
// MODE picks how much besides the row lives in shared memory, largest first
// (the factor_mode option of fsi_options is MODE + 1):
//   0: the pivots D_k of all L blocks of the row, loaded with the row, and the
//      source blocks A_kj of each L block's updates in a cp.async double
//      buffer, one L block ahead (their latency hides behind the previous L
//      block's arithmetic);
//   1: as 0 but D_k read from global memory (L2) when used;
//   2: only the row: D_k and the sources read from global memory when used.
// All three do the same arithmetic in the same order (bitwise identical
// factors). MODE 2 (factor_mode 3, the row only) runs where the pipelined kernel
// below does not fit (see ras_factor_fits), 0 and 1 where they are asked for.
template <class TF>
__device__ __forceinline__ void cp_async_elem(TF* dst, const TF* src) {
  asm volatile("cp.async.ca.shared.global [%0], [%1], %2;" ::"r"((uint32_t)__cvta_generic_to_shared(dst)),
               "l"(src), "n"(sizeof(TF))
               : "memory");
}
__device__ __forceinline__ void cp_async_commit() { asm volatile("cp.async.commit_group;" ::: "memory"); }
__device__ __forceinline__ void cp_async_wait1() { asm volatile("cp.async.wait_group 1;" ::: "memory"); }

template <class TF>
__device__ __forceinline__ void fetch_sources(const RasDev& R, const TF* fac, int64_t e, TF* buf, int tid, int nt) {
  const int64_t ub = R.upd_ptr[e];
  const int ne = (int)(R.upd_ptr[e + 1] - ub);
  for (int idx = tid; idx < 49 * ne; idx += nt) {
    const int u = idx / 49;
    cp_async_elem<TF>(buf + idx, fac + 49 * R.upd_src[ub + u] + (idx - 49 * u));
  }
}

template <class TF, int MODE>
__global__ void __launch_bounds__(256) k_ras_factor_cta(RasDev R, TF* __restrict__ fac, int32_t* err) {
  extern __shared__ __align__(16) unsigned char fsm[];
  const size_t me = MODE <= 1 ? (size_t)R.max_entry_upd * 49 : 0;
  TF* sRow = reinterpret_cast<TF*>(fsm);
  TF* sD = sRow + (size_t)R.max_row_blocks * 49;
  TF* sSrc0 = sD + (MODE == 0 ? (size_t)R.max_row_lent * 49 : 0);
  TF* sSrc1 = sSrc0 + me;
  TF* sScl = sSrc1 + me;
  TF* sAug = sScl + 49;
  const int tid = threadIdx.x, nt = blockDim.x;
  const int s = blockIdx.x;
  for (int64_t q = R.sd_row[s]; q < R.sd_row[s + 1]; ++q) {
    const int64_t rp = R.row_ptr[q];
    const int nblk = (int)(R.row_ptr[q + 1] - rp);
    const int64_t e0 = R.lent_ptr[q], e1 = R.lent_ptr[q + 1];
    const int nl = (int)(e1 - e0);
    if (MODE <= 1) {
      if (e0 < e1) fetch_sources<TF>(R, fac, e0, sSrc0, tid, nt);
      cp_async_commit();
    }
    for (int idx = tid; idx < 49 * nblk; idx += nt) sRow[idx] = fac[49 * rp + idx];
    if (MODE == 0)
      for (int idx = tid; idx < 49 * nl; idx += nt) {
        const int e = idx / 49;
        sD[idx] = fac[49 * R.lent_kdiag[e0 + e] + (idx - 49 * e)];
      }
    __syncthreads();
    for (int64_t e = e0; e < e1; ++e) {
      TF* cur = ((e - e0) & 1) ? sSrc1 : sSrc0;
      TF* nxt = ((e - e0) & 1) ? sSrc0 : sSrc1;
      if (MODE <= 1) {
        if (e + 1 < e1) fetch_sources<TF>(R, fac, e + 1, nxt, tid, nt);
        cp_async_commit();
      }
      TF* Aik = sRow + 49 * (R.lent_pos[e] - rp);
      if (tid < 49) {
        const TF* Dk = MODE == 0 ? sD + 49 * (e - e0) : fac + 49 * R.lent_kdiag[e];
        const int r = tid / 7, c = tid - 7 * r;
        TF v = TF(0);
#pragma unroll
        for (int mm = 0; mm < 7; ++mm) v += Aik[7 * r + mm] * Dk[7 * mm + c];
        sScl[tid] = v;
      }
      if (MODE <= 1) cp_async_wait1();  // this thread's copies of L block e have landed
      __syncthreads();
      if (tid < 49) Aik[tid] = sScl[tid];
      const int64_t ub = R.upd_ptr[e];
      const int ntask = 7 * (int)(R.upd_ptr[e + 1] - ub);
      for (int t = tid; t < ntask; t += nt) {
        const int u = t / 7, cc = t - 7 * u;
        TF* Aij = sRow + 49 * (R.upd_tgt[ub + u] - rp) + cc;
        const TF* Akj = (MODE <= 1 ? cur + 49 * u : fac + 49 * R.upd_src[ub + u]) + cc;
        TF col[7];
#pragma unroll
        for (int mm = 0; mm < 7; ++mm) col[mm] = Akj[7 * mm];
#pragma unroll
        for (int rr = 0; rr < 7; ++rr) {
          TF acc = Aij[7 * rr];
#pragma unroll
          for (int mm = 0; mm < 7; ++mm) acc -= sScl[7 * rr + mm] * col[mm];
          Aij[7 * rr] = acc;
        }
      }
      __syncthreads();
    }
    if (tid < 32) warp_invert7<TF>(sRow + 49 * (R.diag[q] - rp), sAug, err);
    __syncthreads();
    for (int idx = tid; idx < 49 * nblk; idx += nt) fac[49 * rp + idx] = sRow[idx];
    __syncthreads();
  }
}

// 1 / x, correctly rounded (what the division gives), without its call
__device__ __forceinline__ float rcp_rn(float x) { return 1.0f / x; }
__device__ __forceinline__ double rcp_rn(double x) { return __drcp_rn(x); }

// In-place inverse of the 7x7 block B by one warp, the same arithmetic as
// warp_invert7 with a column of [B | I] in each lane's registers (lanes 0..13).
template <class TF>
__device__ __forceinline__ void warp_invert7_regs(TF* B, int32_t* err) {
  const int lane = threadIdx.x & 31;
  TF a[7];
#pragma unroll
  for (int r = 0; r < 7; ++r) a[r] = lane < 7 ? B[7 * r + lane] : (lane - 7 == r ? TF(1) : TF(0));
#pragma unroll
  for (int k = 0; k < 7; ++k) {
    int piv = k;
    TF best = fabs(a[k]);
#pragma unroll
    for (int r = k + 1; r < 7; ++r) {
      const TF v = fabs(a[r]);
      if (v > best) {
        best = v;
        piv = r;
      }
    }
    if (lane == k && !(best > tiny_pivot<TF>())) atomicMax(err, 1);  // (a wait that gave up, 2, stays reported)
    piv = __shfl_sync(0xffffffffu, piv, k);
    const TF ak = a[k];
#pragma unroll
    for (int r = k + 1; r < 7; ++r)
      if (r == piv) {
        a[k] = a[r];
        a[r] = ak;
      }
    const TF inv = rcp_rn(__shfl_sync(0xffffffffu, a[k], k));
    a[k] *= inv;
#pragma unroll
    for (int r = 0; r < 7; ++r)
      if (r != k) {
        const TF f = __shfl_sync(0xffffffffu, a[r], k);
        a[r] -= f * a[k];
      }
  }
  if (lane >= 7 && lane < 14) {
#pragma unroll
    for (int r = 0; r < 7; ++r) B[7 * r + lane - 7] = a[r];
  }
}

__device__ __forceinline__ void pipe_bar_init(uint64_t* b, uint32_t n) {
  asm volatile("mbarrier.init.shared::cta.b64 [%0], %1;" ::"r"((uint32_t)__cvta_generic_to_shared(b)), "r"(n)
               : "memory");
}
__device__ __forceinline__ void pipe_bar_arrive(uint64_t* b) {
  asm volatile("mbarrier.arrive.shared::cta.b64 _, [%0];" ::"r"((uint32_t)__cvta_generic_to_shared(b)) : "memory");
}
// bounded wait: false if the phase did not complete within `tries` looks
__device__ __forceinline__ bool pipe_bar_wait(uint64_t* b, uint32_t parity, uint32_t tries) {
  const uint32_t a = (uint32_t)__cvta_generic_to_shared(b);
  uint32_t it = 0;
  do {  // (tries is looked at after the first miss only)
    uint32_t ok;
    asm volatile(
        "{\n .reg .pred p;\n mbarrier.try_wait.parity.shared::cta.b64 p, [%1], %2;\n selp.u32 %0, 1, 0, p;\n}\n"
        : "=r"(ok)
        : "r"(a), "r"(parity)
        : "memory");
    if (ok) return true;
  } while (++it < tries);
  return false;
}
__device__ __forceinline__ void cp_async16(void* dst, const void* src) {
  asm volatile("cp.async.cg.shared.global [%0], [%1], 16;" ::"r"((uint32_t)__cvta_generic_to_shared(dst)), "l"(src)
               : "memory");
}

// Pipelined block ILU, one CTA per subdomain, rows in order: the arithmetic of
// k_ras_factor_cta in its order (same bits). That kernel is bound by latency: for
// every L block it reads index lists, the pivot, the update lists and the source
// blocks from L2, one after the other, between two barriers. Here
//   - a producer warp copies what each L block needs (the host's word list and row
//     k's blocks from the pivot on) into a ring of slots, up to 8 L blocks ahead and
//     across rows, as soon as row k is finished; the row before stays in shared memory;
//   - the pivot of a row is inverted by a warp of its own, in registers, beside the
//     next row's elimination, which needs it last;
//   - the row's own values are read a row ahead; FP32 has one barrier per L block
//     (every warp forms A_ik D_k^{-1} for itself) and a thread takes a column of a
//     target block with A_ik D_k^{-1} in registers (57 loads per 343 products; one
//     element per thread took 15 instructions per product).
// Measured, us: FP32 14,350-node tube, 64 subdomains, ILU(1) 12,850 -> 4,420; 6-tube
// batch, 255 subdomains, ILU(2) 8,050 -> 3,460; 174k-node tree, 1,088 subdomains, ILU(2)
// 23,750 -> 17,400; FP64 429-node tube, 4 subdomains 7,960 -> 3,130, 14,350-node tube
// 30,870 -> 12,340 (FP64 pipe). The slots must leave two CTAs per SM (one up to 304
// subdomains: 46,657-node tube, FP64, 512 subdomains, one CTA 25,000, the kernel
// above 20,300).
//
// Every wait between the roles (the producer warp, the inverting warp, the threads that
// eliminate) is a bounded wait on an mbarrier or on the row counter. A thread that gives
// one up waits for nothing more and goes on to the end of the rows, so that the barrier
// of the eliminating threads stays matched; the other roles leave; nothing is read through
// an index that was not waited for. The call then reports FSI_ERR_TIMEOUT.
// threads that eliminate (then one producer warp and one warp that inverts the
// pivots). FP32: a thread updates a whole column of a target block; FP64: an element
constexpr int PIPE_HEAD = 160;         // barriers and the row counter
constexpr int PIPE_SCL = 4 * 56 * 4;  // bytes of the scaled L blocks
template <class TF> constexpr int PIPE_THREADS = sizeof(TF) == 4 ? 128 : 256;

template <class TF>
__global__ void __launch_bounds__(PIPE_THREADS<TF> + 64, sizeof(TF) == 4 ? 1 : 2) k_ras_factor_pipe(RasDev R, TF* fac, int32_t* err) {
  constexpr bool F32 = sizeof(TF) == 4;
  constexpr int NT = PIPE_THREADS<TF>, MAXSLOT = 8, PF = F32 ? 12 : 8;
  extern __shared__ __align__(16) unsigned char fsm[];
  uint64_t* full = reinterpret_cast<uint64_t*>(fsm);        // [MAXSLOT]
  uint64_t* empty = full + MAXSLOT;                         // [MAXSLOT]
  uint64_t* inv = empty + MAXSLOT;                          // a row's pivot is inverted
  uint64_t* upd = inv + 1;                                  // a row's updates are done
  volatile int* done = reinterpret_cast<volatile int*>(upd + 1);  // rows finished and stored
  TF* sScl = reinterpret_cast<TF*>(fsm + PIPE_HEAD);              // FP32 [4][56], rows of 8; FP64 [49]
  const int NS = R.pipe_slots;
  const uint32_t slot_bytes = R.pipe_meta + R.pipe_data;
  unsigned char* slots = fsm + PIPE_HEAD + PIPE_SCL;
  TF* sRow = reinterpret_cast<TF*>(slots + NS * slot_bytes);  // [2][max_row_blocks * 49]
  const int tid = threadIdx.x, lane = tid & 31, w = tid >> 5;
  const int s = blockIdx.x;
  const int64_t qb = R.sd_row[s], qe = R.sd_row[s + 1];
  if (tid == 0) {
    for (int i = 0; i < NS; ++i) {
      pipe_bar_init(&full[i], 32);
      pipe_bar_init(&empty[i], 1);
    }
    pipe_bar_init(inv, 1);
    pipe_bar_init(upd, NT / 32);
    *done = 0;
    asm volatile("fence.mbarrier_init.release.cluster;" ::: "memory");
  }
  __syncthreads();
  bool ok = R.pipe_stall != 2 || w >= NT / 32;
  const uint32_t tries = R.pipe_tries;
  int slot = 0, phase = 0;
  auto next_slot = [&]() {
    if (++slot == NS) {
      slot = 0;
      phase ^= 1;
    }
  };

  if (w == NT / 32) {
    // producer warp: for every L block in elimination order, its word list and row k's
    // blocks into the next free slot, once row k is finished
    const int64_t e0 = R.lent_ptr[qb], e1 = R.pipe_stall == 1 ? e0 : R.lent_ptr[qe];
    int fin = 0, issued = 0;
    for (int64_t eb = e0; eb < e1 && ok; eb += 32) {
      const int64_t em = eb + lane < e1 ? eb + lane : e1 - 1;
      const int mk = R.ent_k[em], ml = R.ent_len[em];
      const int64_t mkd = R.lent_kdiag[em], mo = R.meta_off[em];
      const int mn = (int)(R.meta_off[em + 1] - mo);
      const int cnt = (int)(e1 - eb < 32 ? e1 - eb : 32);
      for (int i = 0; i < cnt && ok; ++i) {
        const int k = __shfl_sync(0xffffffffu, mk, i), len = __shfl_sync(0xffffffffu, ml, i);
        const int n16 = __shfl_sync(0xffffffffu, mn, i);
        const int64_t kd = __shfl_sync(0xffffffffu, mkd, i), off = __shfl_sync(0xffffffffu, mo, i);
        if (issued >= NS) ok = pipe_bar_wait(&empty[slot], (uint32_t)(phase ^ 1), tries);
        if (len > 0 && fin <= k) {
          for (uint32_t it = 0; it < 16 * tries && (fin = *done) <= k; ++it) __nanosleep(20);
          ok = ok && fin > k;
          __threadfence_block();
        }
        ok = __all_sync(0xffffffffu, ok);
        if (!ok) break;
        unsigned char* d = slots + slot * slot_bytes;
        const unsigned char* ms = reinterpret_cast<const unsigned char*>(R.meta) + 16 * off;
        for (int x = lane; x < n16; x += 32) cp_async16(d + 16 * x, ms + 16 * x);
        if (len > 0) {
          const int64_t b0 = 49 * kd * (int64_t)sizeof(TF), a0 = b0 & ~(int64_t)15;
          const int n = (int)((49 * (kd + len) * (int64_t)sizeof(TF) - a0 + 15) >> 4);
          const unsigned char* ds = reinterpret_cast<const unsigned char*>(fac) + a0;
          for (int x = lane; x < n; x += 32) cp_async16(d + R.pipe_meta + 16 * x, ds + 16 * x);
        }
        asm volatile("cp.async.mbarrier.arrive.noinc.shared::cta.b64 [%0];" ::"r"(
                         (uint32_t)__cvta_generic_to_shared(&full[slot]))
                     : "memory");
        ++issued;
        next_slot();
      }
    }
    asm volatile("cp.async.wait_all;" ::: "memory");
    if (!ok && lane == 0) atomicExch(err, 2);
    return;
  }

  if (w == NT / 32 + 1) {
    // inverts each row's pivot when its updates are done, beside the next row's elimination
    for (int64_t q = qb; q < qe; ++q) {
      ok = __all_sync(0xffffffffu, pipe_bar_wait(upd, (uint32_t)((q - qb) & 1), tries));
      if (!ok) break;
      TF* B = sRow + (q & 1) * 49 * R.max_row_blocks + 49 * (int)(R.diag[q] - R.row_ptr[q]);
      warp_invert7_regs<TF>(B, err);
      __syncwarp();
      TF* out = fac + 49 * R.diag[q];
      for (int x = lane; x < 49; x += 32) out[x] = B[x];
      __threadfence_block();
      __syncwarp();
      if (lane == 0) {
        *done = (int)(q - qb) + 1;  // (the row's other blocks were stored before upd)
        pipe_bar_arrive(inv);
      }
    }
    if (!ok && lane == 0) atomicExch(err, 2);
    return;
  }

  auto bar = []() { asm volatile("bar.sync 1, %0;" ::"n"(PIPE_THREADS<TF>) : "memory"); };
  // the row's values a row ahead in registers, its offsets two rows ahead
  int64_t rp = R.row_ptr[qb], rp1 = R.row_ptr[qb + 1], rp2 = R.row_ptr[qb + 1 < qe ? qb + 2 : qb + 1];
  int64_t lp = R.lent_ptr[qb], lp1 = R.lent_ptr[qb + 1];
  TF pre[PF];
#pragma unroll
  for (int i = 0; i < PF; ++i) {
    const int64_t x = 49 * rp + tid + NT * i;
    pre[i] = x < 49 * rp1 ? fac[x] : TF(0);
  }
  // FP32: elements lane, lane + 32 of the scaled block
  const int r0 = lane / 7, c0 = lane - 7 * r0, r1 = (lane + 32) / 7, c1 = lane + 32 - 7 * r1;
  int nl_prev = 0;
  for (int64_t q = qb; q < qe; ++q) {
    const int nv = 49 * (int)(rp1 - rp), nl = (int)(lp1 - lp);
    TF* row = sRow + (q & 1) * 49 * R.max_row_blocks;
    const TF* prow = sRow + ((q & 1) ^ 1) * 49 * R.max_row_blocks + 49 * nl_prev;  // previous row, from its pivot on
#pragma unroll
    for (int i = 0; i < PF; ++i)
      if (tid + NT * i < nv) row[tid + NT * i] = pre[i];
    for (int x = tid + NT * PF; x < nv; x += NT) row[x] = fac[49 * rp + x];
    const int64_t rp3 = R.row_ptr[q + 3 <= qe ? q + 3 : qe], lp2 = R.lent_ptr[q + 2 <= qe ? q + 2 : qe];
#pragma unroll
    for (int i = 0; i < PF; ++i) {
      const int64_t x = 49 * rp1 + tid + NT * i;
      pre[i] = q + 1 < qe && x < 49 * rp2 ? fac[x] : TF(0);
    }
    bar();
    bool inverted = q == qb;  // the previous row's pivot
    auto wait_inverse = [&]() {
      if (!inverted && ok) ok = pipe_bar_wait(inv, (uint32_t)((q - qb - 1) & 1), tries);
      inverted = true;
    };
    for (int e = 0; e < nl; ++e) {
      // lanes of a warp may give up apart: they must not meet a barrier on different branches of
      // the block's kind. FP32: the warp votes, so that it takes one; FP64: the barrier is
      // outside the branches. (The kind from global memory for lanes that gave up, instead: 6-tube
      // batch refresh 4,394 us where this takes 4,249.)
      if constexpr (F32) ok = __all_sync(0xffffffffu, ok && pipe_bar_wait(&full[slot], (uint32_t)phase, tries));
      else if (ok) ok = pipe_bar_wait(&full[slot], (uint32_t)phase, tries);
      const uint32_t* meta = reinterpret_cast<const uint32_t*>(slots + slot * slot_bytes);
      const uint32_t head = ok ? meta[0] : 0;
      const int ne = (int)(head & 0xffff);
      const uint32_t kind = head >> 28;
      if (kind == PIPE_PREV) wait_inverse();
      // A_ik D_k^{-1}: FP32 in every warp for itself (one barrier per L block), FP64 once
      auto scale = [&](const TF* D) {
        const TF* A = row + 49 * e;
        if constexpr (F32) {
          TF* scl = sScl + 56 * w;
#pragma unroll
          for (int h = 0; h < 2; ++h) {
            const int x = lane + 32 * h;
            if (x < 49) {
              const int r = h ? r1 : r0, c = h ? c1 : c0;
              TF v = TF(0);
#pragma unroll
              for (int mm = 0; mm < 7; ++mm) v += A[7 * r + mm] * D[7 * mm + c];
              scl[8 * r + c] = v;
              if (w == 0) fac[49 * (rp + e) + x] = v;
            }
          }
        } else if (tid < 49) {
          const int r = tid / 7, c = tid - 7 * r;
          TF v = TF(0);
#pragma unroll
          for (int mm = 0; mm < 7; ++mm) v += A[7 * r + mm] * D[7 * mm + c];
          sScl[tid] = v;
          fac[49 * (rp + e) + tid] = v;
        }
      };
      auto update = [&](const TF* D) {
        if constexpr (F32) {
          if (tid < 7 * ne) {
            const TF* scl = sScl + 56 * w;
            float4 sv[14];  // the scaled block, rows of 8
#pragma unroll
            for (int i = 0; i < 14; ++i) sv[i] = *reinterpret_cast<const float4*>(scl + 4 * i);
            const TF* sc = reinterpret_cast<const TF*>(sv);
            for (int x = tid; x < 7 * ne; x += NT) {
              const int u = x / 7, c = x - 7 * u;
              const uint32_t ts = meta[2 + u];
              TF* T = row + 49 * (ts >> 16) + c;
              const TF* S = D + 49 * (ts & 0xffff) + c;
              TF col[7], acc[7];
#pragma unroll
              for (int mm = 0; mm < 7; ++mm) col[mm] = S[7 * mm], acc[mm] = T[7 * mm];
#pragma unroll
              for (int mm = 0; mm < 7; ++mm)
#pragma unroll
                for (int r = 0; r < 7; ++r) acc[r] -= sc[8 * r + mm] * col[mm];
#pragma unroll
              for (int r = 0; r < 7; ++r) T[7 * r] = acc[r];
            }
          }
        } else {
          for (int x = tid; x < 49 * ne; x += NT) {
            const int u = x / 49, el = x - 49 * u;
            const int r = el / 7, c = el - 7 * r;
            const uint32_t ts = meta[2 + u];
            TF* T = row + 49 * (ts >> 16) + el;
            const TF* S = D + 49 * (ts & 0xffff) + c;
            TF acc = *T;
#pragma unroll
            for (int mm = 0; mm < 7; ++mm) acc -= sScl[7 * r + mm] * S[7 * mm];
            *T = acc;
          }
        }
      };
      const TF* Ds = kind == PIPE_PREV ? prow
                                       : reinterpret_cast<const TF*>(slots + slot * slot_bytes + R.pipe_meta) +
                                             ((head >> 16) & 15);
      if constexpr (F32) {
        auto both = [&](const TF* D) {
          if (ok) scale(D);
          __syncwarp();
          if (ok) update(D);
        };
        if (kind == PIPE_DIRECT) both(fac + 49 * R.lent_kdiag[lp + e]);
        else both(Ds);
      } else {
        const TF* Dg = fac;
        if (kind == PIPE_DIRECT) {
          Dg = fac + 49 * R.lent_kdiag[lp + e];
          if (ok) scale(Dg);
        } else if (ok) {
          scale(Ds);
        }
        bar();
        if (kind == PIPE_DIRECT) {
          if (ok) update(Dg);
        } else if (ok) {
          update(Ds);
        }
      }
      bar();
      // (a slot that was not waited for is not given back: a copy may still be on its way into it)
      if (tid == 0 && ok) pipe_bar_arrive(&empty[slot]);
      next_slot();
    }
    // the pivot goes to the inverting warp, the blocks after it to global memory; the other
    // row buffer may be overwritten once the previous pivot has left it
    for (int x = 49 * (nl + 1) + tid; x < nv; x += NT) fac[49 * rp + x] = row[x];
    wait_inverse();
    __threadfence_block();
    __syncwarp();
    if (lane == 0) pipe_bar_arrive(upd);
    nl_prev = nl;
    rp = rp1;
    rp1 = rp2;
    rp2 = rp3;
    lp = lp1;
    lp1 = lp2;
  }
  if (!ok) atomicExch(err, 2);
}

// Block ILU on nested-dissection ordered subdomains: the CTA's 256 threads
// form G = 2^D groups (D the subdomain's dissection depth); in each phase (the
// leaves, then the separators level by level) every item of the phase is
// factored by its own group, row by row exactly as MODE 2 of k_ras_factor_cta
// does it (the row in shared memory, pivots and sources read from global
// memory), with the group's own barrier instead of the CTA's. Items of one
// phase share no entry, so their rows can be eliminated side by side; the
// arithmetic of every row is that of the sequential kernel, in the same order
// (bitwise identical factors). A CTA barrier separates the phases.
__device__ __forceinline__ void group_sync(int g, int gs) {
  if (gs == 32) {
    __syncwarp();
  } else {
    asm volatile("bar.sync %0, %1;" ::"r"(1 + g), "r"(gs) : "memory");
  }
}

template <class TF>
__global__ void __launch_bounds__(256) k_ras_factor_nd(RasDev R, TF* __restrict__ fac, int32_t* err) {
  extern __shared__ __align__(16) unsigned char fsm[];
  const int s = blockIdx.x;
  const int D = R.sd_depth[s];
  const int G = 1 << D, gs = blockDim.x / G;
  const int g = threadIdx.x / gs, lt = threadIdx.x - g * gs;
  const size_t per = (size_t)(R.max_row_blocks + 1) * 49 + 98;
  TF* sRow = reinterpret_cast<TF*>(fsm) + (size_t)g * per;
  TF* sScl = sRow + (size_t)R.max_row_blocks * 49;
  TF* sAug = sScl + 49;
  const int64_t r0 = R.sd_row[s];
  const int64_t* irow = R.item_row + R.sd_item[s];
  for (int p = 0; p <= D; ++p) {
    const int nit = 1 << (D - p);
    if (g < nit) {
      const int it = (1 << (D + 1)) - (1 << (D - p + 1)) + g;
      const int64_t qb = r0 + (it == 0 ? 0 : irow[it - 1]), qe = r0 + irow[it];
      for (int64_t q = qb; q < qe; ++q) {
        const int64_t rp = R.row_ptr[q];
        const int nblk = (int)(R.row_ptr[q + 1] - rp);
        const int64_t e0 = R.lent_ptr[q], e1 = R.lent_ptr[q + 1];
        for (int idx = lt; idx < 49 * nblk; idx += gs) sRow[idx] = fac[49 * rp + idx];
        group_sync(g, gs);
        for (int64_t e = e0; e < e1; ++e) {
          TF* Aik = sRow + 49 * (R.lent_pos[e] - rp);
          const TF* Dk = fac + 49 * R.lent_kdiag[e];
          for (int x = lt; x < 49; x += gs) {
            const int r = x / 7, c = x - 7 * r;
            TF v = TF(0);
#pragma unroll
            for (int mm = 0; mm < 7; ++mm) v += Aik[7 * r + mm] * Dk[7 * mm + c];
            sScl[x] = v;
          }
          group_sync(g, gs);
          for (int x = lt; x < 49; x += gs) Aik[x] = sScl[x];
          const int64_t ub = R.upd_ptr[e];
          const int ntask = 7 * (int)(R.upd_ptr[e + 1] - ub);
          for (int t = lt; t < ntask; t += gs) {
            const int u = t / 7, cc = t - 7 * u;
            TF* Aij = sRow + 49 * (R.upd_tgt[ub + u] - rp) + cc;
            const TF* Akj = fac + 49 * R.upd_src[ub + u] + cc;
            TF col[7];
#pragma unroll
            for (int mm = 0; mm < 7; ++mm) col[mm] = Akj[7 * mm];
#pragma unroll
            for (int rr = 0; rr < 7; ++rr) {
              TF acc = Aij[7 * rr];
#pragma unroll
              for (int mm = 0; mm < 7; ++mm) acc -= sScl[7 * rr + mm] * col[mm];
              Aij[7 * rr] = acc;
            }
          }
          group_sync(g, gs);
        }
        if (lt < 32) warp_invert7<TF>(sRow + 49 * (R.diag[q] - rp), sAug, err);
        group_sync(g, gs);
        for (int idx = lt; idx < 49 * nblk; idx += gs) fac[49 * rp + idx] = sRow[idx];
        group_sync(g, gs);
      }
    }
    __syncthreads();
  }
}

// Batched RAS apply: grid = one CTA per subdomain; 8-lane groups own one row
// (lane c < 7 computes component c). work holds the subdomain vector.
template <class TF>
__global__ void __launch_bounds__(256) k_ras_apply(RasDev R, const TF* __restrict__ fac,
                                                   const double* __restrict__ rin, TF* __restrict__ work,
                                                   double* __restrict__ z, float* __restrict__ z32,
                                                   const int* __restrict__ guard) {
  if (guard && *guard == 0) return;
  const int s = blockIdx.x;
  const int64_t r0 = R.sd_row[s], m = R.sd_row[s + 1] - r0;
  const int grp = threadIdx.x >> 3, c = threadIdx.x & 7;
  const int ngrp = blockDim.x >> 3;
  TF* w = work + 7 * r0;
  // restriction R_i^delta r
  for (int64_t idx = threadIdx.x; idx < 7 * m; idx += blockDim.x) {
    const int64_t q = idx / 7;
    const int cc = (int)(idx - 7 * q);
    w[idx] = (TF)rin[7 * (int64_t)R.gnode[r0 + q] + cc];
  }
  __syncthreads();
  // forward solve with the unit lower factor
  for (int64_t l = R.sd_lvlL[s]; l < R.sd_lvlL[s + 1]; ++l) {
    const int64_t lb = R.lvlL_ptr[l], le = R.lvlL_ptr[l + 1];
    for (int64_t ri = lb + grp; ri < le; ri += ngrp) {
      const int64_t q = R.lvlL_rows[ri];
      const int64_t gq = r0 + q;
      if (c < 7) {
        TF acc = w[7 * q + c];
        for (int64_t e = R.row_ptr[gq]; e < R.diag[gq]; ++e) {
          const TF* A = fac + 49 * e + 7 * c;
          const TF* xk = work + 7 * (int64_t)R.col[e];
#pragma unroll
          for (int mm = 0; mm < 7; ++mm) acc -= A[mm] * xk[mm];
        }
        w[7 * q + c] = acc;
      }
    }
    __syncthreads();
  }
  // backward solve with the upper factor and inverted pivots
  for (int64_t l = R.sd_lvlU[s]; l < R.sd_lvlU[s + 1]; ++l) {
    const int64_t lb = R.lvlU_ptr[l], le = R.lvlU_ptr[l + 1];
    // rounds are uniform across the warp so that every lane joins the shuffles
    for (int64_t base = lb; base < le; base += ngrp) {
      const int64_t ri = base + grp;
      const bool act = ri < le;
      const int64_t q = act ? R.lvlU_rows[ri] : 0;
      const int64_t gq = r0 + q;
      TF acc = TF(0);
      if (act && c < 7) {
        acc = w[7 * q + c];
        for (int64_t e = R.diag[gq] + 1; e < R.row_ptr[gq + 1]; ++e) {
          const TF* A = fac + 49 * e + 7 * c;
          const TF* xk = work + 7 * (int64_t)R.col[e];
#pragma unroll
          for (int mm = 0; mm < 7; ++mm) acc -= A[mm] * xk[mm];
        }
      }
      // z_q = D_q^{-1} t: gather t from the 7 lanes of the group
      TF tv[7];
#pragma unroll
      for (int mm = 0; mm < 7; ++mm) tv[mm] = __shfl_sync(0xffffffffu, acc, (threadIdx.x & 31 & ~7) + mm);
      if (act && c < 7) {
        const TF* Dinv = fac + 49 * R.diag[gq] + 7 * c;
        TF zz = TF(0);
#pragma unroll
        for (int mm = 0; mm < 7; ++mm) zz += Dinv[mm] * tv[mm];
        w[7 * q + c] = zz;
      }
    }
    __syncthreads();
  }
  // restricted prolongation (R_i^0)^T: owned rows only
  for (int64_t idx = threadIdx.x; idx < 7 * m; idx += blockDim.x) {
    const int64_t q = idx / 7;
    const int cc = (int)(idx - 7 * q);
    if (R.owned[r0 + q]) {
      z[7 * (int64_t)R.gnode[r0 + q] + cc] = (double)w[idx];
      if (z32) z32[7 * (int64_t)R.gnode[r0 + q] + cc] = (float)w[idx];
    }
  }
}

}  // namespace

template <class TV>
void launch_bsr_spmv(int64_t n, const int64_t* row_ptr, const int32_t* col, const TV* vals, const TV* x,
                     double* y, int threads_per_row, const int* guard, cudaStream_t s) {
  if (threads_per_row == 16)
    k_bsr_spmv<TV, 2><<<grid_for(16 * n, 256), 256, 0, s>>>(n, row_ptr, col, vals, x, y, guard);
  else
    k_bsr_spmv<TV, 4><<<grid_for(32 * n, 256), 256, 0, s>>>(n, row_ptr, col, vals, x, y, guard);
}

void launch_to_float(int64_t n, const double* x, float* y, const int* guard, cudaStream_t s) {
  k_to_float<<<grid_for((n + 1) / 2, 256), 256, 0, s>>>(n, x, y, guard);
}

template <class TF, class TJ>
void launch_ras_extract(const RasDev& r, const TJ* vals, TF* fac, cudaStream_t s) {
  k_ras_extract<TF, TJ><<<grid_for(32 * r.nblocks, 256), 256, 0, s>>>(r.nblocks, r.gblk, vals, fac);
}

template <class TF>
size_t ras_factor_smem(const RasDev& r, int mode) {
  if (mode == 4)
    return PIPE_HEAD + PIPE_SCL + (size_t)r.pipe_slots * (r.pipe_meta + r.pipe_data) +
           (size_t)2 * r.max_row_blocks * 49 * sizeof(TF);
  if (mode == 3)  // one row, scaled block and inversion scratch per group
    return ((size_t)1 << r.max_depth) * (((size_t)r.max_row_blocks + 1) * 49 + 98) * sizeof(TF);
  size_t blocks = (size_t)r.max_row_blocks + 1;  // the row and the scaled L block
  if (mode == 0) blocks += (size_t)r.max_row_lent + 2 * (size_t)r.max_entry_upd;
  if (mode == 1) blocks += 2 * (size_t)r.max_entry_upd;
  return (blocks * 49 + 98) * sizeof(TF);  // + the 7 x 14 inversion scratch
}

// Fit check of a factorisation mode. The automatic choice on one-piece subdomains is
// the pipelined kernel (4) where its slots fit as fsi_create asks, else the leanest
// mode (2): of modes 0 to 2 it is the fastest, because the smaller footprint lets more
// subdomain CTAs share an SM, which hides the latency of the pivot and source reads
// better than prefetching them does.
template <class TF>
bool ras_factor_fits(const RasDev& r, int mode) {
  return ras_factor_smem<TF>(r, mode) <= FACTOR_SMEM_MAX;
}

// (the shared-memory limit is the kernel's, not the launch's: set to what one context needs,
// another thread's launch with more could be refused)
template <class TF, int MODE>
void launch_factor_mode(const RasDev& r, TF* fac, int32_t* err, size_t smem, cudaStream_t s) {
  cudaFuncSetAttribute(k_ras_factor_cta<TF, MODE>, cudaFuncAttributePreferredSharedMemoryCarveout,
                       (int)cudaSharedmemCarveoutMaxShared);
  cudaFuncSetAttribute(k_ras_factor_cta<TF, MODE>, cudaFuncAttributeMaxDynamicSharedMemorySize, (int)FACTOR_SMEM_MAX);
  k_ras_factor_cta<TF, MODE><<<r.np, 256, smem, s>>>(r, fac, err);
}

template <class TF>
void launch_ras_factor(const RasDev& r, TF* fac, int32_t* err, cudaStream_t s) {
  const size_t smem = ras_factor_smem<TF>(r, r.factor_mode);
  switch (r.factor_mode) {
    case 0: launch_factor_mode<TF, 0>(r, fac, err, smem, s); break;
    case 1: launch_factor_mode<TF, 1>(r, fac, err, smem, s); break;
    case 2: launch_factor_mode<TF, 2>(r, fac, err, smem, s); break;
    case 3:
      cudaFuncSetAttribute(k_ras_factor_nd<TF>, cudaFuncAttributePreferredSharedMemoryCarveout,
                           (int)cudaSharedmemCarveoutMaxShared);
      cudaFuncSetAttribute(k_ras_factor_nd<TF>, cudaFuncAttributeMaxDynamicSharedMemorySize, (int)FACTOR_SMEM_MAX);
      k_ras_factor_nd<TF><<<r.np, 256, smem, s>>>(r, fac, err);
      break;
    case 4:
      cudaFuncSetAttribute(k_ras_factor_pipe<TF>, cudaFuncAttributePreferredSharedMemoryCarveout,
                           (int)cudaSharedmemCarveoutMaxShared);
      cudaFuncSetAttribute(k_ras_factor_pipe<TF>, cudaFuncAttributeMaxDynamicSharedMemorySize, (int)FACTOR_SMEM_MAX);
      k_ras_factor_pipe<TF><<<r.np, PIPE_THREADS<TF> + 64, smem, s>>>(r, fac, err);
      break;
    default: break;  // fsi_create rejects such plans
  }
}

template size_t ras_factor_smem<float>(const RasDev&, int);
template size_t ras_factor_smem<double>(const RasDev&, int);
template bool ras_factor_fits<float>(const RasDev&, int);
template bool ras_factor_fits<double>(const RasDev&, int);

template <class TF>
void launch_ras_apply(const RasDev& r, const TF* fac, const double* rin, TF* work, double* z, float* z32,
                      const int* guard, cudaStream_t s) {
  k_ras_apply<TF><<<r.np, 256, 0, s>>>(r, fac, rin, work, z, z32, guard);
}

template void launch_bsr_spmv<double>(int64_t, const int64_t*, const int32_t*, const double*, const double*,
                                      double*, int, const int*, cudaStream_t);
template void launch_bsr_spmv<float>(int64_t, const int64_t*, const int32_t*, const float*, const float*, double*,
                                     int, const int*, cudaStream_t);
template void launch_ras_extract<double, double>(const RasDev&, const double*, double*, cudaStream_t);
template void launch_ras_extract<float, float>(const RasDev&, const float*, float*, cudaStream_t);
template void launch_ras_factor<double>(const RasDev&, double*, int32_t*, cudaStream_t);
template void launch_ras_factor<float>(const RasDev&, float*, int32_t*, cudaStream_t);
template void launch_ras_apply<double>(const RasDev&, const double*, const double*, double*, double*, float*,
                                       const int*, cudaStream_t);
template void launch_ras_apply<float>(const RasDev&, const float*, const double*, float*, double*, float*,
                                      const int*, cudaStream_t);

}  // namespace fsi
