// FP64 vector kernels of the batched Krylov loop. The unknowns of P independent
// problems are stored one after the other; every reduction is segmented by
// problem: a fixed table of chunks (each inside one problem) is reduced by one
// block per chunk, and the last block of a problem to finish (a per-problem
// counter) sums that problem's chunk partials in fixed order, so results are
// bitwise reproducible run to run, independent problems never mix, and a
// reduction is one launch (a multi-dot's groups of 8 vectors side by side).
// Per-problem Arnoldi scalars: H (column-major (m+1) x m per problem), g, Givens
// cs/sn, residual estimates, stop flags.
//
// Kernels that run inside a captured GMRES cycle take a guard pointer: while
// *guard == 0 (every problem has converged or broken down) they return at once,
// so the rest of the captured cycle costs only its launches.
#include <cuda_runtime.h>

#include "kernels.cuh"

namespace fsi {

namespace {

constexpr int RB = 256;   // threads per reduction block
constexpr int MD = 8;     // vectors per multi-dot pass

__device__ __forceinline__ bool off(const int* guard) { return guard && *guard == 0; }

__device__ __forceinline__ double warp_sum(double v) {
#pragma unroll
  for (int o = 16; o > 0; o >>= 1) v += __shfl_xor_sync(0xffffffffu, v, o);
  return v;
}

// Sums of v[0..W) over the warp's lanes: every step halves the vectors a lane
// still carries, so 8 vectors take 9 FP64 additions instead of 40 (the FP64 pipe
// bounds the dots; the additions of a plain butterfly per vector cost as much as the
// products: 8 vectors of 326k dofs 31 -> 22 us). Afterwards v[0] of the lanes with
// lane / (32 / W) == k holds vector k's sum.
template <int W>
__device__ __forceinline__ void warp_sums(double (&v)[W]) {
  const int lane = threadIdx.x & 31;
  int o = 16;
#pragma unroll
  for (int h = W / 2; h >= 1; h >>= 1, o >>= 1) {
    const bool up = lane & o;
#pragma unroll
    for (int i = 0; i < h; ++i) {
      const double mine = up ? v[i + h] : v[i], other = up ? v[i] : v[i + h];
      v[i] = mine + __shfl_xor_sync(0xffffffffu, other, o);
    }
  }
  for (; o >= 1; o >>= 1) v[0] += __shfl_xor_sync(0xffffffffu, v[0], o);
}

// The norm of a Gram-Schmidt step's new vector from its second pass (k_seg_mdot):
// after w1 = w0 - V h1 the second pass's dots h2 = V^T w1 come with ||w1||^2 (the
// self product), and since V is orthonormal, ||w1 - V h2||^2 = ||w1||^2 - ||h2||^2.
// The second update then scales in the same sweep (k_seg_maxpy with scal), so the
// step needs no norm or scaling sweep. Where ||w1||^2 - ||h2||^2 keeps at least 3/4
// of ||w1||^2 (the subtraction then loses under two bits) hsub[p * ldsub] is its
// square root and inv[p] the reciprocal (0 for a zero norm); elsewhere (only as a
// Krylov space is exhausted; for every problem with force = 1, tests of that path)
// inv[p] = 1, unsafe[p] = 1 and *flag = 1: the second update (k_seg_maxpy) then forms the
// norm of the updated vector and k_seg_givens scales by it. A problem that has already
// stopped needs no norm: its vector is zeroed (inv[p] = 0).

// one warp: q = ||h2||^2 and s = ||w1||^2, written by other blocks of this launch
__device__ void new_norm(const NewNorm& N, int p, const double* h, int nv) {
  const int lane = threadIdx.x & 31;
  const double s = __ldcg(h + nv);
  double q = 0.0;
  for (int k = lane; k < nv; k += 32) {
    const double v = __ldcg(h + k);
    q += v * v;
  }
  q = warp_sum(q);
  if (lane == 0) {
    const double b2 = s - q;
    if (!N.force && b2 >= 0.75 * s) {
      const double b = sqrt(b2);
      N.hsub[(int64_t)p * N.ldsub] = b;
      N.inv[p] = b > 0.0 ? 1.0 / b : 0.0;
      N.unsafe[p] = 0;
    } else {
      const int a = N.active[p];
      N.inv[p] = a ? 1.0 : 0.0;
      N.unsafe[p] = a;
      if (a) *N.flag = 1;
    }
  }
}

// The partials of chunk c for the vectors of group g, 8g .. 8g + W - 1 (those below nv),
// and, in the last block of problem p for group g, the sums of the problem's partials
// (one warp per vector, lanes over the chunks in fixed order). Each thread takes U
// elements per trip (loads in flight).
template <int W, int U>
__device__ __forceinline__ void dots(const SegDev& sg, int32_t nv, int g, int n_groups, const double* __restrict__ V,
                                     int64_t ldv, const double* __restrict__ w, double* __restrict__ partial,
                                     double* __restrict__ out, int32_t ldo, int take_sqrt, int nself,
                                     const NewNorm& N) {
  __shared__ double red[W][RB / 32];
  __shared__ int s_last;
  const int c = blockIdx.x;
  const int k0 = g * MD;
  const int64_t i0 = sg.chunk_beg[c], i1 = sg.chunk_beg[c + 1];
  double acc[W];
#pragma unroll
  for (int k = 0; k < W; ++k) acc[k] = 0.0;
  const int nvv = nv - nself;  // vectors of V; the rest is w itself
  // vector k of this group: V_{k0+k} while k0 + k < nvv, else w (the self product)
  const double* src[W];
#pragma unroll
  for (int k = 0; k < W; ++k) src[k] = (V && k0 + k < nvv) ? V + (int64_t)(k0 + k) * ldv : w;
  for (int64_t i = i0 + threadIdx.x; i < i1; i += U * RB) {
    double wv[U], v[U][W];
#pragma unroll
    for (int u = 0; u < U; ++u) {
      const int64_t iu = i + u * RB;
      const bool in = iu < i1;
      wv[u] = in ? w[iu] : 0.0;
#pragma unroll
      for (int k = 0; k < W; ++k) v[u][k] = (k0 + k < nv && in) ? src[k][iu] : 0.0;
    }
#pragma unroll
    for (int u = 0; u < U; ++u)
#pragma unroll
      for (int k = 0; k < W; ++k)
        if (k0 + k < nv) acc[k] += v[u][k] * wv[u];
  }
  const int warp = threadIdx.x >> 5, lane = threadIdx.x & 31;
  warp_sums<W>(acc);
  if (lane % (32 / W) == 0) red[lane / (32 / W)][warp] = acc[0];
  __syncthreads();
  // the 8 warps' sums of vector k: lanes 8 k .. 8 k + 7 of the first W / 4 (at least one) warps
  if (threadIdx.x < (W < 4 ? 32 : 8 * W)) {
    const int k = threadIdx.x >> 3;
    double v = k < W ? red[k][threadIdx.x & 7] : 0.0;
#pragma unroll
    for (int o = 4; o >= 1; o >>= 1) v += __shfl_xor_sync(0xffffffffu, v, o);
    if (k < W && (threadIdx.x & 7) == 0 && k0 + k < nv) partial[(int64_t)c * nv + k0 + k] = v;
  }
  // publish the partials, then count this block in
  __threadfence();
  __syncthreads();
  const int p = sg.node_prob[i0 / 7];
  const int64_t c0 = sg.prob_chunk[p], c1 = sg.prob_chunk[p + 1];
  int* cnt = sg.counter + (int64_t)p * SEG_COUNTERS;
  if (threadIdx.x == 0) s_last = atomicAdd(cnt + g, 1) == (int)(c1 - c0) - 1;
  __syncthreads();
  if (!s_last) return;
  __threadfence();
  const int k = k0 + warp;
  if (warp < W && k < nv) {
    double v = 0.0;
    for (int64_t cc = c0 + lane; cc < c1; cc += 32) v += __ldcg(partial + cc * nv + k);
    v = warp_sum(v);
    if (lane == 0) out[(int64_t)p * ldo + k] = take_sqrt ? sqrt(v) : v;
  }
  if (threadIdx.x == 0) cnt[g] = 0;
  if (!N.hsub) return;
  // the last of the problem's groups takes the norm: publish the sums, count the group in
  __threadfence();
  __syncthreads();
  if (warp > 0) return;
  int last = 0;
  if (lane == 0) last = n_groups == 1 || atomicAdd(cnt + SEG_GROUPS, 1) == n_groups - 1;
  if (!__shfl_sync(0xffffffffu, last, 0)) return;
  __threadfence();
  new_norm(N, p, out + (int64_t)p * ldo, nvv);
  if (lane == 0) cnt[SEG_GROUPS] = 0;
}

// out[p * ldo + k] = sum over the dofs of problem p of V_k . w (V null: w . w,
// and take_sqrt gives the 2-norm). With nself = 1 there is one more output, index
// nv - 1: w . w itself. Block (c, g) takes chunk c and the g-th group of 8 vectors;
// the last group has W of them at most (W the next power of two).
// Bound by the FP64 pipe (one FMA per loaded operand) or, for narrow groups, by
// latency: the full groups take W = 8, U = 2, a partial last group a narrower W and a
// deeper U (fewer products, more loads in flight). All groups and the new norm in one
// launch: as two launches and one more for the norm the narrow group ran after the full
// ones with most of the chip idle, and each launch of the cycle's graph costs 1.4 to 4 us
// (seven launches per GMRES iteration instead of eleven, the same bits: a mixed step of the
// 46,657-node tube 157.7 -> 152.7 ms, an FP64 step of the 12 x 8 x 4 tube 100.6 -> 98.2 ms; a
// step's time depends on its random state, both sides are of the same one).
template <int W, int U>
__global__ void __launch_bounds__(RB) k_seg_mdot(SegDev sg, int32_t nv, const double* __restrict__ V, int64_t ldv,
                                                 const double* __restrict__ w, double* __restrict__ partial,
                                                 double* __restrict__ out, int32_t ldo, int take_sqrt, int nself,
                                                 NewNorm N, const int* guard) {
  if (off(guard)) return;
  const int g = blockIdx.y, G = gridDim.y;
  if (W < MD && g < G - 1)
    dots<MD, 2>(sg, nv, g, G, V, ldv, w, partial, out, ldo, take_sqrt, nself, N);
  else
    dots<W, U>(sg, nv, g, G, V, ldv, w, partial, out, ldo, take_sqrt, nself, N);
}

// The second update where some problem's norm is unsafe, chunk by chunk: as k_seg_maxpy,
// and for the unsafe problems hsub[p * ldsub] = norms[p] = ||w_p|| of the updated vector
// (chunk partials, summed by the last block of the problem in fixed order).
__device__ __noinline__ void maxpy_norm(const SegDev* sgp, int32_t nv, const double* V, int64_t ldv, const double* h,
                                        int32_t ldh, double* w, const double* scal, const NewNorm* Np,
                                        double* partial) {
  __shared__ double red[RB / 32];
  __shared__ int s_last;
  const SegDev& sg = *sgp;
  const NewNorm& N = *Np;
  const int warp = threadIdx.x >> 5, lane = threadIdx.x & 31;
  for (int64_t c = blockIdx.x; c < sg.n_chunks; c += gridDim.x) {
    const int64_t i0 = sg.chunk_beg[c], i1 = sg.chunk_beg[c + 1];
    const int p = sg.node_prob[i0 / 7];
    const double* hp = h + (int64_t)p * ldh;
    const double a = scal[p];
    double q = 0.0;
    for (int64_t i = i0 + threadIdx.x; i < i1; i += blockDim.x) {
      double s = w[i];
      for (int k = 0; k < nv; ++k) s -= hp[k] * V[(int64_t)k * ldv + i];
      w[i] = s * a;
      q += s * s;
    }
    if (!N.unsafe[p]) continue;
    q = warp_sum(q);
    if (lane == 0) red[warp] = q;
    __syncthreads();
    if (threadIdx.x == 0) {
      for (int k = 1; k < RB / 32; ++k) q += red[k];
      partial[c] = q;
      __threadfence();
      s_last = atomicAdd(sg.counter + (int64_t)p * SEG_COUNTERS, 1) == (int)(sg.prob_chunk[p + 1] - sg.prob_chunk[p]) - 1;
    }
    __syncthreads();
    if (s_last && warp == 0) {
      __threadfence();
      double v = 0.0;
      for (int64_t cc = sg.prob_chunk[p] + lane; cc < sg.prob_chunk[p + 1]; cc += 32) v += __ldcg(partial + cc);
      v = warp_sum(v);
      if (lane == 0) {
        N.hsub[(int64_t)p * N.ldsub] = N.norms[p] = sqrt(v);
        sg.counter[(int64_t)p * SEG_COUNTERS] = 0;
      }
    }
    __syncthreads();
  }
}

// w_i -= sum_k h[p(i)][k] V_k[i], then (scal non-null) w_i *= scal[p(i)]. N.flag (optional): the
// first update (no scal) clears it, the second takes the form above where it is set.
__global__ void __launch_bounds__(RB, 8) k_seg_maxpy(const __grid_constant__ SegDev sg, int64_t n, int32_t nv,
                                                  const double* __restrict__ V, int64_t ldv,
                                                  const double* __restrict__ h, int32_t ldh, double* __restrict__ w,
                                                  const double* __restrict__ scal, const int* guard,
                                                  const __grid_constant__ NewNorm N, double* partial) {
  if (N.flag && !scal && blockIdx.x == 0 && threadIdx.x == 0) *N.flag = 0;
  if (off(guard)) return;
  if (N.flag && scal && *N.flag) {
    maxpy_norm(&sg, nv, V, ldv, h, ldh, w, scal, &N, partial);
    return;
  }
  for (int64_t i = blockIdx.x * (int64_t)blockDim.x + threadIdx.x; i < n; i += (int64_t)gridDim.x * blockDim.x) {
    const int p = sg.node_prob[i / 7];
    const double* hp = h + (int64_t)p * ldh;
    double s = w[i];
    for (int k = 0; k < nv; ++k) s -= hp[k] * V[(int64_t)k * ldv + i];
    w[i] = scal ? s * scal[p] : s;
  }
}

// y_i = x_i / scal[p(i) * lds] (0 where the scale is 0). The reciprocal is
// formed once per problem a thread meets (consecutive elements of a thread
// mostly share their problem), not once per element: y_i = x_i * (1 / a).
__global__ void k_seg_scale_inv(SegDev sg, int64_t n, const double* __restrict__ x, const double* __restrict__ scal,
                                int32_t lds, double* __restrict__ y, const int* guard) {
  if (off(guard)) return;
  int pc = -1;
  double inv = 0.0;
  for (int64_t i = blockIdx.x * (int64_t)blockDim.x + threadIdx.x; i < n; i += (int64_t)gridDim.x * blockDim.x) {
    const int p = sg.node_prob[i / 7];
    if (p != pc) {
      const double a = scal[(int64_t)p * lds];
      inv = a != 0.0 ? 1.0 / a : 0.0;
      pc = p;
    }
    y[i] = x[i] * inv;
  }
}

// start of a cycle for every problem: g = beta e_1, active while beta > target
__global__ void k_seg_cycle_init(int32_t P, double* __restrict__ g, int32_t ldg, const double* __restrict__ beta,
                                 const double* __restrict__ target, int* __restrict__ active, int* __restrict__ kcols,
                                 int* __restrict__ any) {
  __shared__ int s_any;
  if (threadIdx.x == 0) s_any = 0;
  __syncthreads();
  for (int p = threadIdx.x; p < P; p += blockDim.x) {
    for (int k = 0; k < ldg; ++k) g[(int64_t)p * ldg + k] = k == 0 ? beta[p] : 0.0;
    const int a = beta[p] > target[p] ? 1 : 0;
    active[p] = a;
    kcols[p] = 0;
    if (a) atomicOr(&s_any, 1);
  }
  __syncthreads();
  if (threadIdx.x == 0) *any = s_any;
}

// Selective reorthogonalisation (the criterion of Daniel, Gragg, Kaufman and
// Stewart, 1976): after one classical Gram-Schmidt pass, a second pass is needed
// where the pass removed more than 1 - 1/sqrt(2) of the vector's norm, i.e.
// where ||w_after||^2 < ||w_before||^2 / 2. For every active problem p: s0 =
// ||w_before||^2 (ws[p * lda]), t = ||w_after|| (nrm[p * ldn]); the second-pass
// coefficients hb[p][0..j] are zeroed (a second pass, if it runs, overwrites
// them); *flag = some active problem needs the second pass.
__global__ void k_seg_reorth_decide(int32_t P, const double* __restrict__ ws, const double* __restrict__ nrm,
                                    int32_t ldn, double* __restrict__ hb, int32_t lda, int32_t j,
                                    const int* __restrict__ active, int* __restrict__ flag) {
  __shared__ int s_any;
  if (threadIdx.x == 0) s_any = 0;
  __syncthreads();
  for (int p = threadIdx.x; p < P; p += blockDim.x) {
    for (int i = 0; i <= j; ++i) hb[(int64_t)p * lda + i] = 0.0;
    const double s0 = ws[(int64_t)p * lda], t = nrm[(int64_t)p * ldn];
    if (active[p] && t * t < 0.5 * s0) atomicOr(&s_any, 1);
  }
  __syncthreads();
  if (threadIdx.x == 0) *flag = s_any;
}

// Givens update of column j of every active problem's Hessenberg (formed here
// as the sum of the two Gram-Schmidt passes; H[j+1][j] is already in place): apply the
// previous rotations, form the one that zeroes H[j+1][j], rotate g; |g[j+1]|
// is that problem's GMRES residual. A problem stops at its target or when its
// Krylov space is exhausted (H[j+1][j] = 0). *any = some problem still active.
// One warp per problem (up to 32 at a time): the lanes read the column's sums and the
// rotations at once and hand them to the chain by shuffles (read one by one inside the
// chain of rotations they cost an L2 latency each: 7.3 -> 5.9 us for one problem).
//
// Where *flag (non-null; set by new_norm, a rare path), every block scales its part of the
// unsafe problems' w_p by 1 / norms[p], the norm of the updated vector (0 for a zero
// norm); block 0 alone does the rest. As launches of their own the norm and the scaling
// cost 2 us each a step for nothing; both in this kernel's one block took 829 us a step at
// 1.2 M unknowns where every norm is unsafe, this form 41 (the normal step is not slower).
__global__ void __launch_bounds__(1024) k_seg_givens(int32_t P, const double* __restrict__ ha,
                                                     const double* __restrict__ hb, int32_t lda,
                                                     double* __restrict__ H, int32_t ldh, int32_t m, int32_t j,
                                                     double* __restrict__ cs, double* __restrict__ sn,
                                                     double* __restrict__ g, double* __restrict__ res,
                                                     const double* __restrict__ target, int* __restrict__ active,
                                                     int* __restrict__ kcols, int* __restrict__ any, SegDev sg,
                                                     int64_t n, double* __restrict__ w,
                                                     const __grid_constant__ NewNorm N, const int* guard) {
  __shared__ int s_any;
  const int lane = threadIdx.x & 31;
  if (N.flag && *N.flag) {  // (not under the guard, *any, which block 0 may have stored already)
    int pc = -1;
    double inv = 1.0;
    for (int64_t i = blockIdx.x * (int64_t)blockDim.x + threadIdx.x; i < n; i += (int64_t)gridDim.x * blockDim.x) {
      const int p = sg.node_prob[i / 7];
      if (p != pc) {
        const double a = N.norms[p];
        inv = !N.unsafe[p] ? 1.0 : a != 0.0 ? 1.0 / a : 0.0;
        pc = p;
      }
      if (inv != 1.0) w[i] *= inv;
    }
  }
  if (blockIdx.x > 0 || off(guard)) return;  // *any is the guard, 0 already
  if (threadIdx.x == 0) s_any = 0;
  __syncthreads();
  for (int p = threadIdx.x >> 5; p < P; p += blockDim.x >> 5) {
    if (!active[p]) continue;
    double* h = H + (int64_t)p * ldh * m + (int64_t)j * ldh;
    double* c_ = cs + (int64_t)p * m;
    double* s_ = sn + (int64_t)p * m;
    double* gp = g + (int64_t)p * ldh;
    // entries lane and lane + 32 (restart <= 64)
    double hv[2], cv[2], sv[2];
#pragma unroll
    for (int t = 0; t < 2; ++t) {
      const int i = lane + 32 * t;
      hv[t] = i <= j ? ha[(int64_t)p * lda + i] + hb[(int64_t)p * lda + i] : 0.0;
      cv[t] = i < j ? c_[i] : 0.0;
      sv[t] = i < j ? s_[i] : 0.0;
    }
    const double sub = h[j + 1], gj = gp[j], tg = target[p];
    double a = __shfl_sync(0xffffffffu, hv[0], 0);
    for (int i = 0; i < j; ++i) {
      const double b = i + 1 < 32 ? __shfl_sync(0xffffffffu, hv[0], i + 1) : __shfl_sync(0xffffffffu, hv[1], i - 31);
      const double c = i < 32 ? __shfl_sync(0xffffffffu, cv[0], i) : __shfl_sync(0xffffffffu, cv[1], i - 32);
      const double s = i < 32 ? __shfl_sync(0xffffffffu, sv[0], i) : __shfl_sync(0xffffffffu, sv[1], i - 32);
      const double hi = c * a + s * b;
      a = -s * a + c * b;
      if (lane == (i & 31)) (i < 32 ? hv[0] : hv[1]) = hi;
    }
    const double r = hypot(a, sub);
    double c = 1.0, s = 0.0;
    if (r > 0.0) {
      c = a / r;
      s = sub / r;
    }
    if (lane == (j & 31)) (j < 32 ? hv[0] : hv[1]) = r;
#pragma unroll
    for (int t = 0; t < 2; ++t)
      if (lane + 32 * t <= j) h[lane + 32 * t] = hv[t];
    if (lane == 0) {
      c_[j] = c;
      s_[j] = s;
      h[j + 1] = 0.0;
      gp[j] = c * gj;
      gp[j + 1] = -s * gj;
      const double rn = fabs(s * gj);
      res[p] = rn;
      kcols[p] = j + 1;
      if (!(rn > tg) || sub == 0.0) active[p] = 0;
      else atomicOr(&s_any, 1);
    }
  }
  __syncthreads();
  if (threadIdx.x == 0) *any = s_any;
}

// y[p] = R_p^{-1} g[p] for each problem's kcols[p] x kcols[p] rotated Hessenberg, one
// warp per problem, column by column: lane i holds row i's right-hand side
__global__ void k_seg_lsq(int32_t P, const double* __restrict__ H, int32_t ldh, int32_t m,
                          const int* __restrict__ kcols, const double* __restrict__ g, double* __restrict__ y) {
  const int lane = threadIdx.x & 31;
  for (int p = (blockIdx.x * blockDim.x + threadIdx.x) >> 5; p < P; p += (gridDim.x * blockDim.x) >> 5) {
    const int k = kcols[p];
    const double* Hp = H + (int64_t)p * ldh * m;
    double* yp = y + (int64_t)p * m;
    double r[2];
#pragma unroll
    for (int t = 0; t < 2; ++t) r[t] = lane + 32 * t < k ? g[(int64_t)p * ldh + lane + 32 * t] : 0.0;
    for (int jj = k - 1; jj >= 0; --jj) {
      double c[2];  // column jj
#pragma unroll
      for (int t = 0; t < 2; ++t) c[t] = lane + 32 * t <= jj ? Hp[(int64_t)jj * ldh + lane + 32 * t] : 0.0;
      const double d = jj < 32 ? __shfl_sync(0xffffffffu, c[0], jj) : __shfl_sync(0xffffffffu, c[1], jj - 32);
      const double s = jj < 32 ? __shfl_sync(0xffffffffu, r[0], jj) : __shfl_sync(0xffffffffu, r[1], jj - 32);
      const double v = d != 0.0 ? s / d : 0.0;
      if (lane == 0) yp[jj] = v;
#pragma unroll
      for (int t = 0; t < 2; ++t)
        if (lane + 32 * t < jj) r[t] -= c[t] * v;
    }
  }
}

// x_i += sum_{q < kcols[p(i)]} y[p(i)][q] Z_q[i]
__global__ void k_seg_update_x(SegDev sg, int64_t n, const double* __restrict__ Z, int64_t ldz,
                               const double* __restrict__ y, int32_t m, const int* __restrict__ kcols,
                               double* __restrict__ x) {
  for (int64_t i = blockIdx.x * (int64_t)blockDim.x + threadIdx.x; i < n; i += (int64_t)gridDim.x * blockDim.x) {
    const int p = sg.node_prob[i / 7];
    const int k = kcols[p];
    const double* yp = y + (int64_t)p * m;
    double s = x[i];
    for (int q = 0; q < k; ++q) s += yp[q] * Z[(int64_t)q * ldz + i];
    x[i] = s;
  }
}

// out_i = x_i + alpha[p(i)] y_i
__global__ void k_seg_axpy(SegDev sg, int64_t n, const double* __restrict__ x, const double* __restrict__ alpha,
                           const double* __restrict__ y, double* __restrict__ out) {
  for (int64_t i = blockIdx.x * (int64_t)blockDim.x + threadIdx.x; i < n; i += (int64_t)gridDim.x * blockDim.x) {
    const double a = alpha[sg.node_prob[i / 7]];
    out[i] = a != 0.0 ? x[i] + a * y[i] : x[i];
  }
}

// out_i = mask[p(i)] ? 0 : -x_i
__global__ void k_seg_neg_masked(SegDev sg, int64_t n, const double* __restrict__ x, const int* __restrict__ mask,
                                 double* __restrict__ out) {
  for (int64_t i = blockIdx.x * (int64_t)blockDim.x + threadIdx.x; i < n; i += (int64_t)gridDim.x * blockDim.x)
    out[i] = mask[sg.node_prob[i / 7]] ? 0.0 : -x[i];
}

__global__ void k_axpby(int64_t n, double a, const double* __restrict__ x, double b, const double* __restrict__ y,
                        double* __restrict__ out) {
  for (int64_t i = blockIdx.x * (int64_t)blockDim.x + threadIdx.x; i < n; i += (int64_t)gridDim.x * blockDim.x)
    out[i] = a * x[i] + (b != 0.0 ? b * y[i] : 0.0);
}

__global__ void k_fill(int64_t n, double v, double* __restrict__ x) {
  for (int64_t i = blockIdx.x * (int64_t)blockDim.x + threadIdx.x; i < n; i += (int64_t)gridDim.x * blockDim.x)
    x[i] = v;
}

inline int grid_for(int64_t work, int block) {
  int64_t g = (work + block - 1) / block;
  const int64_t cap = 152 * 32;
  return (int)(g < 1 ? 1 : (g > cap ? cap : g));
}

// one launch; W and U by the size r of the last group
void mdot(const SegDev& sg, int32_t n, const double* V, int64_t ldv, const double* w, double* partial, double* out,
          int32_t ldo, int take_sqrt, int nself, const NewNorm& N, const int* guard, cudaStream_t s) {
  const dim3 grid((unsigned)sg.n_chunks, (unsigned)((n + MD - 1) / MD));
  const int r = n % MD;
  if (r == 1)
    k_seg_mdot<1, 8><<<grid, RB, 0, s>>>(sg, n, V, ldv, w, partial, out, ldo, take_sqrt, nself, N, guard);
  else if (r == 2)
    k_seg_mdot<2, 4><<<grid, RB, 0, s>>>(sg, n, V, ldv, w, partial, out, ldo, take_sqrt, nself, N, guard);
  else if (r == 3 || r == 4)
    k_seg_mdot<4, 4><<<grid, RB, 0, s>>>(sg, n, V, ldv, w, partial, out, ldo, take_sqrt, nself, N, guard);
  else
    k_seg_mdot<8, 2><<<grid, RB, 0, s>>>(sg, n, V, ldv, w, partial, out, ldo, take_sqrt, nself, N, guard);
}

}  // namespace

void launch_seg_mdot(const SegDev& sg, int32_t nv, const double* V, int64_t ldv, const double* w, double* partial,
                     double* out, int32_t ldo, const int* guard, cudaStream_t s, int with_self) {
  mdot(sg, nv + with_self, V, ldv, w, partial, out, ldo, 0, with_self, NewNorm{}, guard, s);
}

void launch_seg_mdot_norm(const SegDev& sg, int32_t nv, const double* V, int64_t ldv, const double* w,
                          double* partial, double* out, int32_t ldo, const NewNorm& N, const int* guard,
                          cudaStream_t s) {
  mdot(sg, nv + 1, V, ldv, w, partial, out, ldo, 0, 1, N, guard, s);
}

void launch_seg_norm(const SegDev& sg, const double* x, double* partial, double* out, int32_t ldo,
                     const int* guard, cudaStream_t s) {
  mdot(sg, 1, nullptr, 0, x, partial, out, ldo, 1, 0, NewNorm{}, guard, s);
}

void launch_seg_reorth_decide(int32_t P, const double* ws, const double* nrm, int32_t ldn, double* hb, int32_t lda,
                              int32_t j, const int* active, int* flag, cudaStream_t s) {
  k_seg_reorth_decide<<<1, 256, 0, s>>>(P, ws, nrm, ldn, hb, lda, j, active, flag);
}

void launch_seg_maxpy(const SegDev& sg, int64_t n, int32_t nv, const double* V, int64_t ldv, const double* h,
                      int32_t ldh, double* w, const int* guard, cudaStream_t s, const double* scal, const NewNorm& N,
                      double* partial) {
  k_seg_maxpy<<<grid_for(n, RB), RB, 0, s>>>(sg, n, nv, V, ldv, h, ldh, w, scal, guard, N, partial);
}

void launch_seg_scale_inv(const SegDev& sg, int64_t n, const double* x, const double* scal, int32_t lds,
                          double* y, const int* guard, cudaStream_t s) {
  k_seg_scale_inv<<<grid_for(n, 256), 256, 0, s>>>(sg, n, x, scal, lds, y, guard);
}

void launch_seg_cycle_init(int32_t P, double* g, int32_t ldg, const double* beta, const double* target, int* active,
                           int* kcols, int* any, cudaStream_t s) {
  k_seg_cycle_init<<<1, 256, 0, s>>>(P, g, ldg, beta, target, active, kcols, any);
}

void launch_seg_givens(int32_t P, const double* a, const double* b, int32_t lda, double* H, int32_t ldh, int32_t m,
                       int32_t j, double* cs, double* sn, double* g, double* res, const double* target, int* active,
                       int* kcols, int* any, const SegDev& sg, int64_t n, double* w, const NewNorm& N,
                       const int* guard, cudaStream_t s) {
  // block 0 with a warp per problem; the blocks that scale (rarely) add up to at most two per SM
  const int warps = P < 32 ? P : 32;
  const int threads = 32 * (N.flag && warps < 8 ? 8 : warps);
  const int64_t blocks = N.flag ? (n + 8 * threads - 1) / (8 * threads) : 1;
  k_seg_givens<<<(int)(blocks < 304 ? blocks : 304), threads, 0, s>>>(P, a, b, lda, H, ldh, m, j, cs, sn, g, res,
                                                                      target, active, kcols, any, sg, n, w, N, guard);
}

void launch_seg_lsq(int32_t P, const double* H, int32_t ldh, int32_t m, const int* kcols, const double* g, double* y,
                    cudaStream_t s) {
  k_seg_lsq<<<(P + 1) / 2, 64, 0, s>>>(P, H, ldh, m, kcols, g, y);
}

void launch_seg_update_x(const SegDev& sg, int64_t n, const double* Z, int64_t ldz, const double* y, int32_t m,
                         const int* kcols, double* x, cudaStream_t s) {
  k_seg_update_x<<<grid_for(n, 256), 256, 0, s>>>(sg, n, Z, ldz, y, m, kcols, x);
}

void launch_seg_axpy(const SegDev& sg, int64_t n, const double* x, const double* alpha, const double* y, double* out,
                     cudaStream_t s) {
  k_seg_axpy<<<grid_for(n, 256), 256, 0, s>>>(sg, n, x, alpha, y, out);
}

void launch_seg_neg_masked(const SegDev& sg, int64_t n, const double* x, const int* mask, double* out,
                           cudaStream_t s) {
  k_seg_neg_masked<<<grid_for(n, 256), 256, 0, s>>>(sg, n, x, mask, out);
}

void launch_axpby(int64_t n, double a, const double* x, double b, const double* y, double* out, cudaStream_t s) {
  k_axpby<<<grid_for(n, 256), 256, 0, s>>>(n, a, x, b, y, out);
}

void launch_copy(int64_t n, const double* x, double* y, cudaStream_t s) {
  cudaMemcpyAsync(y, x, n * sizeof(double), cudaMemcpyDeviceToDevice, s);
}

void launch_fill(int64_t n, double v, double* x, cudaStream_t s) {
  k_fill<<<grid_for(n, 256), 256, 0, s>>>(n, v, x);
}

}  // namespace fsi
