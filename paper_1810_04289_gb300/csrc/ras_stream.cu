// Streamed RAS apply (Sec. 3, Eq. 16) for GB300: one CTA per subdomain; the packed
// factor streams through shared memory (1-D bulk copies, cp.async.bulk, guarded by
// mbarriers) past the subdomain vector, which stays there. The dependency chain of
// an ILU solve on an RCM-ordered subdomain is nearly the row count, so the rows are
// worked off one after the other (forward with the unit lower factor, then backward
// with the upper factor and inverted pivots) by one warp: lane 8 j + c takes row c
// of the blocks j, j + 4, ... of a row. Three kernels:
//   k_ras_apply_chain: subdomains in one piece (every ordering but the dissected);
//   k_ras_apply_team: the same where subdomains are few, four warps each;
//   k_ras_apply_stream: nested-dissection subdomains, one warp and ring per part.
//
// Packed layout (built by k_pack_factors after each factorisation), per subdomain:
//   L part: for every row in increasing order, its L blocks;
//   U part: for every row in decreasing order, its inverted pivot D_q^{-1}, then
//           its U blocks premultiplied and negated, -D_q^{-1} U_qj.
// Each packed block holds its 7 rows as 8-wide rows (the 7 entries, then the
// block's column), cut into 16-byte pieces: the first pieces of the 7 rows, then
// the second pieces, and so on, so that the 7 lanes of a block read consecutive 16
// bytes (8-wide rows in one piece put lanes c and c + 4 on the same banks). The
// subdomain vector in shared memory is 8 wide too.
//
// Every wait on an mbarrier is bounded; on timeout the kernel records
// FSI_ERR_TIMEOUT-style status in *err, drains (bounded) and returns.
#include <cuda_runtime.h>

#include <cstdint>

#include "kernels.cuh"
#include "setup.h"

namespace fsi {

namespace {

__device__ __forceinline__ uint32_t smem_u32(const void* p) {
  return (uint32_t)__cvta_generic_to_shared(p);
}

__device__ __forceinline__ void mbar_init(uint64_t* bar, uint32_t count) {
  asm volatile("mbarrier.init.shared::cta.b64 [%0], %1;" ::"r"(smem_u32(bar)), "r"(count) : "memory");
}

__device__ __forceinline__ void mbar_arrive_expect_tx(uint64_t* bar, uint32_t bytes) {
  asm volatile("mbarrier.arrive.expect_tx.shared::cta.b64 _, [%0], %1;" ::"r"(smem_u32(bar)), "r"(bytes)
               : "memory");
}

__device__ __forceinline__ bool mbar_try_wait(uint64_t* bar, uint32_t parity) {
  uint32_t ok;
  asm volatile(
      "{\n .reg .pred p;\n mbarrier.try_wait.parity.shared::cta.b64 p, [%1], %2;\n selp.u32 %0, 1, 0, p;\n}\n"
      : "=r"(ok)
      : "r"(smem_u32(bar)), "r"(parity)
      : "memory");
  return ok != 0;
}

// bounded wait: returns false if the barrier phase did not complete in time
__device__ __forceinline__ bool mbar_wait(uint64_t* bar, uint32_t parity) {
  for (uint32_t it = 0; it < (1u << 20); ++it)
    if (mbar_try_wait(bar, parity)) return true;
  return false;
}

__device__ __forceinline__ void bulk_g2s(void* dst, const void* src, uint32_t bytes, uint64_t* bar) {
  asm volatile(
      "cp.async.bulk.shared::cluster.global.mbarrier::complete_tx::bytes [%0], [%1], %2, [%3];" ::"r"(
          smem_u32(dst)),
      "l"(src), "r"(bytes), "r"(smem_u32(bar))
      : "memory");
}

template <class TF> struct Pack;
// packed block: 7 rows of 8 values in 16-byte pieces (see above)
template <class TF> struct Pack { static constexpr int stride = 56; };

// the block's column (a row of the subdomain)
template <class TF>
__device__ __forceinline__ int blk_col(const TF* blk) {
  constexpr int V = 16 / sizeof(TF);  // row 0's last value, in its last piece
  return *reinterpret_cast<const int*>(blk + (8 / V - 1) * 7 * V + V - 1);
}

// the 7-term product of row c of a packed block with the node vector x (8 wide):
// 16-byte loads of the row and of x
__device__ __forceinline__ float row7(const float* a, const float* x) {
  const float4 a0 = *reinterpret_cast<const float4*>(a), a1 = *reinterpret_cast<const float4*>(a + 28);
  const float4 x0 = *reinterpret_cast<const float4*>(x), x1 = *reinterpret_cast<const float4*>(x + 4);
  const float p01 = a0.x * x0.x + a0.y * x0.y;
  const float p23 = a0.z * x0.z + a0.w * x0.w;
  const float p45 = a1.x * x1.x + a1.y * x1.y;
  return (p01 + p23) + (p45 + a1.z * x1.z);
}
__device__ __forceinline__ double row7(const double* a, const double* x) {
  const double2 a0 = *reinterpret_cast<const double2*>(a), a1 = *reinterpret_cast<const double2*>(a + 14);
  const double2 a2 = *reinterpret_cast<const double2*>(a + 28), a3 = *reinterpret_cast<const double2*>(a + 42);
  const double2 x0 = *reinterpret_cast<const double2*>(x), x1 = *reinterpret_cast<const double2*>(x + 2);
  const double2 x2 = *reinterpret_cast<const double2*>(x + 4), x3 = *reinterpret_cast<const double2*>(x + 6);
  const double p01 = a0.x * x0.x + a0.y * x0.y;
  const double p23 = a1.x * x1.x + a1.y * x1.y;
  const double p45 = a2.x * x2.x + a2.y * x2.y;
  return (p01 + p23) + (p45 + a3.x * x3.x);
}

constexpr int NSTMAX = 8;  // most ring stages (runtime count R.nst)

// sum over blocks b in [0, nb) of (block b, row c) . w[col(b)], reduced over
// the warp: lane = 7 j + c handles blocks j, j + 4, ...; every block
// gathers its column index first so that all loads of a chunk are independent,
// then forms the 7-term products (16-byte loads of the block row and of the
// 8-wide node vector). The total lands in lanes 0..6.
template <class TF, int STR>
__device__ __forceinline__ TF row_dot(const TF* stg, int nb, const TF* w, int j, int c) {
  TF acc = TF(0);
  if (j < 4) {
    // 32-bit element offsets within the stage (a stage fits in shared memory)
    for (int b = j; b < nb; b += 16) {
      int cols[4];
#pragma unroll
      for (int i = 0; i < 4; ++i) {
        const int bi = b + 4 * i;
        cols[i] = bi < nb ? blk_col(stg + bi * STR) : -1;
      }
#pragma unroll
      for (int i = 0; i < 4; ++i) {
        if (cols[i] >= 0) acc += row7(stg + (b + 4 * i) * STR + (16 / (int)sizeof(TF)) * c, w + 8 * cols[i]);
      }
    }
  }
  acc += __shfl_down_sync(0xffffffffu, acc, 14);
  acc += __shfl_down_sync(0xffffffffu, acc, 7);
  return acc;
}

// One warp's stream of factor stages. The warp walks, in order, the segments of
// the items it solves: forward phases 0..D (its item's L blocks), then backward
// phases D..0 (its item's U blocks). Lane 0 keeps NST bulk copies in flight
// along that sequence, into the warp's own ring, across phase boundaries (the
// factor bytes do not depend on the solve, so the next phase's first stages
// arrive while the CTA waits at the phase barrier).
struct WarpFeed {
  int D, wi;         // nested-dissection depth of the subdomain, warp index
  int seg;           // producer: current segment 0 .. 2D+1 (2D+2 = done)
  int pos, end;      // producer: next block to issue and end block of the current segment
  int issued, used;  // stages issued / consumed by this warp
  int islot;         // producer: ring slot of the next issue (issued mod NST)
  int uslot, uphase; // consumer: ring slot of the next stage (used mod NST) and its mbarrier phase parity
};

// item of segment j for warp wi, or -1 when the warp has no item in that phase
__device__ __forceinline__ int seg_item(int D, int wi, int j) {
  const int p = j <= D ? j : 2 * D + 1 - j;
  if (wi >= (1 << (D - p))) return -1;
  return (1 << (D + 1)) - (1 << (D - p + 1)) + wi;
}

// lane 0: move the producer to the first segment at or after f.seg that has
// blocks left, loading its bounds once (segment changes are rare: 2D + 2 per apply)
__device__ __forceinline__ void feed_seek(WarpFeed& f, const int32_t* ib) {
  while (f.pos >= f.end && f.seg <= 2 * f.D + 1) {
    if (++f.seg > 2 * f.D + 1) break;
    const int it = seg_item(f.D, f.wi, f.seg);
    if (it >= 0) {
      const bool isL = f.seg <= f.D;
      f.pos = ib[4 * it + (isL ? 0 : 2)];
      f.end = ib[4 * it + (isL ? 1 : 3)];
    }
  }
}

// lane 0: issue the next stage of the warp's sequence (if any) into its ring slot.
// The slot was last read by this warp's lanes, whose loads completed before the
// __syncwarp that precedes every call.
template <class TF, int STR>
__device__ __forceinline__ void feed_issue(WarpFeed& f, const int32_t* ib, const TF* Lpack, const TF* Upack, TF* ring,
                                           uint64_t* full, int NST, int SB) {
  feed_seek(f, ib);
  if (f.pos >= f.end) return;
  const int nb = min(SB, f.end - f.pos);
  const int st = f.islot;
  const uint32_t bytes = (uint32_t)(nb * STR * sizeof(TF));
  mbar_arrive_expect_tx(&full[st], bytes);
  bulk_g2s(ring + (size_t)st * SB * STR, (f.seg <= f.D ? Lpack : Upack) + (size_t)f.pos * STR, bytes, &full[st]);
  f.pos += nb;
  f.issued++;
  if (++f.islot == NST) f.islot = 0;
}

// Multi-warp streamed RAS apply (Sec. 3, Eq. 16) on nested-dissection ordered
// subdomains (Sec. 4.5): one CTA per subdomain; in each phase of the forward
// solve (leaves, then the separators level by level up to the root's) every item
// of the phase is solved by its own warp, the items of a phase being independent
// (no edge and no fill between them); the backward solve runs the phases in
// reverse. (Subdomains of a few nodes are one item, depth 0: one warp.)
// Each warp is its own producer: lane 0 streams the packed factor blocks of the
// warp's items through a ring of NST stages of SB blocks (cp.async.bulk with
// mbarrier completion); the warp solves the rows of the current stage (rows may
// straddle stages) on the subdomain vector in shared memory.
template <class TF>
__global__ void __launch_bounds__(256) k_ras_apply_stream(RasStreamDev R, const double* __restrict__ rin,
                                                          double* __restrict__ z, float* __restrict__ z32,
                                                          int32_t* err, const int* __restrict__ guard) {
  if (guard && *guard == 0) return;
  constexpr int STR = Pack<TF>::stride;
  extern __shared__ __align__(128) unsigned char smem[];
  const int NST = R.nst;
  const int SB = R.stage_blocks;
  const int nwarps = blockDim.x >> 5;
  const int wi = threadIdx.x >> 5, lane = threadIdx.x & 31;
  uint64_t* bars = reinterpret_cast<uint64_t*>(smem);                     // [nwarps][NSTMAX]
  TF* rings = reinterpret_cast<TF*>(smem + 128 * ((nwarps * NSTMAX * 8 + 127) / 128));
  TF* ring = rings + (size_t)wi * NST * SB * STR;
  TF* w = rings + (size_t)nwarps * NST * SB * STR;
  unsigned short* Lcnt = reinterpret_cast<unsigned short*>(w + 8 * (size_t)R.max_rows);
  unsigned short* Ucnt = Lcnt + R.max_rows;
  uint64_t* full = bars + wi * NSTMAX;
  const int s = blockIdx.x;
  const int64_t r0 = R.sd_row[s];
  const int m = (int)(R.sd_row[s + 1] - r0);
  const int D = R.sd_depth[s];
  const int32_t* ib = R.item_blk + 4 * R.sd_item[s];        // per item: L begin, L end, U begin, U end
  const int64_t* irow = R.item_row + R.sd_item[s];          // per item: end row
  const TF* Lpack = reinterpret_cast<const TF*>(R.pack) + (size_t)R.L_off[s] * STR;
  const TF* Upack = reinterpret_cast<const TF*>(R.pack) + (size_t)R.U_off[s] * STR;

  if (lane == 0)
    for (int i = 0; i < NST; ++i) mbar_init(&full[i], 1);
  asm volatile("fence.mbarrier_init.release.cluster;" ::: "memory");
  // restriction R_i^delta r into shared memory
  for (int q = threadIdx.x; q < m; q += blockDim.x) {
    const double* src = rin + 7 * (int64_t)R.gnode[r0 + q];
    double v[7];
#pragma unroll
    for (int c = 0; c < 7; ++c) v[c] = src[c];
#pragma unroll
    for (int c = 0; c < 7; ++c) w[8 * q + c] = (TF)v[c];
    w[8 * q + 7] = TF(0);
    Lcnt[q] = (unsigned short)R.L_cnt[r0 + q];
    Ucnt[q] = (unsigned short)R.U_cnt[r0 + q];
  }
  __syncthreads();

  WarpFeed f{D, wi, -1, 0, 0, 0, 0, 0, 0, 0};
  const bool active = wi < (1 << D);
  if (active && lane == 0 && R.stall != 1)
    for (int k = 0; k < NST; ++k) feed_issue<TF, STR>(f, ib, Lpack, Upack, ring, full, NST, SB);
  f.issued = __shfl_sync(0xffffffffu, f.issued, 0);

  const int j = lane / 7, c = lane - 7 * (lane / 7);  // block slot 0..3 (4 = idle), component
  bool ok = R.stall != 2;
  // wait for the next stage of this warp's sequence; null on timeout, for the whole warp if
  // for one lane: the loops below end on it, and the lanes shuffle in them
  auto next_stage = [&]() -> const TF* {
    const int st = f.uslot;
    const bool lost = R.stall == 3 && lane == 1;
    if (!__all_sync(0xffffffffu, !lost && mbar_wait(&full[st], (uint32_t)f.uphase))) return nullptr;
    return ring + (size_t)st * SB * STR;
  };
  // the stage is consumed: lane 0 refills its slot with the next stage in line
  auto release = [&]() {
    __syncwarp();
    f.used++;
    if (++f.uslot == NST) {
      f.uslot = 0;
      f.uphase ^= 1;
    }
    if (lane == 0 && R.stall != 1) feed_issue<TF, STR>(f, ib, Lpack, Upack, ring, full, NST, SB);
    f.issued = __shfl_sync(0xffffffffu, f.issued, 0);
  };

  // forward: phases 0..D, w_q -= sum_k L_qk w_k over the rows of the warp's item
  for (int p = 0; p <= D; ++p) {
    const int it = seg_item(D, wi, p);
    if (it >= 0 && ok) {
      int q = it == 0 ? 0 : (int)irow[it - 1];
      const int qe = (int)irow[it];
      const int nLb = ib[4 * it + 1] - ib[4 * it];
      int rem = 0, done = 0;
      TF acc = TF(0);
      while (done < nLb) {
        const TF* stg = next_stage();
        if (!stg) { ok = false; break; }
        const int cap = min(SB, nLb - done);
        int pos = 0;
        if (rem > 0) {
          const int k = min(rem, cap);
          acc += row_dot<TF, STR>(stg, k, w, j, c);
          pos = k;
          rem -= k;
          if (rem == 0) {
            if (lane < 7) w[8 * q + lane] -= acc;
            __syncwarp();
            ++q;
          }
        }
        if (rem == 0) {
          for (; q < qe; ++q) {
            const int nb = Lcnt[q];
            if (pos + nb > cap) break;
            const TF a = row_dot<TF, STR>(stg + pos * STR, nb, w, j, c);
            if (lane < 7 && nb > 0) w[8 * q + lane] -= a;
            __syncwarp();
            pos += nb;
          }
          if (q < qe && pos < cap) {
            acc = row_dot<TF, STR>(stg + pos * STR, cap - pos, w, j, c);
            rem = Lcnt[q] - (cap - pos);
          }
        }
        done += cap;
        release();
      }
    }
    __syncthreads();
  }
  // backward: phases D..0, w_q = D_q^{-1} w_q - sum_j (D_q^{-1} U_qj) w_j: the
  // U stream holds, per row, the inverted pivot (column q: it multiplies the
  // forward result still in w_q) and then the blocks -D_q^{-1} U_qj, so a row is
  // one dot product over its blocks, as in the forward solve
  for (int p = D; p >= 0; --p) {
    const int it = seg_item(D, wi, 2 * D + 1 - p);
    if (it >= 0 && ok) {
      const int qb = it == 0 ? 0 : (int)irow[it - 1];
      int q = (int)irow[it] - 1;
      const int nUb = ib[4 * it + 3] - ib[4 * it + 2];
      int rem = 0, done = 0;
      TF acc = TF(0);
      while (done < nUb) {
        const TF* stg = next_stage();
        if (!stg) { ok = false; break; }
        const int cap = min(SB, nUb - done);
        int pos = 0;
        if (rem > 0) {
          const int k = min(rem, cap);
          acc += row_dot<TF, STR>(stg, k, w, j, c);
          pos = k;
          rem -= k;
          if (rem == 0) {
            if (lane < 7) w[8 * q + lane] = acc;
            __syncwarp();
            --q;
          }
        }
        if (rem == 0) {
          for (; q >= qb; --q) {
            const int nb = Ucnt[q];
            if (pos + nb > cap) break;
            const TF a = row_dot<TF, STR>(stg + pos * STR, nb, w, j, c);
            if (lane < 7) w[8 * q + lane] = a;
            __syncwarp();
            pos += nb;
          }
          if (q >= qb && pos < cap) {
            acc = row_dot<TF, STR>(stg + pos * STR, cap - pos, w, j, c);
            rem = Ucnt[q] - (cap - pos);
          }
        }
        done += cap;
        release();
      }
    }
    __syncthreads();
  }
  if (!ok) {
    // a wait gave up: record it and let this warp's copies still in flight land
    // (bounded) before the CTA exits
    if (lane == 0) {
      atomicExch(err, 2);
      for (int k = f.used; k < f.issued; ++k) mbar_wait(&full[k % NST], (k / NST) & 1);
    }
  }
  __syncthreads();
  // restricted prolongation (R_i^0)^T: owned rows only
  for (int q = threadIdx.x; q < m; q += blockDim.x) {
    if (R.owned[r0 + q]) {
      const int64_t g7 = 7 * (int64_t)R.gnode[r0 + q];
#pragma unroll
      for (int cc = 0; cc < 7; ++cc) z[g7 + cc] = (double)w[8 * q + cc];
      if (z32) {
#pragma unroll
        for (int cc = 0; cc < 7; ++cc) z32[g7 + cc] = (float)w[8 * q + cc];
      }
    }
  }
}

__device__ __forceinline__ int row_col(const float (&v)[8]) { return __float_as_int(v[7]); }
__device__ __forceinline__ int row_col(const double (&v)[8]) { return __double2loint(v[7]); }

__device__ __forceinline__ void load16(float* v, const float* p) {
  const float4 t = *reinterpret_cast<const float4*>(p);
  v[0] = t.x, v[1] = t.y, v[2] = t.z, v[3] = t.w;
}
__device__ __forceinline__ void load16(double* v, const double* p) {
  const double2 t = *reinterpret_cast<const double2*>(p);
  v[0] = t.x, v[1] = t.y;
}

// acc + (row . x): FP32 in row7's order, so that the chain and the ring kernel give the same bits
__device__ __forceinline__ float row_fma(const float (&a)[8], const float (&x)[8], float acc) {
  const float p01 = a[0] * x[0] + a[1] * x[1];
  const float p23 = a[2] * x[2] + a[3] * x[3];
  const float p45 = a[4] * x[4] + a[5] * x[5];
  return acc + ((p01 + p23) + (p45 + a[6] * x[6]));
}
__device__ __forceinline__ double row_fma(const double (&a)[8], const double (&x)[8], double acc) {
#pragma unroll
  for (int e = 0; e < 7; ++e) acc = fma(a[e], x[e], acc);
  return acc;
}

// Chain apply: one warp per subdomain, the host's entry codes (setup.h, StreamPlan)
// in place of row counts and ring arithmetic. What bounds it is the latency of the
// row chain: with 1,088 subdomains an SM holds 7 warps, and a row costs its
// instructions times 5 to 6 cycles each. So an entry (up to 16 blocks of a row,
// FP64 8) is straight-line code: all its vector loads together, then its products;
// the next entry's rows are read into registers during this entry's reduction;
// entries never straddle a stage, so their rows lie at fixed offsets; columns come
// with the rows, not by a load of their own. Two stages of whole entries, refilled
// by the warp's lane 0.
// Measured against the ring kernel on one-piece subdomains (same bits in mixed
// precision): 174k-node tree, ILU(2), 1,088 subdomains, mixed 757 -> 526 us (2.75 GB:
// 5.2 TB/s); 46,657-node tube, ILU(1), 512 subdomains, FP64 1,243 -> 870 us (the FP64
// pipe: one warp alone issues an FP64 instruction every 64 cycles, and a 4-block
// product takes 7 fused instructions where the tree sum took 10).
template <class TF>
__global__ void __launch_bounds__(32) k_ras_apply_chain(RasStreamDev R, const double* __restrict__ rin,
                                                        double* __restrict__ z, float* __restrict__ z32,
                                                        int32_t* err, const int* __restrict__ guard) {
  if (guard && *guard == 0) return;
  constexpr int STR = Pack<TF>::stride;
  constexpr int V = 16 / sizeof(TF), NV = 8 / V;  // values per 16-byte piece, pieces per block row
  constexpr int G = sizeof(TF) == 4 ? 4 : 2;      // groups of 4 blocks per entry
  constexpr uint32_t BLK = STR * sizeof(TF);
  extern __shared__ __align__(128) unsigned char smem[];
  uint64_t* full = reinterpret_cast<uint64_t*>(smem);  // [2]
  unsigned char* ring = smem + 128;
  const uint32_t cap = R.chain_blocks * BLK;  // bytes of one stage's slot
  TF* w = reinterpret_cast<TF*>(ring + 2 * cap);
  const int lane = threadIdx.x, s = blockIdx.x;
  const int c = lane & 7;
  const int j = c < 7 ? lane >> 3 : 64;  // block of a group this lane works on (c = 7: none)
  const int64_t r0 = R.sd_row[s];
  const int m = (int)(R.sd_row[s + 1] - r0);
  const uint32_t* cw = R.code + R.code_off[s];
  const int nw = (int)(R.code_off[s + 1] - R.code_off[s]) - 2;
  const TF* src = reinterpret_cast<const TF*>(R.pack) + (size_t)R.L_off[s] * STR;
  const uint8_t* sz = R.stage + R.stage_off[s];
  int left = R.stall == 1 ? 0 : (int)(R.stage_off[s + 1] - R.stage_off[s]);  // stages not yet asked for
  int nsz = left > 0 ? sz[0] : 0;                                       // blocks of the next one
  uint64_t win = cw[0] | (uint64_t)cw[1] << 32;  // entry codes ahead
  uint32_t ahead = cw[2];

  // lane 0: ask for the next stage
  auto feed = [&](int slot) {
    if (lane == 0 && left > 0) {
      mbar_arrive_expect_tx(&full[slot], nsz * BLK);
      bulk_g2s(ring + slot * cap, src, nsz * BLK, &full[slot]);
      src += (size_t)nsz * STR;
      ++sz;
      if (--left > 0) nsz = *sz;
    }
  };
  if (lane == 0) {
    mbar_init(&full[0], 1);
    mbar_init(&full[1], 1);
    asm volatile("fence.mbarrier_init.release.cluster;" ::: "memory");
  }
  __syncwarp();
  feed(0);
  feed(1);

  // restriction R_i^delta r into shared memory
#pragma unroll 4
  for (int q = lane; q < m; q += 32) {
    const double* sr = rin + 7 * (int64_t)R.gnode[r0 + q];
    double v[7];
#pragma unroll
    for (int e = 0; e < 7; ++e) v[e] = sr[e];
#pragma unroll
    for (int e = 0; e < 7; ++e) w[8 * q + e] = (TF)v[e];
    w[8 * q + 7] = TF(0);
  }
  __syncwarp();

  int slot = 0, phase = 0;  // stage being worked off and its barrier's phase
  const unsigned char* at = ring + 16 * c + (lane >> 3) * BLK;  // this lane's row of the next entry's first group
  bool ok = R.stall != 2;
  if (!ok) left = 0;
  int fslot = 0, fphase = 0;  // the stage given up on
  // once a wait gives up no stage is asked for any more: a barrier is not armed again
  // while a copy may still be on its way to its slot
  auto wait = [&]() {
    if (ok && !mbar_wait(&full[slot], (uint32_t)phase)) {
      ok = false;
      left = 0;
      fslot = slot;
      fphase = phase;
    }
  };
  // rows of an entry's blocks into registers; what lies behind its blocks is read too and not used
  auto fetch = [&](TF (&A)[G][8], uint32_t code) {
    auto rows = [&](int g) {
#pragma unroll
      for (int e = 0; e < NV; ++e) load16(&A[g][V * e], reinterpret_cast<const TF*>(at + g * 4 * BLK + 112 * e));
    };
#pragma unroll
    for (int g = 0; g < G / 2; ++g) rows(g);
    if (code & (2 * G)) {
#pragma unroll
      for (int g = G / 2; g < G; ++g) rows(g);
    }
    at += ((code & 15) + 1) * BLK;
  };
  auto xrow = [&](TF (&x)[8], const TF (&A)[8]) {
    const TF* xp = w + 8 * min((uint32_t)row_col(A), (uint32_t)m - 1);
#pragma unroll
    for (int e = 0; e < NV; ++e) load16(&x[V * e], xp + V * e);
  };

  int q = 0, dq = 1;
  TF acc = TF(0), tot = TF(-0.0);
  TF A0[G][8], A1[G][8];
  // work off the entry whose rows are in A, fetch the next one's into N
  auto step = [&](TF (&A)[G][8], TF (&N)[G][8], uint32_t code, uint32_t ncode) {
    if (code < ENTRY_NONE) {
      const int nb = (int)(code & 15) + 1 - j;  // this lane: blocks 0, 4, 8, .. below nb
      const TF old = w[8 * q + c];
      TF x[G][8];
#pragma unroll
      for (int g = 0; g < G / 2; ++g) xrow(x[g], A[g]);
      if (code & (2 * G)) {
#pragma unroll
        for (int g = G / 2; g < G; ++g) xrow(x[g], A[g]);
#pragma unroll
        for (int g = 0; g < G; ++g) {
          const TF t = row_fma(A[g], x[g], acc);
          if (4 * g < nb) acc = t;
        }
      } else {
#pragma unroll
        for (int g = 0; g < G / 2; ++g) {
          const TF t = row_fma(A[g], x[g], acc);
          if (4 * g < nb) acc = t;
        }
      }
      if (code & ENTRY_STAGE) {
        // every lane has read the stage: its slot takes the next but one
        __syncwarp();
        feed(slot);
        phase ^= slot;
        slot ^= 1;
        at = ring + slot * cap + 16 * c + (lane >> 3) * BLK;
        wait();
      }
      if (ncode < ENTRY_NONE) fetch(N, ncode);
      if (code & ENTRY_PIECE) {
        TF r = acc + __shfl_xor_sync(0xffffffffu, acc, 16);
        r += __shfl_xor_sync(0xffffffffu, r, 8);
        acc = TF(0);
        if (sizeof(TF) == 4) tot += r;
        else tot = r;
        if (code & ENTRY_ROW) {
          if (lane < 7) w[8 * q + lane] = dq > 0 ? old - tot : tot;
          __syncwarp();
          tot = TF(-0.0);
          q += dq;
        }
      }
    } else {
      if (code == ENTRY_EMPTY) {
        q += dq;
      } else if (code == ENTRY_BACKWARD) {
        q = m - 1;
        dq = -1;
      }
      if (ncode < ENTRY_NONE) fetch(N, ncode);
    }
  };
  wait();
  if ((win & 255) < ENTRY_NONE) fetch(A0, (uint32_t)win & 255);
  // a lane whose wait gave up goes on to the end with the others (the data do not decide any address)
  for (int it = 0; it < 2 * nw; ++it) {
    const uint32_t w3 = (uint32_t)win;
    step(A0, A1, w3 & 255, (w3 >> 8) & 255);
    step(A1, A0, (w3 >> 8) & 255, (w3 >> 16) & 255);
    win >>= 16;
    if (it & 1) {
      win |= (uint64_t)ahead << 32;
      ahead = cw[min((it >> 1) + 3, nw + 1)];
    }
  }
  if (!ok) {
    // record it and let the copies that may still be in flight land (bounded)
    atomicExch(err, 2);
    mbar_wait(&full[fslot], (uint32_t)fphase);
    mbar_wait(&full[fslot ^ 1], (uint32_t)(fphase ^ fslot));
  }

  // restricted prolongation (R_i^0)^T: owned rows only
#pragma unroll 4
  for (int q = lane; q < m; q += 32) {
    if (R.owned[r0 + q]) {
      const int64_t g7 = 7 * (int64_t)R.gnode[r0 + q];
#pragma unroll
      for (int e = 0; e < 7; ++e) z[g7 + e] = (double)w[8 * q + e];
      if (z32) {
#pragma unroll
        for (int e = 0; e < 7; ++e) z32[g7 + e] = (float)w[8 * q + e];
      }
    }
  }
}

// Team apply: four warps per subdomain, for runs with few subdomains, where one warp
// per SM sub-partition is all there is and a row's latency is the whole cost. The
// blocks of an entry (up to 16 of a row) are dealt to the warps, one per 8-lane
// group; the warps hand their products over in shared memory, meet at one barrier, and
// every warp adds them up and writes the row by itself (the same bits), so that the row
// needs no second barrier. The additions keep the chain kernel's order (sums over the
// blocks 0..3 mod 4): the same bits.
// Measured, mixed, 46,657-node tube, ILU(1), us per apply, one warp / team: 64
// subdomains 1,050 / 842, 256: 386 / 349, 384: 275 / 275, 512: 251 / 287.
__global__ void __launch_bounds__(128) k_ras_apply_team(RasStreamDev R, const double* __restrict__ rin,
                                                        double* __restrict__ z, float* __restrict__ z32,
                                                        int32_t* err, const int* __restrict__ guard) {
  if (guard && *guard == 0) return;
  constexpr int STR = Pack<float>::stride;
  constexpr uint32_t BLK = STR * sizeof(float);
  constexpr int PT = 7 * 20;  // products handed over per entry: [c][v][g], 20 per c (no bank conflicts)
  extern __shared__ __align__(128) unsigned char smem[];
  uint64_t* full = reinterpret_cast<uint64_t*>(smem);           // [2]
  float* part = reinterpret_cast<float*>(smem + 128);                 // [2][PT]
  unsigned char* ring = smem + 128 + 1152;
  const uint32_t cap = R.chain_blocks * BLK;
  float* w = reinterpret_cast<float*>(ring + 2 * cap);
  const int lane = threadIdx.x & 31, v = threadIdx.x >> 5, s = blockIdx.x;
  const int c = lane & 7, g = lane >> 3;
  const int b = 4 * g + v;  // this lane's block of an entry
  const int64_t r0 = R.sd_row[s];
  const int m = (int)(R.sd_row[s + 1] - r0);
  const uint32_t* cw = R.code + R.code_off[s];
  const int nw = (int)(R.code_off[s + 1] - R.code_off[s]) - 2;
  const float* src = reinterpret_cast<const float*>(R.pack) + (size_t)R.L_off[s] * STR;
  const uint8_t* sz = R.stage + R.stage_off[s];
  int left = R.stall == 1 ? 0 : (int)(R.stage_off[s + 1] - R.stage_off[s]);
  int nsz = left > 0 ? sz[0] : 0;
  uint64_t win = cw[0] | (uint64_t)cw[1] << 32;
  uint32_t ahead = cw[2];

  auto feed = [&](int slot) {
    if (threadIdx.x == 0 && left > 0) {
      mbar_arrive_expect_tx(&full[slot], nsz * BLK);
      bulk_g2s(ring + slot * cap, src, nsz * BLK, &full[slot]);
      src += (size_t)nsz * STR;
      ++sz;
      if (--left > 0) nsz = *sz;
    }
  };
  if (threadIdx.x == 0) {
    mbar_init(&full[0], 1);
    mbar_init(&full[1], 1);
    asm volatile("fence.mbarrier_init.release.cluster;" ::: "memory");
    feed(0);
    feed(1);
  }
  for (int q = threadIdx.x; q < m; q += 128) {
    const double* sr = rin + 7 * (int64_t)R.gnode[r0 + q];
    double x[7];
#pragma unroll
    for (int e = 0; e < 7; ++e) x[e] = sr[e];
#pragma unroll
    for (int e = 0; e < 7; ++e) w[8 * q + e] = (float)x[e];
    w[8 * q + 7] = float(0);
  }
  __syncthreads();

  int slot = 0, phase = 0, par = 0;
  const unsigned char* at = ring + 16 * c + b * BLK;
  bool ok = R.stall != 2;
  if (!ok) left = 0;
  auto fetch = [&](float (&A)[8], uint32_t code) {
    const int nb = (int)(code & 15) + 1;
    load16(&A[0], reinterpret_cast<const float*>(at));
    load16(&A[4], reinterpret_cast<const float*>(at + 112));
    at += nb * BLK;
  };
  int q = 0, dq = 1;
  // the four partial sums of a row (blocks 0..3 mod 4), in every warp
  float acc[4] = {float(0), float(0), float(0), float(0)}, tot = float(-0.0);
  float A0[8], A1[8];
#pragma unroll
  for (int e = 0; e < 8; ++e) A0[e] = A1[e] = float(0);
  const int cc = c < 7 ? c : 6;
  int fslot = 0, fphase = 0;
  auto wait = [&]() {
    if (ok && !mbar_wait(&full[slot], (uint32_t)phase)) {
      ok = false;
      left = 0;
      fslot = slot;
      fphase = phase;
    }
  };
  auto step = [&](float (&A)[8], float (&N)[8], uint32_t code, uint32_t ncode) {
    if (code < ENTRY_NONE) {
      const int nb = (int)(code & 15) + 1;
      const bool piece = code & ENTRY_PIECE;
      const float old = w[8 * q + c];
      float* const pb = part + par * PT;
      const float* xp = w + 8 * min((uint32_t)row_col(A), (uint32_t)m - 1);
      float x[8];
      load16(&x[0], xp);
      load16(&x[4], xp + 4);
      const float t = row_fma(A, x, float(0));
      if (c < 7) pb[20 * c + 4 * v + g] = b < nb ? t : float(0);
      __syncthreads();
      if (code & ENTRY_STAGE) {
        feed(slot);
        phase ^= slot;
        slot ^= 1;
        at = ring + slot * cap + 16 * c + b * BLK;
        wait();
      }
      if (ncode < ENTRY_NONE) fetch(N, ncode);
#pragma unroll
      for (int i = 0; i < 4; ++i) {
        float t4[4];
        load16(t4, pb + 20 * cc + 4 * i);
#pragma unroll
        for (int e = 0; e < 4; ++e) acc[i] += t4[e];
      }
      par ^= 1;
      if (piece) {
        tot += (acc[0] + acc[2]) + (acc[1] + acc[3]);
#pragma unroll
        for (int i = 0; i < 4; ++i) acc[i] = float(0);
        if (code & ENTRY_ROW) {
          if (lane < 7) w[8 * q + lane] = dq > 0 ? old - tot : tot;
          __syncwarp();
          tot = float(-0.0);
          q += dq;
        }
      }
    } else {
      if (code == ENTRY_EMPTY) {
        q += dq;
      } else if (code == ENTRY_BACKWARD) {
        q = m - 1;
        dq = -1;
      }
      if (ncode < ENTRY_NONE) fetch(N, ncode);
    }
  };
  wait();
  if ((win & 255) < ENTRY_NONE) fetch(A0, (uint32_t)win & 255);
  // a warp whose wait gave up goes on to the end (the data do not decide any address or barrier)
  for (int it = 0; it < 2 * nw; ++it) {
    const uint32_t w3 = (uint32_t)win;
    step(A0, A1, w3 & 255, (w3 >> 8) & 255);
    step(A1, A0, (w3 >> 8) & 255, (w3 >> 16) & 255);
    win >>= 16;
    if (it & 1) {
      win |= (uint64_t)ahead << 32;
      ahead = cw[min((it >> 1) + 3, nw + 1)];
    }
  }
  if (!ok || (R.stall == 3 && lane == 1)) {
    // record it; the thread that asked for the copies lets those that may still be in
    // flight land (bounded; it has waited for all of them if it has not given up itself)
    atomicExch(err, 2);
    if (threadIdx.x == 0) {
      mbar_wait(&full[fslot], (uint32_t)fphase);
      mbar_wait(&full[fslot ^ 1], (uint32_t)(fphase ^ fslot));
    }
  }
  __syncthreads();
  for (int q = threadIdx.x; q < m; q += 128) {
    if (R.owned[r0 + q]) {
      const int64_t g7 = 7 * (int64_t)R.gnode[r0 + q];
#pragma unroll
      for (int e = 0; e < 7; ++e) z[g7 + e] = (double)w[8 * q + e];
      if (z32) {
#pragma unroll
        for (int e = 0; e < 7; ++e) z32[g7 + e] = (float)w[8 * q + e];
      }
    }
  }
}

// FP64 team apply, a step ahead (setup.h, build_lookahead_stream): in step t warp 0
// solves the step's row from the sum over its far blocks, formed in step t - 1, and
// from its near block alone, whose vector it still holds in registers (7-term dots
// spread over its four 8-lane groups: 2 fused multiply-adds, 2 additions), while warps
// 1 to 3 form the far sum of step t + 1's row (12 blocks at a time, 7 + 2 FP64
// instructions of 64 cycles each). One barrier per step. Measured against one warp
// per subdomain (k_ras_apply_chain), us per apply: 46,657-node tube, ILU(1), 64
// subdomains 4,334 / 2,409, 256: 1,545 / 927, 384: 978 / 708, 512: 890 / 767, 768: 759 / 716,
// 1,024: 617 / 694; 103k-node tree, ILU(1), 512: 1,199 / 1,041, 768: 989 / 1,115, ILU(2)
// 512: 1,753 / 1,407, 768: 1,446 / 1,518. Taken up to 608 (four subdomains per SM).
__global__ void __launch_bounds__(128) k_ras_apply_team64(RasStreamDev R, const double* __restrict__ rin,
                                                          double* __restrict__ z, float* __restrict__ z32,
                                                          int32_t* err, const int* __restrict__ guard) {
  if (guard && *guard == 0) return;
  constexpr int STR = Pack<double>::stride;
  constexpr uint32_t BLK = STR * sizeof(double);
  extern __shared__ __align__(128) unsigned char smem[];
  uint64_t* full = reinterpret_cast<uint64_t*>(smem);              // [2]
  double(*part)[4][8] = reinterpret_cast<double(*)[4][8]>(smem + 128);  // [2][warp][component] far sums
  unsigned char* ring = smem + 128 + 1152;
  const uint32_t cap = R.chain_blocks * BLK;
  double* w = reinterpret_cast<double*>(ring + 2 * cap);
  const int lane = threadIdx.x & 31, v = threadIdx.x >> 5, s = blockIdx.x;
  const int c = lane & 7, g = lane >> 3;
  const int b = 4 * (v - 1) + g;  // this lane's far block of an entry (warps 1 to 3)
  const int64_t r0 = R.sd_row[s];
  const int m = (int)(R.sd_row[s + 1] - r0);
  const uint32_t* cw = R.code + R.code_off[s];
  const int nw = (int)(R.code_off[s + 1] - R.code_off[s]) - 2;
  const double* src = reinterpret_cast<const double*>(R.pack) + (size_t)R.L_off[s] * STR;
  const uint8_t* sz = R.stage + R.stage_off[s];
  int left = R.stall == 1 ? 0 : (int)(R.stage_off[s + 1] - R.stage_off[s]);
  int nsz = left > 0 ? sz[0] : 0;
  uint64_t win = cw[0] | (uint64_t)cw[1] << 32;
  uint32_t ahead = cw[2];

  auto feed = [&](int slot) {
    if (threadIdx.x == 0 && left > 0) {
      mbar_arrive_expect_tx(&full[slot], nsz * BLK);
      bulk_g2s(ring + slot * cap, src, nsz * BLK, &full[slot]);
      src += (size_t)nsz * STR;
      ++sz;
      if (--left > 0) nsz = *sz;
    }
  };
  if (threadIdx.x == 0) {
    mbar_init(&full[0], 1);
    mbar_init(&full[1], 1);
    asm volatile("fence.mbarrier_init.release.cluster;" ::: "memory");
    feed(0);
    feed(1);
  }
  if (threadIdx.x < 64) reinterpret_cast<double*>(part)[threadIdx.x] = 0.0;
  for (int q = threadIdx.x; q < m; q += 128) {
    const double* sr = rin + 7 * (int64_t)R.gnode[r0 + q];
#pragma unroll
    for (int e = 0; e < 7; ++e) w[8 * q + e] = sr[e];
    w[8 * q + 7] = 0.0;
  }
  __syncthreads();

  int slot = 0, phase = 0, par = 0, t = 0, fslot = 0, fphase = 0;
  bool ok = R.stall != 2;
  if (!ok) left = 0;
  const unsigned char* at = ring;  // blocks of the next entry to fetch (warp 0: of the current one)
  auto wait = [&]() {
    if (ok && !mbar_wait(&full[slot], (uint32_t)phase)) {
      ok = false;
      left = 0;
      fslot = slot;
      fphase = phase;
    }
  };
  auto next_stage = [&]() {
    feed(slot);
    phase ^= slot;
    slot ^= 1;
    at = ring + slot * cap;
    wait();
  };
  auto size = [](uint32_t code) { return ((code & 15) + ((code & ENTRY_NEAR) ? 1 : 0)) * BLK; };
  wait();

  if (v == 0) {
    double r = 0.0;  // component c of the last step's row (0 for c = 7), in all groups
    const int k1 = g < 3 ? g + 4 : 7;
    auto step = [&](uint32_t code) {
      if (code >= ENTRY_NONE) return;
      if (code & ENTRY_END) {
        const int q = t < m ? t : 2 * m - 1 - t;
        double acc = g == 0 ? (t < m ? -w[8 * q + c] : 0.0) : part[par][g][c];
        if (code & ENTRY_NEAR) {
          // entries g and g + 4 of row c (c = 7: row 6's, not used) of the near block
          const double* A = reinterpret_cast<const double*>(at + (code & 15) * BLK) + 2 * (c < 7 ? c : 6);
          const double x0 = __shfl_sync(0xffffffffu, r, g), x1 = __shfl_sync(0xffffffffu, r, k1);
          acc = fma(A[14 * (g >> 1) + (g & 1)], x0, acc);
          const double y1 = fma(A[14 * ((g + 4) >> 1) + (g & 1)], x1, acc);
          if (g < 3) acc = y1;
        }
        acc += __shfl_xor_sync(0xffffffffu, acc, 16);
        acc += __shfl_xor_sync(0xffffffffu, acc, 8);
        r = c < 7 ? (t < m ? -acc : acc) : 0.0;
        if (lane < 7) w[8 * q + c] = r;
        par ^= 1;
        ++t;
      }
      if (code & (ENTRY_END | ENTRY_STAGE)) __syncthreads();
      if (code & ENTRY_STAGE) next_stage();
      else at += size(code);
    };
    for (int it = 0; it < 2 * nw; ++it) {
      const uint32_t w3 = (uint32_t)win;
      step(w3 & 255);
      step((w3 >> 8) & 255);
      win >>= 16;
      if (it & 1) {
        win |= (uint64_t)ahead << 32;
        ahead = cw[min((it >> 1) + 3, nw + 1)];
      }
    }
  } else {
    double A0[8], A1[8], acc = 0.0;
    bool used = false;  // the warp has had blocks of the row
#pragma unroll
    for (int e = 0; e < 8; ++e) A0[e] = A1[e] = 0.0;
    auto fetch = [&](double (&A)[8], uint32_t code) {
      if (4 * (v - 1) < (int)(code & 15)) {
        const double* p = reinterpret_cast<const double*>(at + b * BLK) + 2 * (c < 7 ? c : 6);
#pragma unroll
        for (int e = 0; e < 4; ++e) load16(&A[2 * e], p + 14 * e);
      }
      at += size(code);
    };
    auto step = [&](double (&A)[8], double (&N)[8], uint32_t code, uint32_t ncode) {
      if (code < ENTRY_NONE) {
        const int nf = (int)(code & 15);
        if (4 * (v - 1) < nf) {
          const double* xp = w + 8 * min((uint32_t)row_col(A), (uint32_t)m - 1);
          double x[8];
#pragma unroll
          for (int e = 0; e < 4; ++e) load16(&x[2 * e], xp + 2 * e);
          const double y = row_fma(A, x, acc);
          if (b < nf) acc = y;
          used = true;
        }
        if (code & ENTRY_END) {
          if (used) {  // (no additions of zeros: they take the FP64 pipe as long)
            acc += __shfl_xor_sync(0xffffffffu, acc, 16);
            acc += __shfl_xor_sync(0xffffffffu, acc, 8);
          }
          par ^= 1;
          if (lane < 7) part[par][v][c] = acc;
          acc = 0.0;
          used = false;
        }
        if (code & (ENTRY_END | ENTRY_STAGE)) __syncthreads();
        if (code & ENTRY_STAGE) next_stage();
      }
      if (ncode < ENTRY_NONE) fetch(N, ncode);
    };
    if ((win & 255) < ENTRY_NONE) fetch(A0, (uint32_t)win & 255);
    for (int it = 0; it < 2 * nw; ++it) {
      const uint32_t w3 = (uint32_t)win;
      step(A0, A1, w3 & 255, (w3 >> 8) & 255);
      step(A1, A0, (w3 >> 8) & 255, (w3 >> 16) & 255);
      win >>= 16;
      if (it & 1) {
        win |= (uint64_t)ahead << 32;
        ahead = cw[min((it >> 1) + 3, nw + 1)];
      }
    }
  }
  if (!ok || (R.stall == 3 && lane == 1)) {
    atomicExch(err, 2);
    if (threadIdx.x == 0) {
      mbar_wait(&full[fslot], (uint32_t)fphase);
      mbar_wait(&full[fslot ^ 1], (uint32_t)(fphase ^ fslot));
    }
  }
  __syncthreads();
  for (int q = threadIdx.x; q < m; q += 128) {
    if (R.owned[r0 + q]) {
      const int64_t g7 = 7 * (int64_t)R.gnode[r0 + q];
#pragma unroll
      for (int e = 0; e < 7; ++e) z[g7 + e] = w[8 * q + e];
      if (z32) {
#pragma unroll
        for (int e = 0; e < 7; ++e) z32[g7 + e] = (float)w[8 * q + e];
      }
    }
  }
}

// copy the factor blocks into the packed stream (7 rows of 8: the row's 7
// entries, then the block's column, in 16-byte pieces); a U block with a pivot
// (piv >= 0) is stored as -D_q^{-1} U_qj, the row's inverted pivot and the L
// blocks as they are. One warp per block: its index list entries are read once per
// block and the products take both blocks from shared memory (one thread per value,
// with 64-bit divisions and the products' 14 operands from L1: 1.27 M blocks 295 -> 195 us).
template <class TF>
__global__ void __launch_bounds__(256) k_pack_factors(int64_t nblk, const int64_t* __restrict__ src,
                                                      const int32_t* __restrict__ col,
                                                      const int64_t* __restrict__ pivs, const TF* __restrict__ fac,
                                                      TF* __restrict__ pack) {
  constexpr int STR = Pack<TF>::stride, V = 16 / sizeof(TF);
  __shared__ TF sm[8][2][56];
  const int lane = threadIdx.x & 31;
  TF* A = sm[threadIdx.x >> 5][0];
  TF* D = sm[threadIdx.x >> 5][1];
  // this lane's values e = lane and lane + 32 (below 56): row and entry
  const int e1 = lane + 32;
  const int r0 = (lane % (7 * V)) / V, k0 = (lane / (7 * V)) * V + lane % V;
  const int r1 = (e1 % (7 * V)) / V, k1 = (e1 / (7 * V)) * V + e1 % V;
  const int64_t step = ((int64_t)gridDim.x * blockDim.x) >> 5;
  for (int64_t b = (blockIdx.x * (int64_t)blockDim.x + threadIdx.x) >> 5; b < nblk; b += step) {
    const int64_t sb = src[b], piv = pivs[b];
    const int cb = col[b];
    A[lane] = fac[49 * sb + lane];
    if (lane < 17) A[lane + 32] = fac[49 * sb + lane + 32];
    if (piv >= 0) {
      D[lane] = fac[49 * piv + lane];
      if (lane < 17) D[lane + 32] = fac[49 * piv + lane + 32];
    }
    __syncwarp();
    auto value = [&](int r, int k) {
      TF v = TF(0);
      if (k == 7) {
        *reinterpret_cast<int*>(&v) = cb;
      } else if (piv < 0) {
        v = A[7 * r + k];
      } else {
        // -(D_q^{-1} U_qj)[r][k]
#pragma unroll
        for (int mm = 0; mm < 7; ++mm) v += D[7 * r + mm] * A[7 * mm + k];
        v = -v;
      }
      return v;
    };
    pack[b * STR + lane] = value(r0, k0);
    if (e1 < STR) pack[b * STR + e1] = value(r1, k1);
    __syncwarp();
  }
}

}  // namespace

template <class TF>
size_t ras_stream_smem(const RasStreamDev& r) {
  const size_t W = (size_t)1 << r.max_depth;
  return 128 * ((W * NSTMAX * 8 + 127) / 128) + W * r.nst * r.stage_blocks * Pack<TF>::stride * sizeof(TF) +
         (size_t)8 * r.max_rows * sizeof(TF) + (size_t)4 * r.max_rows + 16;
}

template <class TF>
void launch_pack_factors(const RasStreamDev& r, const TF* fac, cudaStream_t s) {
  int64_t g = (r.nblk + 7) / 8;
  if (g > 152 * 64) g = 152 * 64;
  k_pack_factors<TF><<<(int)g, 256, 0, s>>>(r.nblk, r.src, r.col, r.piv, fac, (TF*)r.pack);
}

// the ring kernel runs dissected subdomains
static bool takes_ring(const RasStreamDev& r) { return r.max_depth > 0; }

template <class TF>
size_t chain_smem(const RasStreamDev& r) {
  // (an entry's last rows are read up to 15 (FP64, one warp: 7) blocks beyond its own)
  const size_t over = (sizeof(TF) == 4 || r.team ? 15 : 7) * Pack<TF>::stride, vec = (size_t)8 * r.max_rows;
  return (r.team ? 128 + 1152 : 128) +
         ((size_t)2 * r.chain_blocks * Pack<TF>::stride + (vec > over ? vec : over)) * sizeof(TF);
}

template <class TF>
const void* team_kernel() {
  return sizeof(TF) == 4 ? (const void*)k_ras_apply_team : (const void*)k_ras_apply_team64;
}

template <class TF>
cudaError_t ras_stream_init(const RasStreamDev& r) {
  const void* k = takes_ring(r) ? (const void*)k_ras_apply_stream<TF>
                  : r.team      ? team_kernel<TF>()
                                : (const void*)k_ras_apply_chain<TF>;
  // all of the unified L1/shared storage as shared memory: several CTAs per SM;
  // the limit is the kernel's, not the context's: contexts of different sizes share it
  cudaError_t e = cudaFuncSetAttribute(k, cudaFuncAttributePreferredSharedMemoryCarveout,
                                       (int)cudaSharedmemCarveoutMaxShared);
  if (e != cudaSuccess) return e;
  return cudaFuncSetAttribute(k, cudaFuncAttributeMaxDynamicSharedMemorySize, 227 * 1024);
}

template <class TF>
cudaError_t launch_ras_apply_stream(const RasStreamDev& r, const double* rin, double* z, float* z32, int32_t* err,
                                    const int* guard, cudaStream_t s) {
  if (takes_ring(r))
    k_ras_apply_stream<TF><<<r.np, 32 << r.max_depth, ras_stream_smem<TF>(r), s>>>(r, rin, z, z32, err, guard);
  else if (r.team && sizeof(TF) == 4)
    k_ras_apply_team<<<r.np, 128, chain_smem<TF>(r), s>>>(r, rin, z, z32, err, guard);
  else if (r.team)
    k_ras_apply_team64<<<r.np, 128, chain_smem<TF>(r), s>>>(r, rin, z, z32, err, guard);
  else
    k_ras_apply_chain<TF><<<r.np, 32, chain_smem<TF>(r), s>>>(r, rin, z, z32, err, guard);
  return cudaGetLastError();
}

template cudaError_t ras_stream_init<float>(const RasStreamDev&);
template cudaError_t ras_stream_init<double>(const RasStreamDev&);

template size_t ras_stream_smem<float>(const RasStreamDev&);
template size_t ras_stream_smem<double>(const RasStreamDev&);
template void launch_pack_factors<float>(const RasStreamDev&, const float*, cudaStream_t);
template void launch_pack_factors<double>(const RasStreamDev&, const double*, cudaStream_t);
template cudaError_t launch_ras_apply_stream<float>(const RasStreamDev&, const double*, double*, float*, int32_t*,
                                                    const int*, cudaStream_t);
template cudaError_t launch_ras_apply_stream<double>(const RasStreamDev&, const double*, double*, float*, int32_t*,
                                                     const int*, cudaStream_t);

}  // namespace fsi
