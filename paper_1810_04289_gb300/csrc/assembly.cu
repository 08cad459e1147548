// Residual (FuncEval) and Jacobian (JacEval) assembly.
//
// Atomic-free, deterministic two-phase scheme:
//   1. one element kernel computes every tet's contribution into an element
//      buffer (Fe: 4 x 7 rows per tet; Ke: 4 x 4 blocks of 7 x 7 per tet);
//   2. one gather kernel sums, for every node row (resp. BSR block), the buffer
//      slots listed for it in increasing tet order.
// Element rows are routed to node rows by the node flags (strong interface
// coupling, Sec. 2.2): continuity -> p row; fluid momentum -> u rows of
// fluid-only nodes and d rows of interface nodes; mesh motion -> d rows of
// fluid-only nodes; wall momentum -> d rows. Constrained rows receive zeros; the
// residual's gather puts their own residual in place, a kernel after the Jacobian's
// gather their diagonal blocks.
#include <cuda_runtime.h>

#include "kernels.cuh"
#include "setup.h"

namespace fsi {

namespace {

__device__ __forceinline__ void load_tet(const MeshDev& m, int64_t t, int n[4], uint32_t f[4]) {
#pragma unroll
  for (int a = 0; a < 4; ++a) {
    n[a] = m.tets[4 * t + a];
    f[a] = m.nflag[n[a]];
  }
}

__device__ __forceinline__ void load_edges(const MeshDev& m, const int n[4], double e[3][3]) {
  const double* x0 = m.X + 3 * (int64_t)n[0];
#pragma unroll
  for (int k = 0; k < 3; ++k) {
    const double* x = m.X + 3 * (int64_t)n[k + 1];
#pragma unroll
    for (int i = 0; i < 3; ++i) e[k][i] = x[i] - x0[i];
  }
}

// reference geometry from the [GEO][T] array: gradients of vertices 1..3 and volume
__device__ __forceinline__ void load_geo(const MeshDev& m, int64_t t, double g0[3][3], double& vol0) {
#pragma unroll
  for (int k = 0; k < 9; ++k) g0[k / 3][k % 3] = m.geo[k * m.T + t];
  vol0 = m.geo[9 * m.T + t];
}

__global__ void k_geometry(MeshDev m, double* __restrict__ geo) {
  for (int64_t t = blockIdx.x * (int64_t)blockDim.x + threadIdx.x; t < m.T; t += (int64_t)gridDim.x * blockDim.x) {
    int n[4];
    uint32_t f[4];
    load_tet(m, t, n, f);
    double e[3][3], X[4][3], out[GEO];
    load_edges(m, n, e);
#pragma unroll
    for (int i = 0; i < 3; ++i) {
      X[0][i] = 0.0;
#pragma unroll
      for (int k = 0; k < 3; ++k) X[k + 1][i] = e[k][i];
    }
    reference_geometry(X, out);
#pragma unroll
    for (int k = 0; k < GEO; ++k) geo[k * m.T + t] = out[k];
  }
}

// the fluid tet's fields at its vertices
struct FluidFields {
  double u[4][3], p[4], d[4][3], u1[4][3], d1[4][3], de[3][3];
  __device__ __forceinline__ FluidFields(const int n[4], const double* __restrict__ y, const double* __restrict__ y1) {
#pragma unroll
    for (int a = 0; a < 4; ++a) {
      const double* ya = y + 7 * (int64_t)n[a];
      const double* y1a = y1 + 7 * (int64_t)n[a];
#pragma unroll
      for (int i = 0; i < 3; ++i) {
        u[a][i] = ya[i];
        d[a][i] = ya[4 + i];
        u1[a][i] = y1a[i];
        d1[a][i] = y1a[4 + i];
      }
      p[a] = ya[3];
    }
#pragma unroll
    for (int k = 0; k < 3; ++k)
#pragma unroll
      for (int i = 0; i < 3; ++i) de[k][i] = d[k + 1][i] - d[0][i];
  }
};

// One thread per tet. Bound by the FP64 pipe; closed-form integrals and stored
// reference geometry (see element.cuh)
__global__ void __launch_bounds__(128) k_elem_residual(MeshDev m, MatConst mc, const double* __restrict__ y,
                                                       const double* __restrict__ y1, const double* __restrict__ y2,
                                                       double* __restrict__ Fe) {
  for (int64_t t = blockIdx.x * (int64_t)blockDim.x + threadIdx.x; t < m.T; t += (int64_t)gridDim.x * blockDim.x) {
    int n[4];
    uint32_t f[4];
    load_tet(m, t, n, f);
    double g0[3][3], vol0;
    load_geo(m, t, g0, vol0);
    double out[4][7];
    if (t < m.Tf) {
      const FluidFields q(n, y, y1);
      double Xe[3][3];
      load_edges(m, n, Xe);
      FluidValues v;
      fluid_values(Xe, q.de, q.u, q.p, q.d, q.u1, q.d1, m.geo[10 * m.T + t], m.geo[11 * m.T + t], mc, v);
      double Rm[4][3], gr[4], Rc[4], Rh[4][3];
      fluid_momentum(v, Rm);
      fluid_continuity(v, gr, Rc);
      mesh_motion(q.de, g0, vol0, Rh);
#pragma unroll
      for (int a = 0; a < 4; ++a) {
        const bool uc = f[a] & NF_U_CONSTR, pc = f[a] & NF_P_IDENT, dz = f[a] & NF_D_ZERO, itf = f[a] & NF_ITF;
#pragma unroll
        for (int i = 0; i < 3; ++i) {
          out[a][i] = uc ? 0.0 : Rm[a][i];
          out[a][4 + i] = dz ? 0.0 : (itf ? Rm[a][i] : Rh[a][i]);
        }
        out[a][3] = pc ? 0.0 : Rc[a];
      }
    } else {
      double d[4][3], d1[4][3], d2[4][3], de[3][3];
#pragma unroll
      for (int a = 0; a < 4; ++a)
#pragma unroll
        for (int i = 0; i < 3; ++i) {
          d[a][i] = y[7 * (int64_t)n[a] + 4 + i];
          d1[a][i] = y1[7 * (int64_t)n[a] + 4 + i];
          d2[a][i] = y2[7 * (int64_t)n[a] + 4 + i];
        }
#pragma unroll
      for (int k = 0; k < 3; ++k)
#pragma unroll
        for (int i = 0; i < 3; ++i) de[k][i] = d[k + 1][i] - d[0][i];
      double Rw[4][3];
      wall_residual(de, g0, vol0, d, d1, d2, mc, Rw);
#pragma unroll
      for (int a = 0; a < 4; ++a) {
        const bool dz = f[a] & NF_D_ZERO;
#pragma unroll
        for (int i = 0; i < 3; ++i) {
          out[a][i] = 0.0;
          out[a][4 + i] = dz ? 0.0 : Rw[a][i];
        }
        out[a][3] = 0.0;
      }
    }
    double* o = Fe + 28 * t;
#pragma unroll
    for (int a = 0; a < 4; ++a)
#pragma unroll
      for (int r = 0; r < 7; ++r) o[7 * a + r] = out[a][r];
  }
}

// the residual of component r of node i where a flag constrains it, else s (a call of
// its own, taken by the nodes with flags only: inlined, its registers cost the gather
// more than the call)
__device__ __noinline__ double constrained(const MeshDev* m, double idt, double t, const double* y, const double* y1,
                                           int64_t i, int r, uint32_t f, double s) {
  const double* yi = y + 7 * i;
  if (r >= 3) return (r == 3 ? (f & NF_P_IDENT) : (f & NF_D_ZERO)) ? yi[r] : s;
  if (f & NF_U_INLET) {
    const double* in = m->inlet + INLET_STRIDE * m->nprob[i];
    const double* x = m->X + 3 * i;
    const double rx = x[0] - in[0], ry = x[1] - in[1], rz = x[2] - in[2];
    const double ax = rx * in[3] + ry * in[4] + rz * in[5];
    const double r2 = (rx * rx + ry * ry + rz * rz) - ax * ax;
    const double U = in[7] * (1.0 + in[8] * sin(2.0 * 3.141592653589793 * in[9] * t + in[10]));
    const double prof = fmax(0.0, 1.0 - r2 / (in[6] * in[6]));
    return yi[r] - U * prof * in[3 + r];
  }
  if (f & NF_U_IDENT) return yi[r];
  if (f & NF_U_KIN) return yi[r] - (yi[4 + r] - y1[7 * i + 4 + r]) * idt;
  return s;
}

// Each node row is summed from its buffer slots in tet order, then constrained rows
// get their own residual; eight lanes take a node (seven of them a component each),
// four slots in flight. The FP64 additions and the read of the buffer (56 bytes per
// slot) bound it about equally: 912k tets 83 us (76 as two launches; 2,016 tets, one
// launch less: the whole residual 47 -> 38 us).
__global__ void __launch_bounds__(256) k_gather_residual(const __grid_constant__ MeshDev m, MatConst mc, double t,
                                                         const int64_t* __restrict__ nptr,
                                                         const int32_t* __restrict__ nsrc,
                                                         const double* __restrict__ Fe,
                                                         const double* __restrict__ y,
                                                         const double* __restrict__ y1, double* __restrict__ F) {
  const int r = threadIdx.x & 7;
  const int64_t step = ((int64_t)gridDim.x * blockDim.x) >> 3;
  for (int64_t i = (blockIdx.x * (int64_t)blockDim.x + threadIdx.x) >> 3; i < m.N; i += step) {
    if (r == 7) continue;
    double s = 0.0;
    int64_t c = nptr[i];
    const int64_t c1 = nptr[i + 1];
    const uint32_t f = m.nflag[i];
    for (; c + 4 <= c1; c += 4) {
      double v[4];
#pragma unroll
      for (int k = 0; k < 4; ++k) v[k] = Fe[7 * (int64_t)nsrc[c + k] + r];
#pragma unroll
      for (int k = 0; k < 4; ++k) s += v[k];
    }
    for (; c < c1; ++c) s += Fe[7 * (int64_t)nsrc[c] + r];
    if (f & (NF_U_CONSTR | NF_P_IDENT | NF_D_ZERO)) s = constrained(&m, mc.idt, t, y, y1, i, r, f, s);
    F[7 * i + r] = s;
  }
}

// Mixed form: one Jacobian column per thread, 28 threads per tet (column = node b,
// dof k), forward-mode derivative of the element residual along that column in
// T = float. Inputs are already in T: per-tet reference coordinates relative to
// vertex 0 (Xl, 12 per tet) and node states (y, y_old, y_older), so the kernel runs
// no FP64 instruction.
constexpr int JAC_TETS_PER_BLOCK = 8;

template <class T>
__global__ void __launch_bounds__(28 * JAC_TETS_PER_BLOCK)
k_elem_jacobian(MeshDev m, MatConst mc, const T* __restrict__ Xl, const T* __restrict__ y,
                const T* __restrict__ y1, const T* __restrict__ y2, T* __restrict__ Ke, int64_t t0, int64_t t1) {
  const int tl = threadIdx.x / 28;
  const int colid = threadIdx.x - 28 * tl;
  const int b = colid / 7, k = colid - 7 * (colid / 7);
  for (int64_t t = t0 + blockIdx.x * (int64_t)JAC_TETS_PER_BLOCK + tl; t < t1;
       t += (int64_t)gridDim.x * JAC_TETS_PER_BLOCK) {
    int n[4];
    uint32_t f[4];
    load_tet(m, t, n, f);
    T X[4][3];
#pragma unroll
    for (int a = 0; a < 4; ++a)
#pragma unroll
      for (int i = 0; i < 3; ++i) X[a][i] = Xl[12 * t + 3 * a + i];
    T out[4][7];
    if (t < m.Tf) {
      Dual<T> u[4][3], p[4], d[4][3];
      T u1[4][3], d1[4][3];
#pragma unroll
      for (int a = 0; a < 4; ++a) {
        const T* ya = y + 7 * (int64_t)n[a];
        const T* y1a = y1 + 7 * (int64_t)n[a];
#pragma unroll
        for (int i = 0; i < 3; ++i) {
          u[a][i] = Dual<T>(ya[i], (a == b && k == i) ? T(1) : T(0));
          d[a][i] = Dual<T>(ya[4 + i], (a == b && k == 4 + i) ? T(1) : T(0));
          u1[a][i] = y1a[i];
          d1[a][i] = y1a[4 + i];
        }
        p[a] = Dual<T>(ya[3], (a == b && k == 3) ? T(1) : T(0));
      }
      Dual<T> Rm[4][3], Rc[4], Rh[4][3];
      fluid_element<Dual<T>, T>(X, u, p, d, u1, d1, mc, Rm, Rc, Rh);
#pragma unroll
      for (int a = 0; a < 4; ++a) {
        const bool uc = f[a] & NF_U_CONSTR, pc = f[a] & NF_P_IDENT, dz = f[a] & NF_D_ZERO, itf = f[a] & NF_ITF;
#pragma unroll
        for (int i = 0; i < 3; ++i) {
          out[a][i] = uc ? T(0) : Rm[a][i].d;
          out[a][4 + i] = dz ? T(0) : (itf ? Rm[a][i].d : Rh[a][i].d);
        }
        out[a][3] = pc ? T(0) : Rc[a].d;
      }
    } else {
#pragma unroll
      for (int a = 0; a < 4; ++a)
#pragma unroll
        for (int r = 0; r < 7; ++r) out[a][r] = T(0);
      if (k >= 4) {
        Dual<T> d[4][3];
        T d1[4][3], d2[4][3];
#pragma unroll
        for (int a = 0; a < 4; ++a)
#pragma unroll
          for (int i = 0; i < 3; ++i) {
            d[a][i] = Dual<T>(y[7 * (int64_t)n[a] + 4 + i], (a == b && k == 4 + i) ? T(1) : T(0));
            d1[a][i] = y1[7 * (int64_t)n[a] + 4 + i];
            d2[a][i] = y2[7 * (int64_t)n[a] + 4 + i];
          }
        Dual<T> Rw[4][3];
        wall_element<Dual<T>, T>(X, d, d1, d2, mc, Rw);
#pragma unroll
        for (int a = 0; a < 4; ++a) {
          const bool dz = f[a] & NF_D_ZERO;
#pragma unroll
          for (int i = 0; i < 3; ++i) out[a][4 + i] = dz ? T(0) : Rw[a][i].d;
        }
      }
    }
    // Ke[t - t0][a][b][r][k]
    T* o = Ke + 784 * (t - t0) + 49 * b + k;
#pragma unroll
    for (int a = 0; a < 4; ++a)
#pragma unroll
      for (int r = 0; r < 7; ++r) o[196 * a + 7 * r] = out[a][r];
  }
}

// ---------------------------------------------------------------------------
// FP64 element Jacobian in closed form, two kernels. With column (b, k) of a
// fluid tet the derivatives of every intermediate are of rank one in g_b:
//   dG_ij = alpha_i g_b,j, d(grad p) = gamma g_b, d(a_b,k) = eta, d|K| = nu |K|,
//   dg_a = -zeta_a g_b, dD = theta D,
// (u column: alpha = e_k, eta = 1; p: gamma = 1; d: alpha = -G e_k, gamma = -grad p_k,
// eta = -1/dt, nu = g_b,k, zeta_a = g_a,k), so a column is a handful of products of
// per-tet and per-(a, b) values. k_jac_values computes those once per tet (one
// thread per tet), k_elem_jacobian64 one column per thread from them: 28 x ~133
// FP64 instructions per tet in place of 28 x ~1,900 with dual numbers, each of which
// redid the value part. Bound by the FP64 pipe all the same.
// ---------------------------------------------------------------------------
enum : int {  // per-tet values, laid out [JV][tets of the chunk]; fluid tets:
  JV_G = 0,       // gradients g[4][3]
  JV_GU = 12,     // velocity gradient G[3][3]
  JV_GP = 21,     // pressure gradient
  JV_S = 24,      // S_a = sum_c a_c . g_a
  JV_E1 = 28,     // [b][a] factor of alpha_i in the momentum rows
  JV_E2 = 44,     // [b][a] factor of beta_i (the direct part of the inertia's derivative)
  JV_H = 60,      // n_b + W
  JV_Q = 72,      // c Q g_a
  JV_RM = 84,     // momentum residual
  JV_F = 96,      // P g_b
  JV_RC = 108,    // continuity residual
  JV_GR = 112,    // g_a . r |K|/D
  JV_K = 116,     // mesh-motion stiffness [b][a]
  JV_TH = 132,    // theta per unit eta, k = 0..2
  JV_SC = 135,    // |K|, c, |K|/D, |K| tau_C rho div u, |K| tau_C rho
  JV = JAC_VALUES,
  // wall tets: F g0_a, |K0| mu F F^T, [b][a] diagonal part, [b][a] g0_a . g0_b
  JW_F = 0, JW_B = 12, JW_D = 21, JW_GG = 37
};

__global__ void __launch_bounds__(128) k_jac_values(MeshDev m, MatConst mc, const double* __restrict__ y,
                                                    const double* __restrict__ y1, double* __restrict__ val,
                                                    int64_t t0, int64_t t1) {
  const int64_t nt = t1 - t0;
  for (int64_t t = t0 + blockIdx.x * (int64_t)blockDim.x + threadIdx.x; t < t1;
       t += (int64_t)gridDim.x * blockDim.x) {
    double* o = val + (t - t0);
    auto put = [&](int k, double v) { o[k * nt] = v; };
    int n[4];
    uint32_t f[4];
    load_tet(m, t, n, f);
    double g0[3][3], vol0, ga[4][3];
    load_geo(m, t, g0, vol0);
#pragma unroll
    for (int i = 0; i < 3; ++i) {
#pragma unroll
      for (int k = 0; k < 3; ++k) ga[k + 1][i] = g0[k][i];
      ga[0][i] = rest(g0[0][i], g0[1][i], g0[2][i]);
    }
    if (t < m.Tf) {
      FluidValues v;
      {
        const FluidFields q(n, y, y1);
        double Xe[3][3];
        load_edges(m, n, Xe);
        fluid_values(Xe, q.de, q.u, q.p, q.d, q.u1, q.d1, m.geo[10 * m.T + t], m.geo[11 * m.T + t], mc, v);
      }
      const double rho = mc.rho_f, k20 = 0.05 * v.vol;
      {
        double F[4][3], Rm[4][3], gr[4], Rc[4];
        fluid_momentum(v, F, Rm);
        fluid_continuity(v, gr, Rc);
        const double tv = v.ip * v.vol;
#pragma unroll
        for (int a = 0; a < 4; ++a) {
#pragma unroll
          for (int i = 0; i < 3; ++i) {
            put(JV_RM + 3 * a + i, Rm[a][i]);
            put(JV_F + 3 * a + i, F[a][i]);
            put(JV_H + 3 * a + i, v.n[a][i] + v.W[i]);
            put(JV_G + 3 * a + i, v.g[a][i]);
            put(JV_Q + 3 * a + i,
                v.c * (v.Q[i][0] * v.g[a][0] + v.Q[i][1] * v.g[a][1] + v.Q[i][2] * v.g[a][2]));
          }
          put(JV_RC + a, Rc[a]);
          put(JV_GR + a, tv * gr[a]);
        }
#pragma unroll
        for (int i = 0; i < 3; ++i) {
#pragma unroll
          for (int j = 0; j < 3; ++j) put(JV_GU + 3 * i + j, v.G[i][j]);
          put(JV_GP + i, v.gp[i]);
          // dD/D per unit of d(a_b,k): (2 rho / h)^2 (A_k/4) / (4 D^2)
          put(JV_TH + i, mc.ca * m.geo[11 * m.T + t] * v.A[i] * (v.ip * v.ip));
        }
        put(JV_SC + 0, v.vol);
        put(JV_SC + 1, v.c);
        put(JV_SC + 2, tv);
        put(JV_SC + 3, v.vol * v.tc * v.div);
        put(JV_SC + 4, v.vol * v.tc);
      }
      double s[4][4], S[4];  // s[c][a] = a_c . g_a
#pragma unroll
      for (int a = 0; a < 4; ++a) {
#pragma unroll
        for (int c = 0; c < 4; ++c) s[c][a] = v.a[c][0] * v.g[a][0] + v.a[c][1] * v.g[a][1] + v.a[c][2] * v.g[a][2];
        S[a] = (s[0][a] + s[1][a]) + (s[2][a] + s[3][a]);
        put(JV_S + a, S[a]);
      }
      const double rc = rho * v.c, rk = rho * k20, vm = v.vol * mc.mu_f;
#pragma unroll
      for (int b = 0; b < 4; ++b)
#pragma unroll
        for (int a = 0; a < 4; ++a) {
          double zz = S[a] * S[b];
#pragma unroll
          for (int c = 0; c < 4; ++c) zz += s[c][a] * s[c][b];
          const double gg = v.g[a][0] * v.g[b][0] + v.g[a][1] * v.g[b][1] + v.g[a][2] * v.g[b][2];
          put(JV_E1 + 4 * b + a, rc * zz + rk * (S[b] + s[a][b]) + vm * gg);
          put(JV_E2 + 4 * b + a, v.c * (s[b][a] + S[a]) + (a == b ? 2.0 * k20 : k20));
          put(JV_K + 4 * b + a, vol0 * (ga[a][0] * ga[b][0] + ga[a][1] * ga[b][1] + ga[a][2] * ga[b][2]));
        }
    } else {
      double de[3][3], F[3][3], S[3][3];
#pragma unroll
      for (int k = 0; k < 3; ++k)
#pragma unroll
        for (int i = 0; i < 3; ++i) de[k][i] = y[7 * (int64_t)n[k + 1] + 4 + i] - y[7 * (int64_t)n[0] + 4 + i];
      wall_stress(de, g0, mc, F, S);
      const double idt = mc.idt, k20 = vol0 * (1.0 / 20.0) * (mc.rho_s * idt * idt + mc.eta_s * idt);
      double fa[4][3], Sg[4][3];
#pragma unroll
      for (int a = 0; a < 4; ++a)
#pragma unroll
        for (int i = 0; i < 3; ++i) {
          fa[a][i] = F[i][0] * ga[a][0] + F[i][1] * ga[a][1] + F[i][2] * ga[a][2];
          Sg[a][i] = S[i][0] * ga[a][0] + S[i][1] * ga[a][1] + S[i][2] * ga[a][2];
          put(JW_F + 3 * a + i, fa[a][i]);
        }
#pragma unroll
      for (int i = 0; i < 3; ++i)
#pragma unroll
        for (int j = 0; j < 3; ++j)
          put(JW_B + 3 * i + j, vol0 * mc.mu_s * (F[i][0] * F[j][0] + F[i][1] * F[j][1] + F[i][2] * F[j][2]));
#pragma unroll
      for (int b = 0; b < 4; ++b)
#pragma unroll
        for (int a = 0; a < 4; ++a) {
          const double gSg = ga[a][0] * Sg[b][0] + ga[a][1] * Sg[b][1] + ga[a][2] * Sg[b][2];
          put(JW_D + 4 * b + a, vol0 * gSg + (a == b ? 2.0 * k20 : k20));
          put(JW_GG + 4 * b + a, ga[a][0] * ga[b][0] + ga[a][1] * ga[b][1] + ga[a][2] * ga[b][2]);
        }
    }
  }
}

// Column kinds have warps of their own (of a block's 8 tets: three warps of u columns,
// three of d columns, one of p columns): a u column needs 126 FP64 instructions, a d
// column 170, a p column 45, where a mixed warp would run all three.
template <int KIND>  // 0: u column, 1: p, 2: d
__device__ __forceinline__ void fluid_column(const double* s, int b, int kk, double idt, double ridt, double rho, double mu,
                                             const uint32_t f[4], double* o) {
  constexpr bool U = KIND == 0, P = KIND == 1, D = KIND == 2;
  const double* gb = s + JV_G + 3 * b;
  const double vol = s[JV_SC], c = s[JV_SC + 1], tv = s[JV_SC + 2], vmu = vol * mu;
  const double eta = U ? 1.0 : D ? -idt : 0.0;
  const double theta = P ? 0.0 : eta * s[JV_TH + kk];
  const double gam = P ? 1.0 : D ? -s[JV_GP + kk] : 0.0;
  const double nu = D ? gb[kk] : 0.0;
  double al[3], be[3], dr[3];
#pragma unroll
  for (int i = 0; i < 3; ++i) {
    const double Gik = P ? 0.0 : s[JV_GU + 3 * i + kk];
    al[i] = D ? -Gik : 0.0;
    be[i] = P ? 0.0 : rho * eta * Gik;
    if (U && i == kk) be[i] += ridt;
    dr[i] = P ? tv * gb[i] : tv * (0.25 * be[i] + (D ? 0.25 * rho * s[JV_S + b] * al[i] + gam * gb[i] : 0.0));
    if (U && i == kk) dr[i] += tv * (0.25 * rho * s[JV_S + b]);
  }
  const double om = U ? gb[kk] : D ? al[0] * gb[0] + al[1] * gb[1] + al[2] * gb[2] : 0.0;
  const double gac = P ? -0.25 * vol : theta * s[JV_SC + 3] + om * s[JV_SC + 4];
  const double ceta = c * eta, q4 = 0.25 * vol * om, cg5 = 5.0 * c * gam;
#pragma unroll
  for (int a = 0; a < 4; ++a) {
    const double* ga = s + JV_G + 3 * a;
    const double g0 = ga[0], g1 = ga[1], g2 = ga[2];
    const bool uc = f[a] & NF_U_CONSTR, pc = f[a] & NF_P_IDENT, dz = f[a] & NF_D_ZERO, itf = f[a] & NF_ITF;
    const double gk = P ? 0.0 : ga[kk];
    const double e1 = P ? 0.0 : s[JV_E1 + 4 * b + a], e2 = P ? 0.0 : s[JV_E2 + 4 * b + a], hc = ceta * gk;
    const double gbc = U ? vmu * gk
                         : D ? vmu * (al[0] * g0 + al[1] * g1 + al[2] * g2) + cg5 * s[JV_S + a] : cg5 * s[JV_S + a];
    const double K = D ? s[JV_K + 4 * b + a] : 0.0;
#pragma unroll
    for (int i = 0; i < 3; ++i) {
      double r = gb[i] * gbc + (i == 0 ? g0 : i == 1 ? g1 : g2) * gac;
      if (!P) {
        r -= theta * s[JV_Q + 3 * a + i];
        r += be[i] * e2;
        r += s[JV_H + 3 * b + i] * hc;
      }
      if (U && i == kk) r += e1;
      if (D) {
        r += nu * s[JV_RM + 3 * a + i];
        r += al[i] * e1;
        r -= gk * s[JV_F + 3 * b + i];
      }
      o[196 * a + 7 * i] = uc ? 0.0 : r;
      o[196 * a + 7 * (4 + i)] = dz ? 0.0 : (itf ? r : (D && i == kk ? K : 0.0));
    }
    double rc = q4 + g0 * dr[0] + g1 * dr[1] + g2 * dr[2];
    if (!P) rc -= theta * s[JV_GR + a];
    if (D) {
      rc += nu * s[JV_RC + a];
      rc -= gk * s[JV_GR + b];
    }
    o[196 * a + 7 * 3] = pc ? 0.0 : rc;
  }
}

__global__ void __launch_bounds__(28 * JAC_TETS_PER_BLOCK)
k_elem_jacobian64(MeshDev m, MatConst mc, const double* __restrict__ val, double* __restrict__ Ke, int64_t t0,
                  int64_t t1) {
  __shared__ double sv[JAC_TETS_PER_BLOCK][JV + 1];  // odd row length: the tets of a block on other banks
  const int64_t nt = t1 - t0;
  // kind of column, tet of the block, column (b, k)
  const int x = threadIdx.x;
  const int kind = x < 96 ? 0 : x < 192 ? 2 : 1;
  const int y = kind == 0 ? x : kind == 2 ? x - 96 : x - 192;
  const int tl = kind == 1 ? y >> 2 : y / 12, cl = kind == 1 ? y & 3 : y - 12 * tl;
  const int b = kind == 1 ? cl : cl / 3, kk = kind == 1 ? 0 : cl - 3 * b;
  const int k = kind == 0 ? kk : kind == 1 ? 3 : 4 + kk;
  for (int64_t tb = t0 + blockIdx.x * (int64_t)JAC_TETS_PER_BLOCK; tb < t1;
       tb += (int64_t)gridDim.x * JAC_TETS_PER_BLOCK) {
    __syncthreads();
    for (int i = threadIdx.x; i < JV * JAC_TETS_PER_BLOCK; i += 28 * JAC_TETS_PER_BLOCK) {
      const int v = i / JAC_TETS_PER_BLOCK, q = i % JAC_TETS_PER_BLOCK;
      if (tb + q < t1) sv[q][v] = val[v * nt + (tb - t0) + q];
    }
    __syncthreads();
    const int64_t t = tb + tl;
    if (t >= t1) continue;  // (the loop's barriers come before this point for every thread: tb is the block's)
    const double* s = sv[tl];
    int n[4];
    uint32_t f[4];
    load_tet(m, t, n, f);
    double* o = Ke + 784 * (t - t0) + 49 * b + k;
    if (t < m.Tf) {
      const double idt = mc.idt;
      if (kind == 0) fluid_column<0>(s, b, kk, idt, mc.ridt, mc.rho_f, mc.mu_f, f, o);
      else if (kind == 2) fluid_column<2>(s, b, kk, idt, mc.ridt, mc.rho_f, mc.mu_f, f, o);
      else fluid_column<1>(s, b, kk, idt, mc.ridt, mc.rho_f, mc.mu_f, f, o);
    } else if (kind == 2) {
      // d column: |K0| (F S)' g0_a and the inertia
      const double vmu = mc.mu_s * m.geo[9 * m.T + t], vlam = mc.lam_s * m.geo[9 * m.T + t];
      const double fbk = s[JW_F + 3 * b + kk];
#pragma unroll
      for (int a = 0; a < 4; ++a) {
        const bool z = f[a] & NF_D_ZERO;
        const double gg = s[JW_GG + 4 * b + a], fak = vmu * s[JW_F + 3 * a + kk], lb = vlam * fbk;
#pragma unroll
        for (int i = 0; i < 3; ++i) {
          double r = s[JW_B + 3 * i + kk] * gg + s[JW_F + 3 * b + i] * fak + lb * s[JW_F + 3 * a + i];
          if (i == kk) r += s[JW_D + 4 * b + a];
          o[196 * a + 7 * i] = 0.0;
          o[196 * a + 7 * (4 + i)] = z ? 0.0 : r;
        }
        o[196 * a + 7 * 3] = 0.0;
      }
    } else {
#pragma unroll
      for (int a = 0; a < 4; ++a)
#pragma unroll
        for (int r = 0; r < 7; ++r) o[196 * a + 7 * r] = 0.0;
    }
  }
}

__global__ void k_states_to_float(int64_t n, const double* __restrict__ a, const double* __restrict__ b,
                                  const double* __restrict__ c, float* __restrict__ out) {
  for (int64_t i = blockIdx.x * (int64_t)blockDim.x + threadIdx.x; i < n; i += (int64_t)gridDim.x * blockDim.x) {
    out[i] = (float)a[i];
    out[n + i] = (float)b[i];
    out[2 * n + i] = (float)c[i];
  }
}

// Sum into each block the element blocks of the tets [t0, t1) (the buffer holds
// those tets only). Each block's contributions are listed in increasing tet
// order, so a chunk of tets is a contiguous part of every list; the first chunk
// starts the sum at zero, the next ones continue it from vals, so the additions
// happen in the same order as in a single pass (bitwise the same result).
// One warp per block: the lanes read 32 list entries at once and find the chunk's part
// by a ballot, then hold entries lane and lane + 32 of the block, four contributions in
// flight. FP32: bound by memory (the buffer is read once): 527k tets in two chunks 1,255
// -> 664 us against one thread per entry with a 64-bit division each. FP64: by the
// FP64 additions (80k tets 227 -> 218 us).
template <class T>
__global__ void __launch_bounds__(256) k_gather_jacobian(int64_t nnzb, const int64_t* __restrict__ bptr,
                                                         const int32_t* __restrict__ bsrc,
                                                         const T* __restrict__ Ke, T* __restrict__ vals, int64_t t0,
                                                         int64_t t1) {
  const int64_t lo = 16 * t0, hi = 16 * t1;
  const int lane = threadIdx.x & 31;
  const int64_t step = ((int64_t)gridDim.x * blockDim.x) >> 5;
  const bool two = lane < 17;
  for (int64_t kb = (blockIdx.x * (int64_t)blockDim.x + threadIdx.x) >> 5; kb < nnzb; kb += step) {
    T* out = vals + 49 * kb;
    T s0 = T(0), s1 = T(0);
    if (t0 > 0) {
      s0 = out[lane];
      if (two) s1 = out[lane + 32];
    }
    const int64_t c0 = bptr[kb], c1 = bptr[kb + 1];
    bool any = t0 == 0;
    for (int64_t c = c0; c < c1; c += 32) {
      const int src = c + lane < c1 ? bsrc[c + lane] : -1;
      const unsigned in = __ballot_sync(0xffffffffu, src >= lo && src < hi);
      if (in == 0) continue;
      any = true;
      const int b = __ffs(in) - 1, e = b + __popc(in);  // (the chunk's part of the list is contiguous)
      for (int k = b; k < e; k += 4) {
        T v0[4], v1[4];
#pragma unroll
        for (int u = 0; u < 4; ++u) {
          const int64_t q = __shfl_sync(0xffffffffu, src, k + u < e ? k + u : k) - lo;
          v0[u] = k + u < e ? Ke[49 * q + lane] : T(0);
          v1[u] = k + u < e && two ? Ke[49 * q + lane + 32] : T(0);
        }
#pragma unroll
        for (int u = 0; u < 4; ++u)
          if (k + u < e) {
            s0 += v0[u];
            s1 += v1[u];
          }
      }
    }
    if (any) {
      out[lane] = s0;
      if (two) out[lane + 32] = s1;
    }
  }
}

template <class T>
__global__ void k_constraint_jacobian(MeshDev m, MatConst mc, const int32_t* __restrict__ diag, T* __restrict__ vals) {
  for (int64_t i = blockIdx.x * (int64_t)blockDim.x + threadIdx.x; i < m.N; i += (int64_t)gridDim.x * blockDim.x) {
    const uint32_t f = m.nflag[i];
    T* D = vals + 49 * (int64_t)diag[i];
    if (f & (NF_U_KIN | NF_U_IDENT | NF_U_INLET))
      for (int c = 0; c < 3; ++c) D[8 * c] = T(1);
    if (f & NF_U_KIN)
      for (int c = 0; c < 3; ++c) D[7 * c + 4 + c] = T(-1.0 / mc.dt);
    if (f & NF_P_IDENT) D[8 * 3] = T(1);
    if (f & NF_D_ZERO)
      for (int c = 4; c < 7; ++c) D[8 * c] = T(1);
  }
}

inline int grid_for(int64_t work, int block) {
  int64_t g = (work + block - 1) / block;
  const int64_t cap = 152 * 64;
  return (int)(g < 1 ? 1 : (g > cap ? cap : g));
}

}  // namespace

void launch_elem_residual(const MeshDev& m, const MatConst& mc, const double* y, const double* y1,
                          const double* y2, double* Fe, cudaStream_t s) {
  if (m.T == 0) return;
  // one warp per block while that spreads the tets over more SMs: alone on an SM's
  // FP64 pipe a warp issues every 64 cycles, four of them every 76 each
  const int threads = m.T <= 152 * 128 ? 32 : 128;
  k_elem_residual<<<grid_for(m.T, threads), threads, 0, s>>>(m, mc, y, y1, y2, Fe);
}

void launch_gather_residual(const MeshDev& m, const MatConst& mc, double t, const int64_t* nptr, const int32_t* nsrc,
                            const double* Fe, const double* y, const double* y1, double* F, cudaStream_t s) {
  k_gather_residual<<<grid_for(8 * m.N, 256), 256, 0, s>>>(m, mc, t, nptr, nsrc, Fe, y, y1, F);
}

inline int jac_blocks(int64_t nt) {
  const int64_t blocks = (nt + JAC_TETS_PER_BLOCK - 1) / JAC_TETS_PER_BLOCK;
  return (int)(blocks > 152 * 256 ? 152 * 256 : blocks);
}

void launch_geometry(const MeshDev& m, double* geo, cudaStream_t s) {
  if (m.T > 0) k_geometry<<<grid_for(m.T, 128), 128, 0, s>>>(m, geo);
}

void launch_elem_jacobian(const MeshDev& m, const MatConst& mc, const float* Xl, const float* y, const float* y1,
                          const float* y2, float* Ke, int64_t t0, int64_t t1, cudaStream_t s) {
  if (t1 <= t0) return;
  k_elem_jacobian<float><<<jac_blocks(t1 - t0), 28 * JAC_TETS_PER_BLOCK, 0, s>>>(m, mc, Xl, y, y1, y2, Ke, t0, t1);
}

void launch_elem_jacobian(const MeshDev& m, const MatConst& mc, const double* y, const double* y1, double* val,
                          double* Ke, int64_t t0, int64_t t1, cudaStream_t s) {
  if (t1 <= t0) return;
  k_jac_values<<<grid_for(t1 - t0, 128), 128, 0, s>>>(m, mc, y, y1, val, t0, t1);
  k_elem_jacobian64<<<jac_blocks(t1 - t0), 28 * JAC_TETS_PER_BLOCK, 0, s>>>(m, mc, val, Ke, t0, t1);
}

void launch_states_to_float(int64_t n, const double* a, const double* b, const double* c, float* out,
                            cudaStream_t s) {
  k_states_to_float<<<grid_for(n, 256), 256, 0, s>>>(n, a, b, c, out);
}

template <class T>
void launch_gather_jacobian(int64_t nnzb, const int64_t* bptr, const int32_t* bsrc, const T* Ke, T* vals,
                            int64_t t0, int64_t t1, cudaStream_t s) {
  k_gather_jacobian<T><<<grid_for(32 * nnzb, 256), 256, 0, s>>>(nnzb, bptr, bsrc, Ke, vals, t0, t1);
}

template <class T>
void launch_constraint_jacobian(const MeshDev& m, const MatConst& mc, const int32_t* diag, T* vals,
                                cudaStream_t s) {
  k_constraint_jacobian<T><<<grid_for(m.N, 256), 256, 0, s>>>(m, mc, diag, vals);
}

template void launch_gather_jacobian<double>(int64_t, const int64_t*, const int32_t*, const double*, double*,
                                             int64_t, int64_t, cudaStream_t);
template void launch_gather_jacobian<float>(int64_t, const int64_t*, const int32_t*, const float*, float*,
                                            int64_t, int64_t, cudaStream_t);
template void launch_constraint_jacobian<double>(const MeshDev&, const MatConst&, const int32_t*, double*,
                                                 cudaStream_t);
template void launch_constraint_jacobian<float>(const MeshDev&, const MatConst&, const int32_t*, float*,
                                                cudaStream_t);

}  // namespace fsi
