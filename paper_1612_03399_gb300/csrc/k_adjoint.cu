// Adjoint of one step (a vector-Jacobian product): given the cotangents
// (gx', gv') of the new positions and velocities, the cotangents (gx, gv) of
// the old ones and of the per-body elastic constants.
//
// The step (Sec. 2.3, Sec. 5 step 4) is v' = v + dt F(x)/m, x' = x + dt v'
// (symplectic) or x' = x + dt v (forward Euler), F = F_int + F_ext^v; clamped
// nodes keep x and get v' = 0.  So gv = gv' + dt gx', the force cotangent is
// gF = dt (gv' + dt gx')/m (symplectic) or dt gv'/m (forward Euler), zero on
// clamped nodes, and gx = gx' + (dF_int/dx)^T gF + (dF_ext^v/dx)^T gF.
//
// With cotangents g of the spread force fields (Eq. mls_cl), the spread's
// dependence on x (centroid and area of every face) and on v (the face's
// centroid velocity in the marker force) is added as well.
//
// ext_adjoint_kernel (per face): the traction F_ext = mu A (G + G^T) n at the
// probe end p = c + h n (two probes on open sheets) depends on x through A,
// n, c and the MLS velocity gradient G(p); its reverse sweep needs the
// second derivatives of the MLS interpolant at p.  It also sums, per body,
// grad A . gF and grad V . gF (fixed order), which the global area and
// volume terms need.
//
// force_adjoint_kernel (per force patch): the derivatives of the element forces
// along the tangents gF give (dF_int/dx) gF (= its transpose:
// F_int is minus an energy gradient, so its Jacobian is symmetric); the
// constants' cotangents are gF . dF/dk, summed per body in a fixed order.
#include <cuda_runtime.h>

#include <algorithm>

#include "bulk_copy.cuh"
#include "force_elems.cuh"
#include "force_smem.cuh"
#include "ibm_internal.cuh"
#include "mls_closed_form.cuh"

namespace ibm {
namespace {

// gradient (per length) and Hessian (per length squared) of the MLS interpolant
// of velocity component `comp` at tau, and value and gradient on any lattice
__device__ __forceinline__ void grad_hess_at(const float* __restrict__ f, const GlobalRows& R,
                                             const StepConsts& sc, const float (&tau)[3], int comp,
                                             float (&gr)[3], float (&hs)[6]) {
  int c[3];
  float t[3];
  locate(tau, comp, c, t);
  DirH X, Y, Z;
  dir_hess(t[0], sc.mk, X);
  dir_hess(t[1], sc.mk, Y);
  dir_hess(t[2], sc.mk, Z);
  mls_grad_hess(f, R.at(c), X, Y, Z, gr, hs);
#pragma unroll
  for (int j = 0; j < 3; ++j) {
    gr[j] *= sc.kg[j];
    hs[j] *= sc.kg[j] * sc.kg[j];
  }
  hs[3] *= sc.kg[0] * sc.kg[1];
  hs[4] *= sc.kg[0] * sc.kg[2];
  hs[5] *= sc.kg[1] * sc.kg[2];
}
__device__ __forceinline__ void val_grad_at(const float* __restrict__ f, const GlobalRows& R,
                                            const StepConsts& sc, const float (&tau)[3], int comp,
                                            float& val, float (&gr)[3]) {
  int c[3];
  float t[3];
  locate(tau, comp, c, t);
  DirG X, Y, Z;
  dir_grad<true>(t[0], sc.mk, X);
  dir_grad<true>(t[1], sc.mk, Y);
  dir_grad<true>(t[2], sc.mk, Z);
  mls_val_grad(f, R.at(c), X, Y, Z, val, gr);
#pragma unroll
  for (int j = 0; j < 3; ++j) gr[j] *= sc.kg[j];
}

__device__ __forceinline__ float hess_at(const float (&hs)[6], int j, int k) {
  if (j == k) return hs[j];
  const int m = j + k;   // (0,1) -> 1, (0,2) -> 2, (1,2) -> 3
  return hs[2 + m];
}

// force cotangent of vertex gv: dt (gv' + dt gx')/m (symplectic) or dt gv'/m
__device__ __forceinline__ void force_cot(const DeviceTables& T, const StepConsts& sc, int V, int gv,
                                          float inv_mass, const float* __restrict__ gxn,
                                          const float* __restrict__ gvn, float (&o)[3]) {
  if (T.clamp[gv]) {
    o[0] = o[1] = o[2] = 0.f;
    return;
  }
  const float s = sc.dt * inv_mass;
#pragma unroll
  for (int d = 0; d < 3; ++d) {
    const float gvv = __ldg(gvn + d * V + gv);
    o[d] = sc.forward_euler ? s * gvv : s * (gvv + sc.dt * __ldg(gxn + d * V + gv));
  }
}

// Warp sums in float64, which this chip issues at a sixteenth of a warp per cycle
// and SM: after the first exchange each half or quarter of the warp carries one
// quantity, 5 and 6 additions instead of 10 and 15.  Lanes 0 and 16 (0, 8 and 16)
// get the sums; the order is fixed.
__device__ __forceinline__ double warp_sums(double a, double b) {
  const bool up = threadIdx.x & 16;
  double r = up ? b : a;
  r += __shfl_xor_sync(0xffffffffu, up ? a : b, 16);
#pragma unroll
  for (int o = 8; o > 0; o >>= 1) r += __shfl_xor_sync(0xffffffffu, r, o);
  return r;
}
__device__ __forceinline__ double warp_sums(double a, double b, double c) {
  const bool up = threadIdx.x & 16, odd = !up && (threadIdx.x & 8);
  double r = up ? c : a;
  r += __shfl_xor_sync(0xffffffffu, up ? a : c, 16);
  b += __shfl_xor_sync(0xffffffffu, b, 16);
  const double t = __shfl_xor_sync(0xffffffffu, (up || odd) ? r : b, 8);
  r = (odd ? b : r) + t;
#pragma unroll
  for (int o = 4; o > 0; o >>= 1) r += __shfl_xor_sync(0xffffffffu, r, o);
  return r;
}

__device__ __forceinline__ void cross3(const float (&a)[3], const float (&b)[3], float (&o)[3]) {
  o[0] = a[1] * b[2] - a[2] * b[1];
  o[1] = a[2] * b[0] - a[0] * b[2];
  o[2] = a[0] * b[1] - a[1] * b[0];
}

// What bounds it: the latency of the 27-node gathers and of the chain from a
// face to its weights, hidden only by other warps, so registers decide: with the
// values a thread keeps across the gathers in shared memory and the Hessian from
// the closed form's moments (no second-derivative node functions) three blocks
// fit on an SM.  246 k faces (48 bodies): 72.5 us with sixteen derivative
// patterns and two blocks, 55.9 us in this form with two, 52.6 us with three
// (272 bytes of spills), 49.7 us with the packed float64 sums.
__global__ void __launch_bounds__(kMT, 3) ext_adjoint_kernel(
    DeviceTables T, Grid g, StepConsts sc, int32_t V, int32_t F, const float* __restrict__ x,
    const float* __restrict__ vel, const float* __restrict__ u, const float* __restrict__ vv,
    const float* __restrict__ w, const float* __restrict__ pr, const float* __restrict__ accel,
    const float* __restrict__ gxn, const float* __restrict__ gvn, const float* __restrict__ gfx,
    const float* __restrict__ gfy, const float* __restrict__ gfz, float* __restrict__ gve) {
  extern __shared__ __align__(16) float own_[];
  __shared__ double s_red[2][kMT / 32];
  __shared__ int s_last;
  // values a thread needs before and after the field evaluations, kept here and
  // not in registers: normal, force cotangent, edges, probe ends, cotangents of
  // the probe ends, (G + G^T) n and (G + G^T) gF
  float* own = own_ + threadIdx.x;
  enum { kN = 0, kGF = 3, kE1 = 6, kE2 = 9, kTP = 12, kTM = 15, kGP = 18, kGM = 21, kTn = 24, kTg = 27 };
  auto put = [&](int at, const float (&v)[3]) {
#pragma unroll
    for (int d = 0; d < 3; ++d) own[(at + d) * kMT] = v[d];
  };
  auto get = [&](int at, float (&v)[3]) {
#pragma unroll
    for (int d = 0; d < 3; ++d) v[d] = own[(at + d) * kMT];
  };
  const int4 ch = T.chunks[blockIdx.x];
  const BodyDev B = T.body[ch.x];
  const TopoDev topo = T.topo[B.topo];
  double dA = 0.0, dV = 0.0;
  float area = 0.f, inv = 0.f, c[3] = {0.f, 0.f, 0.f};
  int gf = 0, id[3] = {0, 0, 0};
  const bool mine = (int)threadIdx.x < ch.z, two = !B.closed;
  if (mine) {
    const int lf = __ldg(T.mface + topo.mface_off + ch.y + threadIdx.x);
    gf = B.f_off + lf;
    const int* tr = T.tri + topo.tri_off + 3 * lf;
#pragma unroll
    for (int k = 0; k < 3; ++k) id[k] = B.v_off + __ldg(tr + k);
    float p[3][3], ga[3][3];
#pragma unroll
    for (int k = 0; k < 3; ++k) {
#pragma unroll
      for (int d = 0; d < 3; ++d) p[k][d] = __ldg(x + d * V + id[k]);
      force_cot(T, sc, V, id[k], B.inv_mass, gxn, gvn, ga[k]);
    }
    float e1[3], e2[3], N[3];
#pragma unroll
    for (int d = 0; d < 3; ++d) {
      e1[d] = p[1][d] - p[0][d];
      e2[d] = p[2][d] - p[0][d];
    }
    cross3(e1, e2, N);
    const float nn = sqrtf(N[0] * N[0] + N[1] * N[1] + N[2] * N[2]);
    area = 0.5f * nn;
    inv = 1.f / nn;
    const float n[3] = {N[0] * inv, N[1] * inv, N[2] * inv};
    // per-body sums grad A . gF and grad V . gF
    {
      float gVv[3], t[3];
      const float cb[3] = {p[2][0] - p[1][0], p[2][1] - p[1][1], p[2][2] - p[1][2]};
      const float ac[3] = {p[0][0] - p[2][0], p[0][1] - p[2][1], p[0][2] - p[2][2]};
      const float ba[3] = {p[1][0] - p[0][0], p[1][1] - p[0][1], p[1][2] - p[0][2]};
      float sA = 0.f, sV = 0.f;
      cross3(n, cb, t);
      sA += 0.5f * (t[0] * ga[0][0] + t[1] * ga[0][1] + t[2] * ga[0][2]);
      cross3(n, ac, t);
      sA += 0.5f * (t[0] * ga[1][0] + t[1] * ga[1][1] + t[2] * ga[1][2]);
      cross3(n, ba, t);
      sA += 0.5f * (t[0] * ga[2][0] + t[1] * ga[2][1] + t[2] * ga[2][2]);
      if (B.closed) {
        cross3(p[1], p[2], gVv);
        sV += (gVv[0] * ga[0][0] + gVv[1] * ga[0][1] + gVv[2] * ga[0][2]) * (1.f / 6.f);
        cross3(p[2], p[0], gVv);
        sV += (gVv[0] * ga[1][0] + gVv[1] * ga[1][1] + gVv[2] * ga[1][2]) * (1.f / 6.f);
        cross3(p[0], p[1], gVv);
        sV += (gVv[0] * ga[2][0] + gVv[1] * ga[2][1] + gVv[2] * ga[2][2]) * (1.f / 6.f);
      }
      dA = sA;
      dV = sV;
    }
    // traction cotangent: F_ext^v = sum over faces F_ext/3
    float gF[3];
#pragma unroll
    for (int d = 0; d < 3; ++d) gF[d] = (ga[0][d] + ga[1][d] + ga[2][d]) * (1.f / 3.f);
    const float third = 1.f / 3.f;
    float tpp[3], tpm[3];
#pragma unroll
    for (int d = 0; d < 3; ++d) {
      c[d] = (p[0][d] + p[1][d] + p[2][d]) * third;
      tpp[d] = fmaf(c[d] + sc.probe_h * n[d], g.invh[d], B.frac[d]);
      tpm[d] = fmaf(c[d] - sc.probe_h * n[d], g.invh[d], B.frac[d]);
    }
    const float zero[3] = {0.f, 0.f, 0.f};
    put(kN, n);
    put(kGF, gF);
    put(kE1, e1);
    put(kE2, e2);
    put(kTP, tpp);
    put(kTM, tpm);
    put(kGP, zero);
    put(kGM, zero);
    put(kTn, zero);
    put(kTg, zero);
  }
  // fixed-order per-body sums of grad A . gF and grad V . gF
  {
    const double r = warp_sums(dA, dV);
    if ((threadIdx.x & 15) == 0) s_red[(threadIdx.x >> 4) & 1][threadIdx.x >> 5] = r;
  }
  if (mine) {
    // one gradient-and-Hessian evaluation per component and probe end: the
    // gradient forms G, of which (G + G^T) n and (G + G^T) gF are needed, the
    // Hessian the position cotangent of the probe ends,
    // gp_k = sum_ij gG_ij H_ijk with gG_ij = mu A (gF_i n_j + gF_j n_i), which
    // does not depend on G
    const GlobalRows rows{g, {B.G[0], B.G[1], B.G[2]}};
    const float s = sc.mu * area;
#pragma unroll 1
    for (int i = 0; i < 3; ++i) {
      const float* f = i == 0 ? u : (i == 1 ? vv : w);
      float Gi[3] = {0.f, 0.f, 0.f};
#pragma unroll 1
      for (int l = 0; l < (two ? 2 : 1); ++l) {
        const float sg = l == 0 ? 1.f : -1.f;
        float t[3], gr[3], hs[6], n[3], gF[3], gp[3];
        get(kTP + 3 * l, t);
        grad_hess_at(f, rows, sc, t, i, gr, hs);
        get(kN, n);
        get(kGF, gF);
        get(kGP + 3 * l, gp);
        const float ni = own[(kN + i) * kMT], gi = own[(kGF + i) * kMT];
#pragma unroll
        for (int j = 0; j < 3; ++j) {
          Gi[j] += sg * gr[j];
          const float gG = sg * s * (gi * n[j] + gF[j] * ni);
#pragma unroll
          for (int k = 0; k < 3; ++k) gp[k] += gG * hess_at(hs, j, k);
        }
        put(kGP + 3 * l, gp);
      }
      // row i of G: (G n)_i and (G gF)_i, and n_i G_i. and gF_i G_i. for the transposes
      float n[3], gF[3], Tn[3], TgF[3];
      get(kN, n);
      get(kGF, gF);
      get(kTn, Tn);
      get(kTg, TgF);
      const float ni = own[(kN + i) * kMT], gi = own[(kGF + i) * kMT];
      const float gn = Gi[0] * n[0] + Gi[1] * n[1] + Gi[2] * n[2];
      const float gg = Gi[0] * gF[0] + Gi[1] * gF[1] + Gi[2] * gF[2];
#pragma unroll
      for (int j = 0; j < 3; ++j) {
        Tn[j] = fmaf(ni, Gi[j], Tn[j] + (i == j ? gn : 0.f));
        TgF[j] = fmaf(gi, Gi[j], TgF[j] + (i == j ? gg : 0.f));
      }
      put(kTn, Tn);
      put(kTg, TgF);
    }
    float n[3], gF[3], Tn[3], TgF[3], gpp[3], gpm[3];
    get(kN, n);
    get(kGF, gF);
    get(kTn, Tn);
    get(kTg, TgF);
    get(kGP, gpp);
    get(kGM, gpm);
    const float third = 1.f / 3.f;
    // F = mu A (G + G^T) n
    float gArea = sc.mu * (gF[0] * Tn[0] + gF[1] * Tn[1] + gF[2] * Tn[2]);
    float gn[3] = {sc.mu * area * TgF[0], sc.mu * area * TgF[1], sc.mu * area * TgF[2]};
    // p+- = c +- h n
    float gc[3];
#pragma unroll
    for (int d = 0; d < 3; ++d) {
      gc[d] = gpp[d] + gpm[d];
      gn[d] += sc.probe_h * (gpp[d] - gpm[d]);
    }
    if (pr) {
      // pressure load -A P n with P = p*(c + h n) [- p*(c - h n)] + k h a.n,
      // k = 1 (closed) or 2 (open; each side with its own normal); the
      // marker acceleration a is an input and is held fixed
      float am[3] = {0.f, 0.f, 0.f};
      if (accel) {
#pragma unroll
        for (int d = 0; d < 3; ++d)
          am[d] = (__ldg(accel + d * V + id[0]) + __ldg(accel + d * V + id[1]) +
                   __ldg(accel + d * V + id[2])) * third;
      }
      float P, gpr[3], dPdc[3], dPdn[3];
      float t[3];
      get(kTP, t);
      val_grad_at(pr, rows, sc, t, 3, P, gpr);
#pragma unroll
      for (int d = 0; d < 3; ++d) {
        dPdc[d] = gpr[d];
        dPdn[d] = sc.probe_h * dPdc[d];
      }
      if (two) {
        float Pm;
        get(kTM, t);
        val_grad_at(pr, rows, sc, t, 3, Pm, gpr);
        P -= Pm;
#pragma unroll
        for (int d = 0; d < 3; ++d) {
          const float gd = gpr[d];
          dPdc[d] -= gd;
          dPdn[d] += sc.probe_h * gd;
        }
      }
      const float kh = (two ? 2.f : 1.f) * sc.probe_h;
      P += kh * (am[0] * n[0] + am[1] * n[1] + am[2] * n[2]);
      const float gFn = gF[0] * n[0] + gF[1] * n[1] + gF[2] * n[2];
      gArea -= P * gFn;
#pragma unroll
      for (int d = 0; d < 3; ++d) {
        gn[d] -= area * (P * gF[d] + gFn * (dPdn[d] + kh * am[d]));
        gc[d] -= area * gFn * dPdc[d];
      }
    }
    if (gfx) {
      // the spread f_i^k = c_l phi_k(c) F_i with F_i = (V^b_i - U_i(c))/dt,
      // c_l = A cl_scale (Eq. mls_cl), against the field cotangents g_i: with
      // G_i = sum_k phi_k(c) g_i^k (spreading transposed is interpolation),
      // dL/dF_i = c_l G_i, so the vertex velocities get c_l G_i / (3 dt)
      // each, the centroid c_l (F_i grad G_i - G_i grad U_i / dt) and the
      // area cl_scale sum_i F_i G_i
      float tcc[3], vb[3];
#pragma unroll
      for (int d = 0; d < 3; ++d) {
        tcc[d] = fmaf(c[d], g.invh[d], B.frac[d]);
        vb[d] = (__ldg(vel + d * V + id[0]) + __ldg(vel + d * V + id[1]) +
                 __ldg(vel + d * V + id[2])) * third;
      }
      const float cl = area * sc.cl_scale;
      float gAs = 0.f;
#pragma unroll 1
      for (int i = 0; i < 3; ++i) {
        float Uv, Ug[3], Gv, Gg[3];
        val_grad_at(i == 0 ? u : (i == 1 ? vv : w), rows, sc, tcc, i, Uv, Ug);
        val_grad_at(i == 0 ? gfx : (i == 1 ? gfy : gfz), rows, sc, tcc, i, Gv, Gg);
        const float Fi = ((i == 0 ? vb[0] : (i == 1 ? vb[1] : vb[2])) - Uv) * sc.inv_dt;
        gAs += Fi * Gv;
#pragma unroll
        for (int d = 0; d < 3; ++d) gc[d] += cl * (Fi * Gg[d] - Gv * sc.inv_dt * Ug[d]);
        gve[i * (size_t)F + gf] = cl * Gv * sc.inv_dt * third;
      }
      gArea += sc.cl_scale * gAs;
    }
    // n = N/|N|, A = |N|/2
    const float gnn = gn[0] * n[0] + gn[1] * n[1] + gn[2] * n[2];
    float gN[3];
#pragma unroll
    for (int d = 0; d < 3; ++d) gN[d] = (gn[d] - gnn * n[d]) * inv + 0.5f * gArea * n[d];
    // N = e1 x e2
    float ge1[3], ge2[3], e1[3], e2[3];
    get(kE1, e1);
    get(kE2, e2);
    cross3(e2, gN, ge1);
    cross3(gN, e1, ge2);
#pragma unroll
    for (int d = 0; d < 3; ++d) {
      const float gcd = gc[d] * third;
      T.gxe[(0 * 3 + d) * (size_t)F + gf] = -ge1[d] - ge2[d] + gcd;
      T.gxe[(1 * 3 + d) * (size_t)F + gf] = ge1[d] + gcd;
      T.gxe[(2 * 3 + d) * (size_t)F + gf] = ge2[d] + gcd;
    }
  }
  __syncthreads();
  if (threadIdx.x == 0) {
    double a = 0.0, b = 0.0;
    for (int k = 0; k < kMT / 32; ++k) {
      a += s_red[0][k];
      b += s_red[1][k];
    }
    const int gc = B.chunk_off + ch.w;
    T.partial2[2 * gc] = a;
    T.partial2[2 * gc + 1] = b;
    __threadfence();
    s_last = (atomicAdd(T.counter2 + ch.x, 1) == B.n_chunk - 1);
  }
  __syncthreads();
  if (s_last && threadIdx.x < 32) {   // lanes take every 32nd chunk: a fixed order again
    __threadfence();
    double a = 0.0, b = 0.0;
    for (int k = threadIdx.x; k < B.n_chunk; k += 32) {
      a += __ldcg(T.partial2 + 2 * (B.chunk_off + k));
      b += __ldcg(T.partial2 + 2 * (B.chunk_off + k) + 1);
    }
    const double r = warp_sums(a, b);
    if ((threadIdx.x & 15) == 0) T.dmeas[2 * ch.x + (threadIdx.x >> 4)] = r;
    if (threadIdx.x == 0) T.counter2[ch.x] = 0;
  }
}

constexpr size_t kExtBytes = 30 * sizeof(float) * kMT;   // ext_adjoint_kernel's values per thread

// What bounds it: latency (record -> index -> position, tractions' cotangents)
// and its barriers, as the force kernel; float64 instructions issue at a
// sixteenth of a warp per cycle and SM, so only what must be float64 is, once
// per block where it can be.  48 bodies (246 k faces, 960 patches): 64.9 us with
// generic forward-mode numbers, narrow slots and a float64 division per thread;
// 48.1 us with the derivatives written out (*_tangent) and float4 slots; 41.9 us
// with the division per block and the packed warp sums; 36.1 us with the faces
// and their corners' cotangents on the edges instead of a chain of loads per
// vertex.  Three blocks of at most 160 threads fit an SM's registers: 35.7 us,
// 40.6 with 192.  The layout goes by the force kernel's rule: float4 where it costs
// no resident block.
template <bool WIDE>
__global__ void __launch_bounds__(kAdjointThreads, 3) force_adjoint_kernel(
    DeviceTables T, StepConsts sc, int32_t V, int32_t F, const float* __restrict__ x,
    const float* __restrict__ gxn, const float* __restrict__ gvn, float* __restrict__ gx,
    float* __restrict__ gvo, double* __restrict__ gparams, const float* __restrict__ gve) {
  extern __shared__ __align__(16) float sm[];
  __shared__ double s_red[3][kAdjointThreads / 32];
  __shared__ int s_last;
  __shared__ __align__(8) unsigned long long bar;
  const FWork P = T.fwork[blockIdx.x];
  const BodyDev& B = T.body[P.body];
  // the forward kernel's blob (edge and face records, slot starts) with the
  // adjoint's tail (each own vertex's faces and corners), the rest data,
  // positions and tangents of the local vertices, contribution slots
  const int pe = pad4(P.n_edge), pf = pad4(P.n_face);
  const uint4* rec = reinterpret_cast<const uint4*>(sm);
  const uint2* frec = reinterpret_cast<const uint2*>(sm + 4 * P.n_edge);
  const uint16_t* ptr = reinterpret_cast<const uint16_t*>(sm + 4 * P.n_edge + 2 * P.n_face);
  const uint16_t* vptr = reinterpret_cast<const uint16_t*>(sm + P.blob_words);
  const uint32_t* vent = reinterpret_cast<const uint32_t*>(sm + P.blob_words) + (P.n_own + 2) / 2;
  const float* rest = sm + P.blob_words + P.vf_words;
  // S: positions and slots; Y: tangents (its slots are S's)
  Smem<WIDE> S, Y;
  {
    float* at = sm + P.blob_words + P.vf_words + P.rest_words;
    Y.init(at, P.n_loc, P.n_slot);
    S.init(at + (WIDE ? 4 : 3) * P.n_loc, P.n_loc, P.n_slot);
  }
  if (threadIdx.x == 0) {
    mbar_init(&bar, 1);
    const unsigned nb = 4u * (unsigned)(P.blob_words + P.vf_words),
                   nr = 4u * (unsigned)P.rest_words;
    mbar_arrive_tx(&bar, nb + nr + (unsigned)sc.starve_tx);
    if (nb) bulk_load(sm, T.fblob + P.blob_off, nb, &bar);
    if (nr) bulk_load(sm + P.blob_words + P.vf_words, T.frest + P.rest, nr, &bar);
  }
  for (int i = threadIdx.x; i < P.n_loc; i += blockDim.x) {
    const int gvx = P.v_off + __ldg(T.loc_vert + P.loc_off + i);
    S.set(i, __ldg(x + gvx), __ldg(x + V + gvx), __ldg(x + 2 * V + gvx));
    float o[3];
    force_cot(T, sc, V, gvx, B.inv_mass, gxn, gvn, o);
    Y.set(i, o[0], o[1], o[2]);
  }
  // global-term coefficients and their derivatives along gF
  const float2 cf = T.coef[P.body];
  if (threadIdx.x == 0) {   // (in every thread the divisions took 2 us a block)
    s_red[0][0] = B.kA / B.A0 * T.dmeas[2 * P.body];
    s_red[0][1] = B.closed ? B.kv / B.V0 * T.dmeas[2 * P.body + 1] : 0.0;
  }
  const float Bks = B.ks, Bkb = B.kb, Bka = B.ka;
  double gks = 0.0, gkb = 0.0, gka = 0.0;
  __syncthreads();   // positions and tangents staged, barrier initialised
  if (!__syncthreads_and(mbar_wait(&bar, kCopyWaitClocks))) {
    // the copies did not land: flag it, give them one more bounded wait
    // (they write this block's shared memory) and leave
    if (threadIdx.x == 0) {
      atomicOr(T.err, ERR_TIMEOUT);
      mbar_wait(&bar, kCopyWaitClocks);
    }
    __syncthreads();
    return;
  }
  const float cAd = (float)s_red[0][0], cVd = (float)s_red[0][1];   // before the barriers below
  // edges: spring, bending and the face attached to the edge (edge k's face is
  // face k)
  for (int k = threadIdx.x; k < P.n_edge; k += blockDim.x) {
    const uint4 r = rec[k];
    const bool face = k < P.n_face;
    uint2 fr = make_uint2(0u, 0u);
    Vec<float> tc[3] = {};
    if (face) {
      fr = frec[k];
      const float* t = T.gxe + P.f_off + fr.y;
      int corner = (fr.x >> 28) & 3;
#pragma unroll
      for (int j = 0; j < 3; ++j) {
        const float* tj = t + 3 * (size_t)corner * F;
        tc[j] = {__ldg(tj), __ldg(tj + F), __ldg(tj + 2 * (size_t)F)};
        corner = corner == 2 ? 0 : corner + 1;
      }
    }
    const int la = r.x & 0xFFFF, lb = r.x >> 16, lc = r.y & 0xFFFF, ld = r.y >> 16;
    const bool hinge = ld != kNone;
    const int wd = hinge ? ld : la;
    const Vec<float> pa = S.pos(la), ya = Y.pos(la);
    const Vec<float> e = vsub(S.pos(lb), pa), ed = vsub(Y.pos(lb), ya);
    const Vec<float> ac = vsub(S.pos(lc), pa), acd = vsub(Y.pos(lc), ya);
    const Vec<float> ad = vsub(S.pos(wd), pa), add = vsub(Y.pos(wd), ya);
    // per-element multipliers m: the forces use m k, the constants' cotangents
    // scale the per-unit-k forces by m
    const float ms = P.varied ? rest[3 * pe + pf + k] : 1.f;
    const float mb = P.varied ? rest[4 * pe + pf + k] : 1.f;
    Vec<float> fa, fb, fc = {0.f, 0.f, 0.f}, fd = {0.f, 0.f, 0.f};
    float l, ld_, il, ild, us, ub = 0.f;
    spring_tangent(e, ed, rest[k], Bks * ms, l, ld_, il, ild, fa, us);
    fb = {-fa.x, -fa.y, -fa.z};
    const Vec<float> N1 = vcross(e, ac), N2 = vcross(ad, e);
    const Vec<float> N1d = vadd(vcross(ed, ac), vcross(e, acd));
    const Vec<float> N2d = vadd(vcross(add, e), vcross(ad, ed));
    const float r1 = rsqrtf(vdot(N1, N1)), r2 = rsqrtf(vdot(N2, N2));
    const float h1 = r1 * r1 * vdot(N1, N1d), h2 = r2 * r2 * vdot(N2, N2d);
    if (hinge)
      hinge_tangent(e, ed, l, ld_, il, ild, ac, acd, ad, add, N1, N1d, N2, N2d, r1, r2, h1, h2,
                    rest[pe + k], rest[2 * pe + k], Bkb * mb, fa, fb, fc, fd, ub);
    if (face) {
      const bool right = (fr.x >> 30) & 1u;
      const float ma = P.varied ? rest[5 * pe + pf + k] : 1.f;
      Vec<float> fw = right ? fd : fc;
      float ua;
      face_tangent(e, ed, right ? ad : ac, right ? add : acd, right ? N2 : N1, right ? N2d : N1d,
                   right ? r2 : r1, right ? h2 : h1, right ? -1.f : 1.f, rest[3 * pe + k], Bka * ma,
                   cf.x, cAd, cf.y, cVd, fa, fb, fw, ua);
      if (right)
        fd = fw;
      else
        fc = fw;
      if (fr.x >> 31) gka += ma * ua;
      // traction part: the cotangents the face left for its corners
      const Vec<float>&t0 = right ? tc[1] : tc[0], &t1 = right ? tc[0] : tc[1];
      fa = vadd(fa, t0);
      fb = vadd(fb, t1);
      if (right)
        fd = vadd(fd, tc[2]);
      else
        fc = vadd(fc, tc[2]);
    }
    S.put(r.z & 0xFFFF, fa);
    S.put(r.z >> 16, fb);
    S.put(r.w & 0xFFFF, fc);
    S.put(r.w >> 16, fd);
    if ((r.z & 0xFFFF) != kNone) {   // owned edge: constants' cotangents
      gks += ms * us;
      gkb += mb * ub;
    }
  }
  __syncthreads();
  for (int i = threadIdx.x; i < P.n_own; i += blockDim.x) {
    const Vec<float> js = slot_sum(S, i, ptr[i], ptr[i + 1]);
    const float jx = js.x, jy = js.y, jz = js.z;
    const int gvx = P.v_off + P.own0 + i;
    float wx = 0.f, wy = 0.f, wz = 0.f;   // the spread's velocity cotangent
    if (gve) {
      for (int q = vptr[i]; q < vptr[i + 1]; ++q) {
        const size_t gf = (size_t)P.f_off + (vent[q] & 0x3FFFFFFFu);
        wx += __ldg(gve + gf);
        wy += __ldg(gve + (size_t)F + gf);
        wz += __ldg(gve + 2 * (size_t)F + gf);
      }
    }
    const bool cl = T.clamp[gvx] != 0;
    const float gx0 = __ldg(gxn + gvx), gx1 = __ldg(gxn + V + gvx), gx2 = __ldg(gxn + 2 * V + gvx);
    gx[gvx] = gx0 + jx;
    gx[V + gvx] = gx1 + jy;
    gx[2 * V + gvx] = gx2 + jz;
    // a clamped node's new state does not depend on its velocity; the spread
    // (the centroid velocity of its faces) does
    gvo[gvx] = (cl ? 0.f : __ldg(gvn + gvx) + sc.dt * gx0) + wx;
    gvo[V + gvx] = (cl ? 0.f : __ldg(gvn + V + gvx) + sc.dt * gx1) + wy;
    gvo[2 * V + gvx] = (cl ? 0.f : __ldg(gvn + 2 * V + gvx) + sc.dt * gx2) + wz;
  }
  const int n_patch = T.topo[B.topo].n_patch;
  // constants' cotangents: fixed-order per-patch sums, then per body
  {
    const double r = warp_sums(gks, gkb, gka);
    const int q = (threadIdx.x & 31) >> 3;
    if ((threadIdx.x & 7) == 0 && q < 3) s_red[q][threadIdx.x >> 5] = r;
  }
  __syncthreads();
  if (threadIdx.x == 0) {
    double a = 0.0, b = 0.0, c = 0.0;
    for (int k = 0; k < (int)(blockDim.x >> 5); ++k) {
      a += s_red[0][k];
      b += s_red[1][k];
      c += s_red[2][k];
    }
    T.wpart[3 * (size_t)blockIdx.x] = a;
    T.wpart[3 * (size_t)blockIdx.x + 1] = b;
    T.wpart[3 * (size_t)blockIdx.x + 2] = c;
    __threadfence();
    s_last = (atomicAdd(T.wcounter + P.body, 1) == n_patch - 1);
  }
  __syncthreads();
  if (s_last && threadIdx.x < 32) {
    __threadfence();
    double a = 0.0, b = 0.0, c = 0.0;
    for (int k = threadIdx.x; k < n_patch; k += 32) {
      const double* W = T.wpart + 3 * (size_t)(B.work_off + k);
      a += __ldcg(W);
      b += __ldcg(W + 1);
      c += __ldcg(W + 2);
    }
    const double r = warp_sums(a, b, c);
    const int q = threadIdx.x >> 3;
    if ((threadIdx.x & 7) == 0 && q < 3) gparams[5 * P.body + q] = r;
    if (threadIdx.x == 0) {
      const double Ab = T.meas[2 * P.body], Vb = T.meas[2 * P.body + 1];
      gparams[5 * P.body + 3] = -(Ab - B.A0) / B.A0 * T.dmeas[2 * P.body];
      gparams[5 * P.body + 4] = B.closed ? -(Vb - B.V0) / B.V0 * T.dmeas[2 * P.body + 1] : 0.0;
      T.wcounter[P.body] = 0;
    }
  }
}

}  // namespace

cudaError_t launch_backward(ibm_ctx* c, const float* x, const float* v, const float* u,
                            const float* vv, const float* w, const float* pr, const float* accel,
                            const float* gx_next, const float* gv_next, const float* gfx,
                            const float* gfy, const float* gfz, float* gx, float* gv,
                            double* gparams) {
  if (c->n_chunks == 0) return cudaSuccess;
  // area, volume and the global-term coefficients at x
  cudaError_t e = zero_body_sums(c);
  if (e == cudaSuccess)
    e = launch_mls(c, x, nullptr, nullptr, nullptr, nullptr, nullptr, nullptr, nullptr, nullptr,
                   nullptr, nullptr, nullptr, nullptr, nullptr, true, false, false, false, false);
  if (e == cudaSuccess) e = launch_measure_finalize(c);
  if (e != cudaSuccess) return e;
  // per-face velocity cotangents of the spread go to the step's F_ext scratch,
  // unused by the adjoint otherwise
  float* gve = gfx ? c->d.fext : nullptr;
  ext_adjoint_kernel<<<c->n_chunks, kMT, kExtBytes, c->stream>>>(
      c->d, c->grid, c->sc, (int32_t)c->V, (int32_t)c->F, x, v, u, vv, w, pr, accel, gx_next, gv_next,
      gfx, gfy, gfz, gve);
  e = cudaGetLastError();
  if (e != cudaSuccess) return e;
  auto kernel = c->adjoint_wide ? force_adjoint_kernel<true> : force_adjoint_kernel<false>;
  kernel<<<c->n_work, std::min(c->force_threads, kAdjointThreads), c->adjoint_smem, c->stream>>>(
      c->d, c->sc, (int32_t)c->V, (int32_t)c->F, x, gx_next, gv_next, gx, gv, gparams, gve);
  return cudaGetLastError();
}

static cudaError_t adjoint_smem_room(size_t* room) {
  *room = SIZE_MAX;
  const cudaError_t e = smem_room(force_adjoint_kernel<true>, room);
  return e == cudaSuccess ? smem_room(force_adjoint_kernel<false>, room) : e;
}
cudaError_t set_adjoint_smem_limit(size_t bytes) {
  const cudaError_t e = allow_smem(force_adjoint_kernel<true>, bytes);
  return e == cudaSuccess ? allow_smem(force_adjoint_kernel<false>, bytes) : e;
}

cudaError_t adjoint_occupancy(int threads, size_t wide_bytes, size_t narrow_bytes, int* wide, int* narrow) {
  size_t room = 0;
  cudaError_t e = adjoint_smem_room(&room);
  *wide = *narrow = 0;
  threads = std::min(threads, kAdjointThreads);
  if (e == cudaSuccess) e = set_adjoint_smem_limit(0);
  if (e == cudaSuccess && wide_bytes <= room)
    e = cudaOccupancyMaxActiveBlocksPerMultiprocessor(wide, force_adjoint_kernel<true>, threads, wide_bytes);
  if (e == cudaSuccess && narrow_bytes <= room)
    e = cudaOccupancyMaxActiveBlocksPerMultiprocessor(narrow, force_adjoint_kernel<false>, threads,
                                                      narrow_bytes);
  return e;
}

}  // namespace ibm
