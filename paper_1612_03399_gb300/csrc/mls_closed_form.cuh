// Closed-form MLS shape functions of the factorised weight and their use on
// 3x3x3 supports (Sec. 2.2, Eqs. mls..mls_Q), shared by the marker, tile-spread
// and adjoint kernels.
//
// MLS with the linear basis and a weight that factorises over directions
// (W = prod_d exp(-kappa delta_d^2), delta in cells) has an exact closed-form
// solution of the 4x4 moment system.  Per direction, for the point at the
// offset t in [-1/2, 1/2) from its nearest node and the nodes s = -1, 0, 1,
// with the normalised weights a_s (sum 1), their mean m = sum a_s s, the
// centred nodes e_s = s - m, the variance s2 = sum a_s e_s^2 and r = (m - t)/s2:
//   phi(sx,sy,sz) = a_x a_y a_z (1 - r_x e_x - r_y e_y - r_z e_z).
// Everything is a function of central moments, because the Gaussian weight has
// da_s/dt = 2 kappa a_s e_s, hence dm/dt = 2 kappa s2.  With the node functions
//   alpha = a_s,  gamma = a_s e_s,  delta = a_s (e_s^2 - s2)
// (delta sums to 0 like gamma), so that d alpha/dt = 2 kappa gamma and
// d gamma/dt = 2 kappa delta,
//   phi       = aaa - r_x gaa - r_y aga - r_z aag,
//   d phi/dtx = 2 kappa (h_x gaa - r_x daa - r_y gga - r_z gag)   (y, z alike),
// a, g, d short for alpha, gamma, delta and h = 1 - dr/dt / (2 kappa)
// = (1/(2 kappa) + r mu3)/s2, mu3 the third central moment.  A gradient needs
// nine tensor sums of the three node functions instead of the sixteen
// products of (a, b = a beta) and their derivatives, and the factors of a
// direction take two exponentials, two reciprocals and about twenty
// operations.
//
// The sums are formed from differences to the middle node (alpha sums to 1,
// gamma and delta to 0): a constant offset of the field never enters a
// product, so the gradient carries no rounding of the field's magnitude.
// Against float64 the float32 gradient of a field of magnitude 1 with
// increments of 5 % per cell is 1e-7 .. 1e-6 relative (6e-6 from the plain
// weighted sums), the value 6e-8 (1.3e-7).
#pragma once

#include <cuda_runtime.h>
#include <limits.h>
#include <math.h>

#include "ibm_internal.cuh"

namespace ibm {
namespace {

// 2^x and 1/x by the special-function unit (1/x: the marker and spread kernels).
// Arguments are in its full precision range: |x| <= 2 kappa log2(e) / 2, and sums of
// weights or variances of at least the smallest normal number (below it the closed
// form has no float32 value).
__device__ __forceinline__ float ex2_fast(float x) {
  float y;
  asm("ex2.approx.ftz.f32 %0, %1;" : "=f"(y) : "f"(x));
  return y;
}
__device__ __forceinline__ float rcp_fast(float x) {
  float y;
  asm("rcp.approx.ftz.f32 %0, %1;" : "=f"(y) : "f"(x));
  return y;
}

// weights of one direction: a_s, and b_s = a_s r e_s of the outer nodes (the
// middle one is -(b0 + b2))
struct DirW {
  float a0, a1, a2, b0, b2;
};
// node functions of one direction at the outer nodes, r and h
struct DirG {
  float a0, a2, c0, c2, g0, g2, r, h;
};

// The weights enter only through their ratios to the nearest node's,
//   w(-1)/w(0) = e^-kappa 2^-z,  w(+1)/w(0) = e^-kappa 2^z,  z = 2 kappa log2(e) t,
// both in (0, 1].
__device__ __forceinline__ void dir_weights(float t, const MlsK& K, DirW& o) {
  const float z = K.z * t;
  const float rm = K.ek * ex2_fast(-z), rp = K.ek * ex2_fast(z);
  o.a1 = rcp_fast(1.f + rm + rp);
  o.a0 = rm * o.a1;
  o.a2 = rp * o.a1;
  const float m = o.a2 - o.a0;
  const float s2 = fmaf(-m, m, o.a0 + o.a2);
  const float r = (m - t) * rcp_fast(s2);
  o.b0 = -r * fmaf(o.a0, m, o.a0);
  o.b2 = r * fmaf(-o.a2, m, o.a2);
}

// IEEE: the reciprocals rounded correctly (the adjoint's); returns 1/s2
template <bool IEEE = false>
__device__ __forceinline__ float dir_grad(float t, const MlsK& K, DirG& o) {
  auto rcp = [](float x) { return IEEE ? 1.f / x : rcp_fast(x); };
  const float z = K.z * t;
  const float rm = K.ek * ex2_fast(-z), rp = K.ek * ex2_fast(z);
  const float i = rcp(1.f + rm + rp);
  o.a0 = rm * i;
  o.a2 = rp * i;
  const float m = o.a2 - o.a0, q = o.a0 + o.a2;
  const float s2 = fmaf(-m, m, q);
  const float is2 = rcp(s2);
  o.r = (m - t) * is2;
  o.c0 = -fmaf(o.a0, m, o.a0);
  o.c2 = fmaf(-o.a2, m, o.a2);
  o.g0 = -fmaf(o.c0, 1.f + m, o.a0 * s2);   // a0 e0^2 - a0 s2
  o.g2 = fmaf(o.c2, 1.f - m, -o.a2 * s2);
  const float mu3 = m * fmaf(-3.f, q, fmaf(2.f * m, m, 1.f));
  o.h = fmaf(o.r, mu3, K.hk) * is2;
  return is2;
}

__device__ __forceinline__ int wrap(int i, int n) {
  if (i >= 0 && i < n) return i;
  if (i < 0 && i >= -n) return i + n;
  if (i >= n && i < 2 * n) return i - n;
  i %= n;
  return i < 0 ? i + n : i;
}

// Centre node (lattice index relative to the cell G that tau is measured from)
// and fractional offset of a point, in every direction, on the lattice of
// velocity component `comp` (node offset 0 along the component's own
// direction, 1/2 across it; comp 3: the cell centres).
__device__ __forceinline__ void locate(const float (&tau)[3], int comp, int (&c)[3],
                                       float (&tp)[3]) {
#pragma unroll
  for (int d = 0; d < 3; ++d) {
    const float u = tau[d] - (d == comp ? 0.f : 0.5f);
    const float cc = floorf(u + 0.5f);
    tp[d] = u - cc;
    c[d] = (int)cc;
  }
}

// addressing of a 3x3x3 support: row (sy, sz) of three nodes in x
struct GlobalAcc {   // wrapped indices into a full [nz][ny][nx] field
  int ix[3], iy[3], iz[3];
  int nx, ny;
  __device__ __forceinline__ void init(const int (&c)[3], const int (&G)[3], const Grid& g) {
    nx = g.n[0];
    ny = g.n[1];
#pragma unroll
    for (int s = 0; s < 3; ++s) {
      ix[s] = wrap(G[0] + c[0] - 1 + s, g.n[0]);
      iy[s] = wrap(G[1] + c[1] - 1 + s, g.n[1]);
      iz[s] = wrap(G[2] + c[2] - 1 + s, g.n[2]);
    }
  }
  __device__ __forceinline__ size_t row(int sy, int sz) const {
    return (size_t)(unsigned)(iz[sz] * ny + iy[sy]) * (unsigned)nx;   // (rows fit 32 bits)
  }
  __device__ __forceinline__ void load(const float* __restrict__ f, int sy, int sz,
                                       float (&u)[3]) const {
    const float* r = f + row(sy, sz);
#pragma unroll
    for (int s = 0; s < 3; ++s) u[s] = __ldg(r + ix[s]);
  }
};
struct RowAcc {      // rows staged in shared memory
  const unsigned char* sm;   // the block's shared memory; the row table lies at its start
  int off;           // index of the table entry of the support's first row (centre - 1 in y, z)
  int sy;            // rows per z plane of the table
  int x4;            // byte offset of the buffer + 4 (centre x - 1)
  // byte offset of row (a, b) of the support
  __device__ __forceinline__ int row(int a, int b) const {
    return reinterpret_cast<const int*>(sm)[off + a + sy * b] + x4;
  }
  __device__ __forceinline__ void load(const float*, int a, int b, float (&u)[3]) const {
    const float* r = reinterpret_cast<const float*>(sm + row(a, b));
    u[0] = r[0];
    u[1] = r[1];
    u[2] = r[2];
  }
};

// value: per row the a-sum A and the (a - b)-sum W, per plane S = sum_y a_y A
// and T = sum_y (a_y W - b_y A), then sum_z (a_z T - b_z S)
template <class Acc>
__device__ __forceinline__ float mls_value(const float* __restrict__ f, const Acc& A, const DirW& X,
                                           const DirW& Y, const DirW& Z) {
  const float w0 = X.a0 - X.b0, w2 = X.a2 - X.b2;
  float S[3], T[3];
#pragma unroll
  for (int sz = 0; sz < 3; ++sz) {
    float a[3], w[3];
#pragma unroll
    for (int sy = 0; sy < 3; ++sy) {
      float u[3];
      A.load(f, sy, sz, u);
      const float d0 = u[0] - u[1], d2 = u[2] - u[1];
      a[sy] = fmaf(X.a2, d2, fmaf(X.a0, d0, u[1]));
      w[sy] = fmaf(w2, d2, fmaf(w0, d0, u[1]));
    }
    const float d0 = a[0] - a[1], d2 = a[2] - a[1];
    S[sz] = fmaf(Y.a2, d2, fmaf(Y.a0, d0, a[1]));
    T[sz] = fmaf(Y.a2, w[2] - w[1], fmaf(Y.a0, w[0] - w[1], w[1]));
    T[sz] = fmaf(-Y.b2, d2, fmaf(-Y.b0, d0, T[sz]));
  }
  const float U = fmaf(Z.a2, T[2] - T[1], fmaf(Z.a0, T[0] - T[1], T[1]));
  return fmaf(-Z.b2, S[2] - S[1], fmaf(-Z.b0, S[0] - S[1], U));
}

// sums of one z plane over (x, y): aa, ca, ac, ga, ag, cc (first letter x)
struct PlaneG {
  float aa, ca, ac, ga, ag, cc;
};
template <class Acc>
__device__ __forceinline__ PlaneG plane_sums(const float* __restrict__ f, const Acc& A, int sz,
                                             const DirG& X, const DirG& Y) {
  float a[3], c[3], g[3];
#pragma unroll
  for (int sy = 0; sy < 3; ++sy) {
    float u[3];
    A.load(f, sy, sz, u);
    const float d0 = u[0] - u[1], d2 = u[2] - u[1];
    a[sy] = fmaf(X.a2, d2, fmaf(X.a0, d0, u[1]));
    c[sy] = fmaf(X.c2, d2, X.c0 * d0);
    g[sy] = fmaf(X.g2, d2, X.g0 * d0);
  }
  PlaneG P;
  const float a0 = a[0] - a[1], a2 = a[2] - a[1];
  const float c0 = c[0] - c[1], c2 = c[2] - c[1];
  P.aa = fmaf(Y.a2, a2, fmaf(Y.a0, a0, a[1]));
  P.ac = fmaf(Y.c2, a2, Y.c0 * a0);
  P.ag = fmaf(Y.g2, a2, Y.g0 * a0);
  P.ca = fmaf(Y.a2, c2, fmaf(Y.a0, c0, c[1]));
  P.cc = fmaf(Y.c2, c2, Y.c0 * c0);
  P.ga = fmaf(Y.a2, g[2] - g[1], fmaf(Y.a0, g[0] - g[1], g[1]));
  return P;
}

// full-derivative gradient in cells, divided by 2 kappa
template <class Acc>
__device__ __forceinline__ void mls_grad(const float* __restrict__ f, const Acc& A, const DirG& X,
                                         const DirG& Y, const DirG& Z, float (&gr)[3]) {
  const PlaneG P1 = plane_sums(f, A, 1, X, Y);
  float caa = P1.ca, aca = P1.ac, aac = 0.f, gaa = P1.ga, aga = P1.ag, aag = 0.f, cca = P1.cc,
        cac = 0.f, acc = 0.f;
#pragma unroll
  for (int k = 0; k < 2; ++k) {
    const PlaneG P = plane_sums(f, A, 2 * k, X, Y);
    const float za = k ? Z.a2 : Z.a0, zc = k ? Z.c2 : Z.c0, zg = k ? Z.g2 : Z.g0;
    const float daa = P.aa - P1.aa, dca = P.ca - P1.ca, dac = P.ac - P1.ac;
    aac = fmaf(zc, daa, aac);
    aag = fmaf(zg, daa, aag);
    caa = fmaf(za, dca, caa);
    cac = fmaf(zc, dca, cac);
    aca = fmaf(za, dac, aca);
    acc = fmaf(zc, dac, acc);
    gaa = fmaf(za, P.ga - P1.ga, gaa);
    aga = fmaf(za, P.ag - P1.ag, aga);
    cca = fmaf(za, P.cc - P1.cc, cca);
  }
  gr[0] = fmaf(X.h, caa, -fmaf(X.r, gaa, fmaf(Y.r, cca, Z.r * cac)));
  gr[1] = fmaf(Y.h, aca, -fmaf(Y.r, aga, fmaf(X.r, cca, Z.r * acc)));
  gr[2] = fmaf(Z.h, aac, -fmaf(Z.r, aag, fmaf(X.r, cac, Y.r * acc)));
}

// Second derivatives (the adjoint's).  On three nodes s^3 = s, so the next
// function of the sequence is one of the two before: d delta/dt / (2 kappa) =
// (1 - 3q) gamma - 3m delta, q = a_0 + a_2, and no further node function is
// needed: with D = d/dt / (2 kappa) per direction,
//   D_x D_x phi = (Dh - (1 - 3q) r)_x gaa + (2h - 1 + 3 m r)_x daa - r_y dga - r_z dag
//   D_x D_y phi = (h_x + h_y - 1) gga - r_x dga - r_y gda - r_z ggg
// with Dh = ((1 - 2h) mu3 + r (mu4 - 3 s2^2)) / s2.
struct DirH : DirG {
  float k1, k2;   // the coefficients of gaa and daa above
};
__device__ __forceinline__ void dir_hess(float t, const MlsK& K, DirH& o) {
  const float is2 = dir_grad<true>(t, K, o);
  const float m = o.a2 - o.a0, q = o.a0 + o.a2, m2 = m * m;
  const float s2 = q - m2;
  const float mu3 = m * fmaf(-3.f, q, fmaf(2.f, m2, 1.f));
  const float mu4 = fmaf(-3.f * m, mu3, fmaf(-3.f, m2, 1.f) * s2);
  const float dh = fmaf(fmaf(-2.f, o.h, 1.f), mu3, o.r * fmaf(-3.f * s2, s2, mu4)) * is2;
  o.k1 = fmaf(-o.r, fmaf(-3.f, q, 1.f), dh);
  o.k2 = fmaf(3.f * m, o.r, fmaf(2.f, o.h, -1.f));
}

// gradient in cells / (2 kappa) and Hessian in cells / (2 kappa)^2 (xx, yy, zz,
// xy, xz, yz)
template <class Acc>
__device__ __forceinline__ void mls_grad_hess(const float* __restrict__ f, const Acc& A,
                                              const DirH& X, const DirH& Y, const DirH& Z,
                                              float (&gr)[3], float (&hs)[6]) {
  // per z plane the sums over (x, y): aa ac ad ca cc cd da dc (c, d: gamma, delta)
  auto plane = [&](int sz, float (&P)[8]) {
    float a[3], c[3], g[3];
#pragma unroll
    for (int sy = 0; sy < 3; ++sy) {
      float u[3];
      A.load(f, sy, sz, u);
      const float d0 = u[0] - u[1], d2 = u[2] - u[1];
      a[sy] = fmaf(X.a2, d2, fmaf(X.a0, d0, u[1]));
      c[sy] = fmaf(X.c2, d2, X.c0 * d0);
      g[sy] = fmaf(X.g2, d2, X.g0 * d0);
    }
    const float a0 = a[0] - a[1], a2 = a[2] - a[1], c0 = c[0] - c[1], c2 = c[2] - c[1],
                g0 = g[0] - g[1], g2 = g[2] - g[1];
    P[0] = fmaf(Y.a2, a2, fmaf(Y.a0, a0, a[1]));
    P[1] = fmaf(Y.c2, a2, Y.c0 * a0);
    P[2] = fmaf(Y.g2, a2, Y.g0 * a0);
    P[3] = fmaf(Y.a2, c2, fmaf(Y.a0, c0, c[1]));
    P[4] = fmaf(Y.c2, c2, Y.c0 * c0);
    P[5] = fmaf(Y.g2, c2, Y.g0 * c0);
    P[6] = fmaf(Y.a2, g2, fmaf(Y.a0, g0, g[1]));
    P[7] = fmaf(Y.c2, g2, Y.c0 * g0);
  };
  float M[8], sa[8], sc[8], sg[4];   // the middle plane; sums with alpha, gamma, delta in z
  plane(1, M);
#pragma unroll
  for (int q = 0; q < 8; ++q) {
    sa[q] = M[q];
    sc[q] = 0.f;
    if (q < 4) sg[q] = 0.f;
  }
#pragma unroll
  for (int k = 0; k < 2; ++k) {
    float P[8];
    plane(2 * k, P);
    const float za = k ? Z.a2 : Z.a0, zc = k ? Z.c2 : Z.c0, zg = k ? Z.g2 : Z.g0;
#pragma unroll
    for (int q = 0; q < 8; ++q) {
      const float d = P[q] - M[q];
      sa[q] = fmaf(za, d, sa[q]);
      sc[q] = fmaf(zc, d, sc[q]);
      if (q < 4) sg[q] = fmaf(zg, d, sg[q]);
    }
  }
  // names: x, y, z letters
  const float caa = sa[3], aca = sa[1], aac = sc[0], daa = sa[6], ada = sa[2], aad = sg[0];
  const float cca = sa[4], cac = sc[3], acc = sc[1];
  const float dca = sa[7], cda = sa[5], dac = sc[6], cad = sg[3], adc = sc[2], acd = sg[1];
  const float ccc = sc[4];
  gr[0] = fmaf(X.h, caa, -fmaf(X.r, daa, fmaf(Y.r, cca, Z.r * cac)));
  gr[1] = fmaf(Y.h, aca, -fmaf(Y.r, ada, fmaf(X.r, cca, Z.r * acc)));
  gr[2] = fmaf(Z.h, aac, -fmaf(Z.r, aad, fmaf(X.r, cac, Y.r * acc)));
  hs[0] = fmaf(X.k1, caa, fmaf(X.k2, daa, -fmaf(Y.r, dca, Z.r * dac)));
  hs[1] = fmaf(Y.k1, aca, fmaf(Y.k2, ada, -fmaf(X.r, cda, Z.r * adc)));
  hs[2] = fmaf(Z.k1, aac, fmaf(Z.k2, aad, -fmaf(X.r, cad, Y.r * acd)));
  hs[3] = fmaf(X.h + Y.h - 1.f, cca, -fmaf(X.r, dca, fmaf(Y.r, cda, Z.r * ccc)));
  hs[4] = fmaf(X.h + Z.h - 1.f, cac, -fmaf(X.r, dac, fmaf(Z.r, cad, Y.r * ccc)));
  hs[5] = fmaf(Y.h + Z.h - 1.f, acc, -fmaf(Y.r, adc, fmaf(Z.r, acd, X.r * ccc)));
}

// value, and gradient in cells / (2 kappa)
template <class Acc>
__device__ __forceinline__ void mls_val_grad(const float* __restrict__ f, const Acc& A,
                                             const DirG& X, const DirG& Y, const DirG& Z,
                                             float& val, float (&gr)[3]) {
  const PlaneG M = plane_sums(f, A, 1, X, Y);
  float aaa = M.aa, caa = M.ca, aca = M.ac, aac = 0.f, daa = M.ga, ada = M.ag, aad = 0.f,
        cca = M.cc, cac = 0.f, acc = 0.f;
#pragma unroll
  for (int k = 0; k < 2; ++k) {
    const PlaneG P = plane_sums(f, A, 2 * k, X, Y);
    const float za = k ? Z.a2 : Z.a0, zc = k ? Z.c2 : Z.c0, zg = k ? Z.g2 : Z.g0;
    const float d0 = P.aa - M.aa, d1 = P.ca - M.ca, d2 = P.ac - M.ac;
    aaa = fmaf(za, d0, aaa);
    aac = fmaf(zc, d0, aac);
    aad = fmaf(zg, d0, aad);
    caa = fmaf(za, d1, caa);
    cac = fmaf(zc, d1, cac);
    aca = fmaf(za, d2, aca);
    acc = fmaf(zc, d2, acc);
    daa = fmaf(za, P.ga - M.ga, daa);
    ada = fmaf(za, P.ag - M.ag, ada);
    cca = fmaf(za, P.cc - M.cc, cca);
  }
  val = aaa - fmaf(X.r, caa, fmaf(Y.r, aca, Z.r * aac));
  gr[0] = fmaf(X.h, caa, -fmaf(X.r, daa, fmaf(Y.r, cca, Z.r * cac)));
  gr[1] = fmaf(Y.h, aca, -fmaf(Y.r, ada, fmaf(X.r, cca, Z.r * acc)));
  gr[2] = fmaf(Z.h, aac, -fmaf(Z.r, aad, fmaf(X.r, cac, Y.r * acc)));
}

// x >= 0 folded into [0, n)
__device__ __forceinline__ int wrap_pos(int x, int n) {
  if (x >= n) {
    x -= n;
    if (x >= n) x %= n;
  }
  return x;
}

// asynchronous global -> shared copies (cp.async: no register round trip, so
// one thread's copies are all in flight at once)
__device__ __forceinline__ void cp_async16(float* sdst, const float* gsrc) {
  const unsigned d = (unsigned)__cvta_generic_to_shared(sdst);
  asm volatile("cp.async.cg.shared.global [%0], [%1], 16;\n" ::"r"(d), "l"(gsrc) : "memory");
}
__device__ __forceinline__ void cp_async4(float* sdst, const float* gsrc) {
  const unsigned d = (unsigned)__cvta_generic_to_shared(sdst);
  asm volatile("cp.async.ca.shared.global [%0], [%1], 4;\n" ::"r"(d), "l"(gsrc) : "memory");
}
__device__ __forceinline__ void cp_async_commit() { asm volatile("cp.async.commit_group;\n" ::: "memory"); }
template <int N>
__device__ __forceinline__ void cp_async_wait() {
  asm volatile("cp.async.wait_group %0;\n" ::"n"(N) : "memory");
}

// the staged rows of the block, one float4 group (4 consecutive staged nodes
// of one row) per entry: the global offset of the group's first node
struct RowTable {
  const int* gofs;             // global offset of each group's first node
  int nx, vec4;
  // global offset of node j (0..3) of group q (without vector access a group
  // may cross the periodic x boundary: its nodes are wrapped one by one)
  __device__ __forceinline__ size_t node(int q, int j) const {
    const int g = gofs[q];
    if (vec4 || j == 0) return (size_t)g + j;
    const int x = g % nx;
    return (size_t)(g - x) + (x + j < nx ? x + j : x + j - nx);
  }
};

// issue the copies of one field component's staged rows into dst
template <int MT>
__device__ __forceinline__ void stage_async(float* dst, const float* __restrict__ src,
                                            const RowTable& R, int ngroups) {
#pragma unroll 1
  for (int q = threadIdx.x; q < ngroups; q += MT) {
    if (R.vec4) {
      cp_async16(dst + 4 * q, src + R.gofs[q]);   // x multiple of 4 and nx % 4 == 0
    } else {
#pragma unroll
      for (int j = 0; j < 4; ++j) cp_async4(dst + 4 * q + j, src + R.node(q, j));
    }
  }
}

// addressing factories: staged rows (a table at the start of the shared memory
// with, per (y, z) row, the byte offset of its staged start - 4 x its first x)
// or the global field
struct StagedRows {
  const unsigned char* sm;
  int r0, sy;        // -(ylo + sy zlo): first row relative to the body's cell; rows per z plane
  __device__ __forceinline__ RowAcc at(const int (&c)[3], int buf) const {
    return RowAcc{sm, r0 + (c[1] - 1) + sy * (c[2] - 1), sy, buf + 4 * (c[0] - 1)};
  }
};
struct GlobalRows {
  Grid g;
  int G[3];
  __device__ __forceinline__ GlobalAcc at(const int (&c)[3]) const {
    GlobalAcc A;
    A.init(c, G, g);
    return A;
  }
};

// nearest node and node functions of one component at a probe point
struct ProbeW {
  int cc[3];
  DirG X, Y, Z;
  __device__ __forceinline__ void prepare(const float (&t)[3], int comp, const MlsK& K) {
    float t3[3];
    locate(t, comp, cc, t3);
    dir_grad(t3[0], K, X);
    dir_grad(t3[1], K, Y);
    dir_grad(t3[2], K, Z);
  }
};

// spread coef * phi onto the 27 nodes of a full field
__device__ __forceinline__ void mls_spread(float* f, const GlobalAcc& A, const DirW& X,
                                           const DirW& Y, const DirW& Z, float coef) {
  const float xa[3] = {X.a0, X.a1, X.a2}, xb[3] = {X.b0, -(X.b0 + X.b2), X.b2};
  const float ya[3] = {Y.a0, Y.a1, Y.a2}, yb[3] = {Y.b0, -(Y.b0 + Y.b2), Y.b2};
  const float za[3] = {Z.a0, Z.a1, Z.a2}, zb[3] = {Z.b0, -(Z.b0 + Z.b2), Z.b2};
#pragma unroll
  for (int sz = 0; sz < 3; ++sz) {
#pragma unroll
    for (int sy = 0; sy < 3; ++sy) {
      float* r = f + A.row(sy, sz);
      const float t0 = ya[sy] * za[sz] * coef, t1 = fmaf(yb[sy], za[sz], ya[sy] * zb[sz]) * coef;
#pragma unroll
      for (int sx = 0; sx < 3; ++sx)
        atomicAdd(r + A.ix[sx], fmaf(xa[sx], t0 - t1, -xb[sx] * t0));
    }
  }
}

// Spread in exact fixed point, one 32-bit word per node: the contribution
// coef*phi, already scaled by the block's power of two so that all a node can
// take stays below 2^31, rounded to an integer and added with a native shared
// atomic; the sum is independent of the order of the additions.
__device__ __forceinline__ void mls_spread_fixed(unsigned char* sm, const RowAcc& A, const DirW& X,
                                                 const DirW& Y, const DirW& Z, float coef) {
  const float xb1 = -(X.b0 + X.b2);
  const float ya[3] = {Y.a0, Y.a1, Y.a2}, yb[3] = {Y.b0, -(Y.b0 + Y.b2), Y.b2};
  const float za[3] = {Z.a0 * coef, Z.a1 * coef, Z.a2 * coef};
  const float zb[3] = {Z.b0 * coef, -(Z.b0 + Z.b2) * coef, Z.b2 * coef};
#pragma unroll
  for (int sz = 0; sz < 3; ++sz) {
#pragma unroll
    for (int sy = 0; sy < 3; ++sy) {
      int* r = reinterpret_cast<int*>(sm + A.row(sy, sz));
      const float t0 = ya[sy] * za[sz], t1 = fmaf(yb[sy], za[sz], ya[sy] * zb[sz]);
      const float t = t0 - t1;
      atomicAdd(r, __float2int_rn(fmaf(X.a0, t, -X.b0 * t0)));
      atomicAdd(r + 1, __float2int_rn(fmaf(X.a1, t, -xb1 * t0)));
      atomicAdd(r + 2, __float2int_rn(fmaf(X.a2, t, -X.b2 * t0)));
    }
  }
}

// x (|x| < 2^62) rounded to a 64-bit integer without a 64-bit conversion:
// hi = floor(x / 2^32) is exact and the remainder x - 2^32 hi lies in [0, 2^32)
__device__ __forceinline__ long long to_fixed(float x) {
  const float hf = floorf(x * 0x1p-32f);
  const unsigned lo = __float2uint_rn(fmaf(-hf, 0x1p32f, x));
  return (long long)(int)hf * 4294967296ll + (long long)lo;
}

// 2^k as a float, k in [-126, 127]
__device__ __forceinline__ float pow2f(int k) { return __int_as_float((k + 127) << 23); }

}  // namespace
}  // namespace ibm
