// Element forces of the interaction potentials (Sec. 2.3, Eqs.
// elaspot..areapot): the forces themselves (edge_forward, face_forward: the
// force kernel) and their derivatives along the tangents y the positions carry
// (edge_tangent, face_tangent: the adjoint).  The derivative is the
// Jacobian-vector product J y; J = -Hessian of the energy is symmetric, so the
// same product is the vector-Jacobian product the adjoint needs.
// Edge e = (a, b) with wings c (face (a, b, c)) and d (face (b, a, d)):
//   spring   W = k_s/2 (l - l0)^2      F_a = k_s (l - l0) e/l, F_b = -F_a
//   bending  W = k_b (1 - cos(theta - theta0)),  F = -k_b sin(theta - theta0) grad theta,
//            cos theta = n1.n2, sin theta = (n1 x n2).e/|e|, and with
//            N1 = e x (c - a), N2 = (d - b) x e, s_c = (c - a).e/|e|^2, s_d likewise,
//            grad_c theta = -|e| N1/|N1|^2, grad_d theta = -|e| N2/|N2|^2,
//            grad_a theta = -(1 - s_c) grad_c - (1 - s_d) grad_d,
//            grad_b theta = -s_c grad_c - s_d grad_d
//            (the unique gradient that is invariant under translations and
//            rotations and moves the wings about the hinge).
// Face (a, b, c), A_f = |N|/2, n = N/|N|:
//   grad_a A_f = n x (c - b)/2 (cyclic), grad_a V = b x c / 6 (cyclic, body frame),
//   F = -(k_A (A - A0)/A0 + k_a (A_f - A0_f)/A0_f) grad A_f - k_v (V - V0)/V0 grad V.
#pragma once

#include <cuda_runtime.h>

namespace ibm {

template <class T>
struct Vec {
  T x, y, z;
};
template <class T>
__device__ __forceinline__ Vec<T> vsub(const Vec<T>& a, const Vec<T>& b) {
  return {a.x - b.x, a.y - b.y, a.z - b.z};
}
template <class T>
__device__ __forceinline__ Vec<T> vadd(const Vec<T>& a, const Vec<T>& b) {
  return {a.x + b.x, a.y + b.y, a.z + b.z};
}
template <class T>
__device__ __forceinline__ Vec<T> vcross(const Vec<T>& a, const Vec<T>& b) {
  return {a.y * b.z - a.z * b.y, a.z * b.x - a.x * b.z, a.x * b.y - a.y * b.x};
}
template <class T>
__device__ __forceinline__ T vdot(const Vec<T>& a, const Vec<T>& b) {
  return a.x * b.x + a.y * b.y + a.z * b.z;
}
template <class T>
__device__ __forceinline__ Vec<T> vscale(const Vec<T>& a, T s) {
  return {a.x * s, a.y * s, a.z * s};
}

// Spring and bending of one edge, values only.  With N1 = e x ac, N2 = ad x e:
// (n1 x n2).e/|e| = -|e| (ad.N1)/(|N1||N2|), the force on b is what makes the
// four sum to zero, and energies are formed only where they are used.
__device__ __forceinline__ void edge_forward(const Vec<float>& pa, const Vec<float>& pb,
                                             const Vec<float>& pc, const Vec<float>& pd,
                                             bool has_hinge, float l0, float cos0, float sin0,
                                             float ks, float kb, Vec<float>& fa, Vec<float>& fb,
                                             Vec<float>& fc, Vec<float>& fd, float& e_spring,
                                             float& e_bend) {
  const Vec<float> e = vsub(pb, pa);
  const float l2 = vdot(e, e);
  const float inv_l = rsqrtf(l2);
  const float l = l2 * inv_l, dl = l - l0;
  fa = vscale(e, ks * dl * inv_l);
  fb = {-fa.x, -fa.y, -fa.z};
  fc = fd = {0.f, 0.f, 0.f};
  e_spring = 0.5f * ks * dl * dl;
  e_bend = 0.f;
  if (!has_hinge) return;
  const Vec<float> ac = vsub(pc, pa), ad = vsub(pd, pa);
  const Vec<float> N1 = vcross(e, ac), N2 = vcross(ad, e);
  const float r1 = rsqrtf(vdot(N1, N1)), r2 = rsqrtf(vdot(N2, N2));
  const float r12 = r1 * r2;
  const float cth = vdot(N1, N2) * r12, sth = -l * vdot(ad, N1) * r12;
  const float s = kb * l * (sth * cos0 - cth * sin0);   // k_b |e| sin(theta - theta0)
  fc = vscale(N1, s * r1 * r1);
  fd = vscale(N2, s * r2 * r2);
  const float inv_l2 = inv_l * inv_l;
  const float sc = vdot(ac, e) * inv_l2, sd = vdot(ad, e) * inv_l2;
  const Vec<float> g = {sc * fc.x + sd * fd.x, sc * fc.y + sd * fd.y, sc * fc.z + sd * fd.z};
  fa = {fa.x + (g.x - (fc.x + fd.x)), fa.y + (g.y - (fc.y + fd.y)), fa.z + (g.z - (fc.z + fd.z))};
  fb = vsub(fb, g);
  e_bend = kb * (1.f - (cth * cos0 + sth * sin0));
}

// Local area, global area and volume forces of one face, values only.  The
// area part is (m x (c - b), m x (a - c), minus their sum) with
// m = -(c_A + k_a strain) n / 2.  The volume part gives every corner a third of
// the face's normal, -c_V N / 6: grad_a V = b x c / 6 differs from N / 6 by
// a x (c - b) / 6, whose sum over the closed fan of faces around a vertex is
// zero (c_V is zero on open sheets), and N carries no products of the
// body-frame coordinates.
__device__ __forceinline__ void face_forward(const Vec<float>& pa, const Vec<float>& pb,
                                             const Vec<float>& pc, float A0f, float ka, float cA,
                                             float cV, Vec<float> (&f)[3], float& e_area) {
  const Vec<float> ab = vsub(pb, pa), ac = vsub(pc, pa), bc = vsub(ac, ab);
  const Vec<float> N = vcross(ab, ac);
  const float q = vdot(N, N);
  const float rn = rsqrtf(q);
  const float da = 0.5f * q * rn - A0f;
  const Vec<float> m = vscale(N, -0.5f * rn * (cA + ka * __fdividef(da, A0f)));
  const Vec<float> v = vscale(N, cV * (-1.f / 6.f));
  const Vec<float> fa = vcross(m, bc), fb = vcross(ac, m);   // m x (a - c) = ac x m
  f[0] = vadd(fa, v);
  f[1] = vadd(fb, v);
  f[2] = {v.x - (fa.x + fb.x), v.y - (fa.y + fb.y), v.z - (fa.z + fb.z)};
  e_area = 0.5f * ka * da * da / A0f;
}

// k u + l v
__device__ __forceinline__ Vec<float> vmad(float k, const Vec<float>& u, float l,
                                           const Vec<float>& v) {
  return {fmaf(k, u.x, l * v.x), fmaf(k, u.y, l * v.y), fmaf(k, u.z, l * v.z)};
}

// Derivatives (suffix d) of an edge's forces along the tangents: e, ac, ad with
// their tangents ed, acd, add (differences of the vertices').  fa..fd receive
// the derivatives of the forces on a, b, c, d.  uk_s and uk_b receive y . dF/dk_s
// and y . dF/dk_b, the forces per unit constant against the same tangents, which
// are the force cotangents: sums of products already at hand.
__device__ __forceinline__ void edge_tangent(const Vec<float>& e, const Vec<float>& ed,
                                             const Vec<float>& ac, const Vec<float>& acd,
                                             const Vec<float>& ad, const Vec<float>& add,
                                             bool has_hinge, float l0, float cos0, float sin0,
                                             float ks, float kb, Vec<float>& fa, Vec<float>& fb,
                                             Vec<float>& fc, Vec<float>& fd, float& uk_s,
                                             float& uk_b) {
  const float l2 = vdot(e, e), eed = vdot(e, ed);
  const float il = rsqrtf(l2), l = l2 * il, ld = eed * il;
  const float il2 = il * il, ild = -il2 * ld;            // (1/l)' = -l'/l^2
  const float st = (l - l0) * il, std_ = ld * il + (l - l0) * ild;
  fa = vmad(ks * std_, e, ks * st, ed);
  fb = {-fa.x, -fa.y, -fa.z};
  fc = fd = {0.f, 0.f, 0.f};
  uk_s = -st * eed;
  uk_b = 0.f;
  if (!has_hinge) return;
  const Vec<float> N1 = vcross(e, ac), N2 = vcross(ad, e);
  const Vec<float> N1d = vadd(vcross(ed, ac), vcross(e, acd));
  const Vec<float> N2d = vadd(vcross(add, e), vcross(ad, ed));
  const float r1 = rsqrtf(vdot(N1, N1)), r2 = rsqrtf(vdot(N2, N2));
  const float R1 = r1 * r1, R2 = r2 * r2, r12 = r1 * r2;
  const float h1 = R1 * vdot(N1, N1d), h2 = R2 * vdot(N2, N2d);   // |N|'/|N|
  const float r12d = -r12 * (h1 + h2);
  const float D = vdot(N1, N2), Dd = vdot(N1d, N2) + vdot(N1, N2d);
  const float t = vdot(ad, N1), td = vdot(add, N1) + vdot(ad, N1d);
  const float cth = D * r12, cthd = Dd * r12 + D * r12d;
  const float sth = -l * t * r12, sthd = -(ld * t * r12 + l * (td * r12 + t * r12d));
  const float sn = sth * cos0 - cth * sin0, snd = sthd * cos0 - cthd * sin0;
  const float s = l * sn, sd_ = ld * sn + l * snd;
  const float a1 = s * R1, a1d = sd_ * R1 - 2.f * a1 * h1;
  const float a2 = s * R2, a2d = sd_ * R2 - 2.f * a2 * h2;
  const Vec<float> uc = vscale(N1, a1), ucd = vmad(a1d, N1, a1, N1d);   // per unit k_b
  const Vec<float> ud = vscale(N2, a2), udd = vmad(a2d, N2, a2, N2d);
  const float il2d = 2.f * il * ild;
  const float pc = vdot(ac, e), pd = vdot(ad, e);
  const float sc = pc * il2, scd = (vdot(acd, e) + vdot(ac, ed)) * il2 + pc * il2d;
  const float sd = pd * il2, sdd = (vdot(add, e) + vdot(ad, ed)) * il2 + pd * il2d;
  const Vec<float> g = vmad(sc, uc, sd, ud);
  const Vec<float> gd = vadd(vmad(scd, uc, sc, ucd), vmad(sdd, ud, sd, udd));
  fa = vadd(fa, vscale(vsub(gd, vadd(ucd, udd)), kb));
  fb = vsub(fb, vscale(gd, kb));
  fc = vscale(ucd, kb);
  fd = vscale(udd, kb);
  uk_b = vdot(uc, acd) + vdot(ud, add) - vdot(g, ed);
}

// The same for a face: ab, ac with their tangents; cA, cV and their derivatives
// cAd, cVd; uk_a receives y . dF/dk_a = -strain A'.
__device__ __forceinline__ void face_tangent(const Vec<float>& ab, const Vec<float>& abd,
                                             const Vec<float>& ac, const Vec<float>& acd,
                                             float A0f, float ka, float cA, float cAd, float cV,
                                             float cVd, Vec<float> (&f)[3], float& uk_a) {
  const Vec<float> bc = vsub(ac, ab), bcd = vsub(acd, abd);
  const Vec<float> N = vcross(ab, ac), Nd = vadd(vcross(abd, ac), vcross(ab, acd));
  const float q = vdot(N, N);
  const float rn = rsqrtf(q);
  const float Afd = 0.5f * vdot(N, Nd) * rn;
  const float strain = __fdividef(0.5f * q * rn - A0f, A0f);
  const float gA = cA + ka * strain, gAd = cAd + __fdividef(ka * Afd, A0f);
  const float rnd = -2.f * rn * rn * Afd;                  // (1/|N|)' = -|N|'/|N|^2
  const float k = -0.5f * rn * gA, kd = -0.5f * fmaf(rnd, gA, rn * gAd);
  const Vec<float> m = vscale(N, k), md = vmad(kd, N, k, Nd);
  const Vec<float> v = vmad(cVd * (-1.f / 6.f), N, cV * (-1.f / 6.f), Nd);
  const Vec<float> fa = vadd(vcross(md, bc), vcross(m, bcd));
  const Vec<float> fb = vadd(vcross(acd, m), vcross(ac, md));
  f[0] = vadd(fa, v);
  f[1] = vadd(fb, v);
  f[2] = vsub(v, vadd(fa, fb));
  uk_a = -strain * Afd;
}

}  // namespace ibm
