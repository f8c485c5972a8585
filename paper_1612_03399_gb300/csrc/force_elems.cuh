// Element forces of the interaction potentials (Sec. 2.3, Eqs.
// elaspot..areapot): the forces themselves (*_forward: the force kernel) and their derivatives along the tangents y the positions carry
// (*_tangent: the adjoint).  The derivative is the
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

// k u + l v
__device__ __forceinline__ Vec<float> vmad(float k, const Vec<float>& u, float l,
                                           const Vec<float>& v) {
  return {fmaf(k, u.x, l * v.x), fmaf(k, u.y, l * v.y), fmaf(k, u.z, l * v.z)};
}

// Values only.  An edge with its hinge: e = pb - pa, ac and ad from a to the
// wings, N1 = e x ac and N2 = bd x e the normals of its left face (a, b, c) and
// right face (b, a, d), r1 and r2 their inverse lengths.  Energies are formed only
// where they are used.  (With sin theta = -|e| (ad.N1)/(|N1||N2|), N2 = ad x e and F_a
// from the sum of the four the bending forces of strongly folded sheets were 5 %
// further from float64; with products of unit normals those of drops 15 %.)
__device__ __forceinline__ void spring_forward(const Vec<float>& e, float l0, float ks, float& l,
                                               float& inv_l, Vec<float>& fa, float& e_spring) {
  const float l2 = vdot(e, e);
  inv_l = rsqrtf(l2);
  l = l2 * inv_l;
  const float dl = l - l0;
  fa = vscale(e, ks * dl * inv_l);
  e_spring = 0.5f * ks * dl * dl;
}
__device__ __forceinline__ void hinge_forward(const Vec<float>& e, float l, float inv_l,
                                              const Vec<float>& ac, const Vec<float>& ad,
                                              const Vec<float>& N1, const Vec<float>& N2, float r1,
                                              float r2, float cos0, float sin0, float kb,
                                              Vec<float>& fa, Vec<float>& fb, Vec<float>& fc,
                                              Vec<float>& fd, float& e_bend) {
  const float r12 = r1 * r2;
  const float cth = vdot(N1, N2) * r12, sth = vdot(vscale(vcross(N1, N2), r12), e) * inv_l;
  const float s = kb * l * (sth * cos0 - cth * sin0);   // k_b |e| sin(theta - theta0)
  fc = vscale(N1, s * r1 * r1);
  fd = vscale(N2, s * r2 * r2);
  const float inv_l2 = inv_l * inv_l;
  const float sc = vdot(ac, e) * inv_l2, sd = vdot(ad, e) * inv_l2;
  fa = vsub(fa, vmad(1.f - sc, fc, 1.f - sd, fd));
  fb = vsub(fb, vmad(sc, fc, sd, fd));
  e_bend = kb * (1.f - (cth * cos0 + sth * sin0));
}

// Local area, global area and volume forces of the face on one side of an edge:
// N its normal, rn = 1/|N|, w the vector from a to its third vertex, side = 1
// (left face) or -1 (right face, which runs from b to a).  fa, fb, fw are added
// to.  The area part is m x (w - e), -m x w and m x e with m = -side (c_A + k_a
// strain) n / 2.  The volume part gives every corner a third of the face's
// normal, -c_V N / 6: grad_a V = b x c / 6 differs from N / 6 by a x (c - b) / 6,
// whose sum over the closed fan of faces around a vertex is zero (c_V is zero on
// open sheets), and N carries no products of the body-frame coordinates.  t: a
// load every corner gets besides.
__device__ __forceinline__ void face_forward(const Vec<float>& e, const Vec<float>& w,
                                             const Vec<float>& N, float rn, float side, float A0f,
                                             float ka, float cA, float cV, const Vec<float>& t,
                                             Vec<float>& fa, Vec<float>& fb, Vec<float>& fw,
                                             float& e_area) {
  const float da = 0.5f * vdot(N, N) * rn - A0f;
  const float k = -0.5f * side * rn * (cA + ka * (da / A0f)), kv = cV * (-1.f / 6.f);
  const Vec<float> m = vscale(N, k);
  const Vec<float> X = vcross(m, w), Y = vcross(m, e);
  const Vec<float> v = {fmaf(kv, N.x, t.x), fmaf(kv, N.y, t.y), fmaf(kv, N.z, t.z)};
  fa = vadd(fa, vadd(vsub(X, Y), v));
  fb = vadd(fb, vsub(v, X));
  fw = vadd(fw, vadd(Y, v));
  e_area = 0.5f * ka * da * da / A0f;
}

// Derivatives (suffix d) of the same along the tangents: e, ac, ad, w with their
// tangents ed, acd, add, wd (differences of the vertices').  fa..fd receive the
// derivatives of the forces.  uk_s, uk_b and uk_a receive y . dF/dk_s, y . dF/dk_b
// and y . dF/dk_a, the forces per unit constant against the same tangents, which
// are the force cotangents: sums of products already at hand.
__device__ __forceinline__ void spring_tangent(const Vec<float>& e, const Vec<float>& ed, float l0,
                                               float ks, float& l, float& ld, float& il, float& ild,
                                               Vec<float>& fa, float& uk_s) {
  const float l2 = vdot(e, e), eed = vdot(e, ed);
  il = rsqrtf(l2);
  l = l2 * il;
  ld = eed * il;
  ild = -il * il * ld;                                   // (1/l)' = -l'/l^2
  const float st = (l - l0) * il, std_ = ld * il + (l - l0) * ild;
  fa = vmad(ks * std_, e, ks * st, ed);
  uk_s = -st * eed;
}
// N1d, N2d: the normals' tangents; h1, h2: |N|'/|N|
__device__ __forceinline__ void hinge_tangent(
    const Vec<float>& e, const Vec<float>& ed, float l, float ld, float il, float ild,
    const Vec<float>& ac, const Vec<float>& acd, const Vec<float>& ad, const Vec<float>& add,
    const Vec<float>& N1, const Vec<float>& N1d, const Vec<float>& N2, const Vec<float>& N2d,
    float r1, float r2, float h1, float h2, float cos0, float sin0, float kb, Vec<float>& fa,
    Vec<float>& fb, Vec<float>& fc, Vec<float>& fd, float& uk_b) {
  const float R1 = r1 * r1, R2 = r2 * r2, r12 = r1 * r2;
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
  const float il2 = il * il, il2d = 2.f * il * ild;
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
// h = |N|'/|N|; cA, cV and their derivatives cAd, cVd
__device__ __forceinline__ void face_tangent(const Vec<float>& e, const Vec<float>& ed,
                                             const Vec<float>& w, const Vec<float>& wd,
                                             const Vec<float>& N, const Vec<float>& Nd, float rn,
                                             float h, float side, float A0f, float ka, float cA,
                                             float cAd, float cV, float cVd, Vec<float>& fa,
                                             Vec<float>& fb, Vec<float>& fw, float& uk_a) {
  const float Af = 0.5f * vdot(N, N) * rn, Afd = Af * h;
  const float iA = 1.f / A0f, strain = (Af - A0f) * iA;
  const float gA = cA + ka * strain, gAd = cAd + ka * Afd * iA;
  const float k0 = -0.5f * side * rn;
  const float k = k0 * gA, kd = k0 * (gAd - h * gA);     // (1/|N|)' = -h/|N|
  const Vec<float> m = vscale(N, k), md = vmad(kd, N, k, Nd);
  const Vec<float> v = vmad(cVd * (-1.f / 6.f), N, cV * (-1.f / 6.f), Nd);
  const Vec<float> X = vadd(vcross(md, w), vcross(m, wd));
  const Vec<float> Y = vadd(vcross(md, e), vcross(m, ed));
  fa = vadd(fa, vadd(vsub(X, Y), v));
  fb = vadd(fb, vsub(v, X));
  fw = vadd(fw, vadd(Y, v));
  uk_a = -strain * Afd;
}

}  // namespace ibm
