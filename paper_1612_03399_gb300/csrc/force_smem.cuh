// Shared-memory layout of a force patch's vertices and contribution slots (the
// force kernel and its adjoint).
#pragma once

#include "force_elems.cuh"
#include "ibm_internal.cuh"

namespace ibm {
namespace {

// Positions and contribution slots in shared memory: as float4 (WIDE, one
// shared load or store each), or as three arrays, a quarter smaller, for
// patches whose float4 form would cost a resident block.
template <bool WIDE>
struct Smem;
template <>
struct Smem<true> {
  float4 *p, *c;
  __device__ __forceinline__ void init(float* s, int n_loc, int) {
    p = reinterpret_cast<float4*>(s);
    c = p + n_loc;
  }
  __device__ __forceinline__ void set(int i, float x, float y, float z) const {
    p[i] = make_float4(x, y, z, 0.f);
  }
  __device__ __forceinline__ Vec<float> pos(int i) const {
    const float4 t = p[i];
    return {t.x, t.y, t.z};
  }
  __device__ __forceinline__ Vec<float> slot(int s) const {
    const float4 t = c[s];
    return {t.x, t.y, t.z};
  }
  __device__ __forceinline__ void put(int s, const Vec<float>& f) const {
    if (s != kNone) c[s] = make_float4(f.x, f.y, f.z, 0.f);
  }
};
template <>
struct Smem<false> {
  float *p, *c;
  int np, nc;
  __device__ __forceinline__ void init(float* s, int n_loc, int n_slot) {
    p = s;
    np = n_loc;
    c = s + 3 * n_loc;
    nc = n_slot;
  }
  __device__ __forceinline__ void set(int i, float x, float y, float z) const {
    p[i] = x;
    p[np + i] = y;
    p[2 * np + i] = z;
  }
  __device__ __forceinline__ Vec<float> pos(int i) const { return {p[i], p[np + i], p[2 * np + i]}; }
  __device__ __forceinline__ Vec<float> slot(int s) const { return {c[s], c[nc + s], c[2 * nc + s]}; }
  __device__ __forceinline__ void put(int s, const Vec<float>& f) const {
    if (s == kNone) return;
    c[s] = f.x;
    c[nc + s] = f.y;
    c[2 * nc + s] = f.z;
  }
};

// Sum of own vertex i's slots [s0, s1) in a fixed order.  A vertex of a regular
// mesh has 12 slots, so eight neighbours reading their first, second, ... slots
// together would meet two of the eight 16-byte banks; each starts elsewhere in
// its run instead.
template <class S>
__device__ __forceinline__ Vec<float> slot_sum(const S& sm, int i, int s0, int s1) {
  Vec<float> f = {0.f, 0.f, 0.f};
  int s = s0 + (i & 7);
  if (s >= s1) s = s0;
  for (int k = s0; k < s1; ++k) {
    f = vadd(f, sm.slot(s));
    if (++s == s1) s = s0;
  }
  return f;
}

}  // namespace
}  // namespace ibm
