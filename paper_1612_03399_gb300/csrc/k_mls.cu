// Marker kernel: face geometry, per-body area/volume reductions, MLS
// interpolation at the centroid, direct-forcing marker force, probe gradient
// and traction, and spreading (Sec. 2.2, Eqs. mls..mls_cl; Sec. 5 steps 1-3).
//
// One block = one surface patch of ONE body (up to 128 or 256 faces, built by
// recursive coordinate bisection of the rest mesh), one thread per face.
// The block builds a ROW MAP of its grid footprint: for every (y, z) row of
// the nodes its 3x3x3 supports (centroids and probe ends) touch, the x-range
// touched in whole groups of 4 nodes (float4-aligned when the grid allows),
// found with one shared bit mask per row.  The velocity components are staged
// in shared memory one after the other with asynchronous copies, differentiated
// and interpolated from there, and each component's marker forces are spread as
// soon as they are known, in place of the staged component: exact fixed point
// (32-bit shared atomics, a power-of-two scale per block and component),
// flushed with float4 global atomics.  The rows that received a nonzero spread
// are recorded so the next step's clear zeroes exactly those.  A patch whose
// footprint does not fit takes the direct global path (scalar loads and float
// atomics) and records its bounding box.
//
// What bounds it: instruction issue and the shared-memory pipe (162 loads and
// 81 atomics per face at about three conflicting words each), at the number
// of warps that registers and shared memory allow; not HBM (20 % busy).
// Hence the closed form in central moments (mls_closed_form.cuh; 20 % fewer
// instructions), the spread right after the interpolation (its factors are
// computed once), and 24 warps per SM: 80 registers, for which the probe
// kernels keep what a component needs once or twice per thread in shared
// memory.  Kept in local memory instead it cost more than the 24 warps gave:
// next to 220 KB of shared memory little L1 is left for it.  Measured, this
// kernel alone (us; before: 128 registers, 16 warps, spread after all three
// components): whole step 437 -> 354 (319 with what followed: the variants, buffers
// by block) for 1000 drops (1.28 M faces) on 512^3, 151 -> 117 (111) for 460 k faces of
// uneven bodies, 147 -> 114 (112) for a membrane of 377 k faces; interpolation and
// spread 232 -> 170 and probes with body sums 233 -> 162 for the 1000 drops on 256^3.
#include <cuda_runtime.h>
#include <limits.h>
#include <math.h>

#include "bulk_copy.cuh"
#include "ibm_internal.cuh"
#include "mls_closed_form.cuh"

namespace ibm {
namespace {

// The global-memory path of a marker block whose footprint does not fit its
// shared memory (rare): out of line, so that it does not crowd the
// instruction cache of the staged path it sits beside.  All loads of a support are
// issued before the first is used (a step of 200 drops of 14 cells, 140 of 1000
// patches on this path: 274 -> 264 us).
// (body cell G: read again here, so that it is not kept for this path; FEW: a
// copy with the registers of the kernel's variant for few blocks)
__device__ __forceinline__ GlobalRows global_rows(const Grid& g, const BodyDev* b) {
  return GlobalRows{g, {b->G[0], b->G[1], b->G[2]}};
}
// the 27 nodes of a support, all loads in flight
struct Loaded {
  float v[3][3][3];
  __device__ __forceinline__ Loaded(const float* __restrict__ f, const GlobalAcc& A) {
#pragma unroll
    for (int sz = 0; sz < 3; ++sz)
#pragma unroll
      for (int sy = 0; sy < 3; ++sy) A.load(f, sy, sz, v[sz][sy]);
  }
  __device__ __forceinline__ void load(const float*, int sy, int sz, float (&u)[3]) const {
#pragma unroll
    for (int s = 0; s < 3; ++s) u[s] = v[sz][sy][s];
  }
};
template <bool FEW>
__device__ __noinline__ float value_global(const float* f, Grid g, const BodyDev* b, int c0, int c1,
                                          int c2, DirW X, DirW Y, DirW Z) {
  const int c[3] = {c0, c1, c2};
  return mls_value(f, Loaded(f, global_rows(g, b).at(c)), X, Y, Z);
}
template <bool FEW>
__device__ __noinline__ float3 gradient_global(const float* f, Grid g, const BodyDev* b, ProbeW P) {
  float gr[3];
  mls_grad(f, Loaded(f, global_rows(g, b).at(P.cc)), P.X, P.Y, P.Z, gr);
  return make_float3(gr[0], gr[1], gr[2]);
}
template <bool FEW>
__device__ __noinline__ void spread_global(float* f, Grid g, const BodyDev* b, int c0, int c1,
                                           int c2, DirW X, DirW Y, DirW Z, float coef) {
  const int c[3] = {c0, c1, c2};
  mls_spread(f, global_rows(g, b).at(c), X, Y, Z, coef);
}

// sum over the warp of 64-bit integers, as three 32-bit reductions (24, 24
// and 16 bits: 32 addends cannot overflow the unsigned words)
__device__ __forceinline__ long long warp_sum_i64(long long q) {
  const unsigned lo = __reduce_add_sync(0xffffffffu, (unsigned)q & 0xffffffu);
  const unsigned mid = __reduce_add_sync(0xffffffffu, (unsigned)(q >> 24) & 0xffffffu);
  const int hi = __reduce_add_sync(0xffffffffu, (int)(q >> 48));
  return (long long)lo + ((long long)mid << 24) + ((long long)hi << 48);
}

// REC (record mode): instead of spreading, write each marker's spread record
// (centroid in cells, c_l F) and count it under the tiles of the tile-owned
// spread, with the tile's largest |c_l F| per component.  PLAIN: all bodies
// closed and no pressure, so one probe and three components; without the code
// for the second probe and the pressure the step's kernel needs no spills at
// 80 registers (354 -> 339 us for the 1000 drops, 117 -> 111 us for the uneven
// bodies).
// FEW: 128 registers, 16 warps per SM, for launches that cannot use more: at most
// two blocks of 256 faces per SM in all, or a shape of one or two blocks.  23 drops
// with pressure (115 blocks): 26.4 -> 21.3 us; three large drops (15 blocks, every
// footprint past its shape, all loads of a support in flight): a step 157 -> 139 us.
// With more blocks the 24 warps are worth more: 500 drops 152 us against 177.
enum MarkerVariant { kAll, kPlain, kFew };
template <int MT, bool MEASURE, bool INTERP, bool PROBE, bool SPREAD, bool REC, int VAR>
__global__ void __launch_bounds__(MT, (VAR == kFew ? 512 : 768) / MT) marker_kernel(
    DeviceTables T, Grid g, StepConsts sc, int32_t V, int32_t F, const float* __restrict__ x,
    const float* __restrict__ v, const float* __restrict__ u, const float* __restrict__ vv,
    const float* __restrict__ w, const float* __restrict__ pr, const float* __restrict__ accel,
    float* __restrict__ U, float* __restrict__ Fm, const float* __restrict__ Fm_in,
    float* __restrict__ Fext, float* __restrict__ fx, float* __restrict__ fy,
    float* __restrict__ fz, int record, int vec4, TileDev td, float phi_bound_all,
    int cache, int* __restrict__ cache_tab, float4* __restrict__ cache_face, MarkerShape shape) {
  constexpr bool PLAIN = VAR == kPlain, FEW = VAR == kFew;
  constexpr bool FIELD = INTERP || PROBE || SPREAD;
  // the coupled forcing launch (interpolation and spread at the centroids)
  // may save its face geometry and row tables (cache 1) and, in the later
  // substeps of the same step, load them instead of recomputing (cache 2)
  constexpr bool CACHEABLE = !MEASURE && INTERP && !PROBE && SPREAD && !REC;
  const bool load = CACHEABLE && cache == 2;
  const bool save = CACHEABLE && cache == 1;
  constexpr bool VEL = INTERP || PROBE;
  constexpr bool FLUSH = SPREAD && !REC;      // spreads into the fields
  constexpr bool ROWMAP = VEL || FLUSH;
  extern __shared__ __align__(16) unsigned char dyn[];
  const int MR = shape.rows, mn = shape.nodes;  // (y, z) rows, staged nodes
  int* s_off4 = reinterpret_cast<int*>(dyn);   // [MR] 4 (staged start of the row - its first x)
  unsigned short* s_grp = reinterpret_cast<unsigned short*>(s_off4 + MR);   // [MR + 1] first group
  unsigned* s_mask = reinterpret_cast<unsigned*>(s_grp + MR + 8);    // a bit per group: nonzero
  int* s_gofs = reinterpret_cast<int*>(s_mask + marker_mask_words(mn));   // [mn/4] global offsets
  float* bufA = reinterpret_cast<float*>(s_gofs + mn / 4);
  // probe kernels keep per-thread values that a component needs once or twice
  // here, not in registers: probe end(s), normal, centroid velocity, a.n
  float* s_own = bufA + mn + threadIdx.x;      // [kOwn][MT]
  unsigned* s_xbits = reinterpret_cast<unsigned*>(bufA);   // [MR] x-intervals each row touches,
                                                           //  while the rows are found
  __shared__ int s_lo[3], s_hi[3];
  __shared__ int s_N;
  __shared__ int s_warp[MT / 32];
  // bound on a node's contributions: per component the largest |c_l F|, or (FEW) per
  // warp the sum of |c_l F| / 256
  __shared__ unsigned s_bmax[3];
  __shared__ float s_bsum[3][FEW ? MT / 32 : 1];
  __shared__ __align__(8) unsigned long long s_bar;
  __shared__ unsigned long long s_q[2][MT / 32];   // per-warp fixed-point body sums
  // what the end of the block needs again: body, its cell G, closed, patch
  // record, faces
  __shared__ int s_hdr[8];

  // a force kernel launched after this one may start once every block of
  // this grid runs (it waits for this grid's results before using them)
  asm volatile("griddepcontrol.launch_dependents;");
  const int4 ch = T.chunks[blockIdx.x];  // body, face-list offset, count, chunk index in body
  const BodyDev B = T.body[ch.x];
  const TopoDev topo = T.topo[B.topo];
  const int lane = threadIdx.x & 31;
  const bool active = threadIdx.x < ch.z;
  if (threadIdx.x == 0) {
    s_hdr[0] = ch.x;
    s_hdr[1] = B.G[0];
    s_hdr[2] = B.G[1];
    s_hdr[3] = B.G[2];
    s_hdr[4] = B.closed;
    s_hdr[5] = B.chunk_off + ch.w;
    s_hdr[6] = ch.z;
  }
  if (FIELD && threadIdx.x < 3) {
    s_lo[threadIdx.x] = INT_MAX;
    s_hi[threadIdx.x] = INT_MIN;
    s_bmax[threadIdx.x] = 0u;
  }
  if (ROWMAP && !load) {
    // every row starts empty; done first, so that the stores overlap the
    // geometry loads (the barriers of the bounding-box reduction make them
    // visible)
    for (int q = threadIdx.x; q < MR / 4; q += MT)
      reinterpret_cast<uint4*>(s_xbits)[q] = make_uint4(0u, 0u, 0u, 0u);
  }
  if (FLUSH)
    for (int r = threadIdx.x; r < marker_mask_words(mn); r += MT) s_mask[r] = 0u;
  float Af = 0.f, Vf = 0.f;
  float nrm[3] = {0.f, 0.f, 0.f}, area = 0.f;
  float tc[3] = {0.f, 0.f, 0.f}, tp[3] = {0.f, 0.f, 0.f}, tm[3] = {0.f, 0.f, 0.f};
  float vb[3] = {0.f, 0.f, 0.f};     // centroid velocity, or the given marker force; then F
  float am[3] = {0.f, 0.f, 0.f};     // marker acceleration
  bool ok = false;
  int gf = 0;
  if (load && active) {
    const float4 c0 = cache_face[2 * ((size_t)blockIdx.x * kMT + threadIdx.x)];
    const float4 c1 = cache_face[2 * ((size_t)blockIdx.x * kMT + threadIdx.x) + 1];
    tc[0] = c0.x; tc[1] = c0.y; tc[2] = c0.z;
    area = c0.w;
    vb[0] = c1.x; vb[1] = c1.y; vb[2] = c1.z;
    ok = c1.w != 0.f;
  }
  if (active && !load) {
    // full patches are stored so that a warp's faces are spread over the patch
    // (its shared atomics of the spread rarely meet on a node) while thread t
    // reads record t
    const int4 mt = __ldg(T.mtri + topo.mface_off + ch.y + threadIdx.x);
    gf = B.f_off + mt.w;
    const int ia = B.v_off + mt.x, ib = B.v_off + mt.y, ic = B.v_off + mt.z;
    float xa[3], xb[3], xc[3];
#pragma unroll
    for (int d = 0; d < 3; ++d) {
      xa[d] = __ldg(x + d * V + ia);
      xb[d] = __ldg(x + d * V + ib);
      xc[d] = __ldg(x + d * V + ic);
    }
    // issued now, used after the row map: the velocity of the centroid
    // (interpolation) or the given marker force (spread only)
    if (INTERP) {
      const float third = 1.f / 3.f;
#pragma unroll
      for (int d = 0; d < 3; ++d)
        vb[d] = (__ldg(v + d * V + ia) + __ldg(v + d * V + ib) + __ldg(v + d * V + ic)) * third;
    } else if (SPREAD) {
#pragma unroll
      for (int d = 0; d < 3; ++d) vb[d] = __ldg(Fm_in + d * F + gf);
    }
    // marker acceleration (pressure correction): mean of the vertices'
    if (PROBE && !PLAIN && pr && accel) {
      const float third = 1.f / 3.f;
#pragma unroll
      for (int d = 0; d < 3; ++d)
        am[d] = (__ldg(accel + d * V + ia) + __ldg(accel + d * V + ib) +
                 __ldg(accel + d * V + ic)) * third;
    }
    const float e1[3] = {xb[0] - xa[0], xb[1] - xa[1], xb[2] - xa[2]};
    const float e2[3] = {xc[0] - xa[0], xc[1] - xa[1], xc[2] - xa[2]};
    const float N[3] = {e1[1] * e2[2] - e1[2] * e2[1], e1[2] * e2[0] - e1[0] * e2[2],
                        e1[0] * e2[1] - e1[1] * e2[0]};
    const float nn = sqrtf(N[0] * N[0] + N[1] * N[1] + N[2] * N[2]);
    area = 0.5f * nn;
    if (MEASURE) {
      Af = area;
      if (B.closed) {
        Vf = (xa[0] * (xb[1] * xc[2] - xb[2] * xc[1]) + xa[1] * (xb[2] * xc[0] - xb[0] * xc[2]) +
              xa[2] * (xb[0] * xc[1] - xb[1] * xc[0])) * (1.f / 6.f);
      }
    }
    if (FIELD) {
      const float third = 1.f / 3.f;
      const float inv = 1.f / nn;
      ok = nn > 0.f;
#pragma unroll
      for (int d = 0; d < 3; ++d) {
        const float c = (xa[d] + xb[d] + xc[d]) * third;
        nrm[d] = N[d] * inv;
        tc[d] = fmaf(c, g.invh[d], B.frac[d]);
        tp[d] = fmaf(c + sc.probe_h * nrm[d], g.invh[d], B.frac[d]);
        tm[d] = fmaf(c - sc.probe_h * nrm[d], g.invh[d], B.frac[d]);
        ok = ok && fabsf(tc[d]) < 4.0e6f && fabsf(tp[d]) < 4.0e6f && fabsf(tm[d]) < 4.0e6f;
      }
      if (!ok) atomicOr(T.err, ERR_NONFINITE);
    }
    if (PROBE) {
#pragma unroll
      for (int d = 0; d < 3; ++d) {
        s_own[d * MT] = tp[d];
        if (!PLAIN) s_own[(3 + d) * MT] = tm[d];
        s_own[(6 + d) * MT] = nrm[d];
        s_own[(9 + d) * MT] = vb[d];
      }
      if (!PLAIN) s_own[12 * MT] = am[0] * nrm[0] + am[1] * nrm[1] + am[2] * nrm[2];
#pragma unroll
      for (int d = 0; d < 3; ++d) {
        s_own[(13 + d) * MT] = tc[d];
        s_own[(16 + d) * MT] = 0.f;      // (G + G^T) n
      }
    }
    if (save) {
      cache_face[2 * ((size_t)blockIdx.x * kMT + threadIdx.x)] = make_float4(tc[0], tc[1], tc[2], area);
      cache_face[2 * ((size_t)blockIdx.x * kMT + threadIdx.x) + 1] =
          make_float4(vb[0], vb[1], vb[2], ok ? 1.f : 0.f);
    }
  }

  // ---- per-body area and volume: exact fixed-point sums -------------------
  // q = rint(value * 2^e) per face (2^e from the rest value), summed per warp
  // and added with 64-bit integer atomics: the body's sum does not depend on
  // the order of the additions.  The atomics follow the wait for the launch
  // before this one (a footprint clear zeroes the sums).
  if (MEASURE) {
    long long qa = 0, qv = 0;
    if (active) {
      const float ya = Af * B.sA, yv = Vf * B.sV;
      if (fabsf(ya) < B.qlim && fabsf(yv) < B.qlim) {
        qa = to_fixed(ya);
        qv = to_fixed(yv);
      } else {
        atomicOr(T.err, ERR_NONFINITE);
      }
    }
    qa = warp_sum_i64(qa);
    qv = warp_sum_i64(qv);
    if (lane == 0) {
      s_q[0][threadIdx.x >> 5] = (unsigned long long)qa;
      s_q[1][threadIdx.x >> 5] = (unsigned long long)qv;
    }
  }

  const bool mine = FIELD && active && ok;
  const bool two = PROBE && !PLAIN && !B.closed;   // open sheet: probes on both sides

  // ---- row map of the block's footprint -----------------------------------
  int ylo = 0, zlo = 0, sy = 0, sz = 0, xlo = 0, sx = 0;
  bool fit = false;
  int N = 0;
  if (ROWMAP && load) {
    // the tables of substep 0 of this coupled step: header, then one bulk
    // copy per table
    const int* hd = cache_tab + (size_t)blockIdx.x * cache_words(shape);
    xlo = hd[0];
    ylo = hd[1];
    zlo = hd[2];
    sx = hd[3];
    sy = hd[4];
    sz = hd[5];
    N = hd[6];
    fit = hd[7] != 0;
    const int nrows = fit ? sy * sz : 0;
    if (threadIdx.x == 0) {
      mbar_init(&s_bar, 1);
      const unsigned rb = 4u * (unsigned)pad4(nrows);
      const unsigned gb = fit ? 2u * (unsigned)((nrows + 1 + 7) & ~7) : 0u;
      const unsigned ob = fit ? 4u * (unsigned)pad4(N / 4) : 0u;
      mbar_arrive_tx(&s_bar, rb + gb + ob + (unsigned)sc.starve_tx);
      if (fit) {
        bulk_load(s_off4, hd + 16, rb, &s_bar);
        bulk_load(s_grp, hd + cache_groups_at(shape), gb, &s_bar);
        bulk_load(s_gofs, hd + cache_offsets_at(shape), ob, &s_bar);
      }
    }
    __syncthreads();   // barrier initialised
    if (!__syncthreads_and(mbar_wait(&s_bar, kCopyWaitClocks))) {
      // the copies did not land: flag it, give them one more bounded wait
      // (they write this block's shared memory) and leave
      if (threadIdx.x == 0) {
        atomicOr(T.err, ERR_TIMEOUT);
        mbar_wait(&s_bar, kCopyWaitClocks);
      }
      __syncthreads();
      return;
    }
    if (!fit && threadIdx.x == 0) atomicAdd(T.stats, 1);
  } else if (ROWMAP) {
    int mlo[3] = {INT_MAX, INT_MAX, INT_MAX}, mhi[3] = {INT_MIN, INT_MIN, INT_MIN};
    if (mine) {
#pragma unroll
      for (int l = 0; l < 3; ++l) {
        if ((l == 1 && !PROBE) || (l == 2 && !two)) continue;
        const float(&t)[3] = l == 0 ? tc : (l == 1 ? tp : tm);
#pragma unroll
        for (int d = 0; d < 3; ++d) {
          const int f0 = (int)floorf(t[d]);   // relative to the body's cell
          mlo[d] = min(mlo[d], f0 - 2);    // generous: every support lies in f0-1 .. f0+2
          mhi[d] = max(mhi[d], f0 + 3);
        }
      }
    }
#pragma unroll
    for (int d = 0; d < 3; ++d) {
      mlo[d] = __reduce_min_sync(0xffffffffu, mlo[d]);
      mhi[d] = __reduce_max_sync(0xffffffffu, mhi[d]);
    }
    __syncthreads();
    if (lane == 0) {
#pragma unroll
      for (int d = 0; d < 3; ++d) {
        atomicMin(&s_lo[d], mlo[d]);
        atomicMax(&s_hi[d], mhi[d]);
      }
    }
    __syncthreads();
    xlo = s_lo[0];
    ylo = s_lo[1];
    zlo = s_lo[2];
    sx = s_hi[0] >= s_lo[0] ? s_hi[0] - s_lo[0] + 1 : 0;
    sy = s_hi[1] >= s_lo[1] ? s_hi[1] - s_lo[1] + 1 : 0;
    sz = s_hi[2] >= s_lo[2] ? s_hi[2] - s_lo[2] + 1 : 0;
    const long long nrows = (long long)sy * sz;
    const bool rows_ok = nrows > 0 && nrows <= MR && sx <= 30000;
    if (rows_ok) {
      // a row's touched x in a 32-bit mask, one bit per interval of 4 nodes
      // (aligned to float4 in global memory when the grid allows vector
      // access; 4 x 2^k nodes where the patch is longer than 32 of them)
      const int xb = vec4 ? ((B.G[0] + xlo) & ~3) - B.G[0] : xlo;
      int ks = 2;
      while (((xlo + sx - 1 - xb) >> ks) >= 32) ++ks;
      if (mine) {
        // every component's support at a point with f = floor(tau) lies in
        // the 4x4x4 window f - 1 .. f + 2 (the nearest-node choice is exact
        // for |tau| < 2^22, which the position check guarantees)
#pragma unroll 1
        for (int l = 0; l < 3; ++l) {
          if ((l == 1 && !PROBE) || (l == 2 && !two)) continue;
          const float(&t)[3] = l == 0 ? tc : (l == 1 ? tp : tm);
          const int fx0 = (int)floorf(t[0]) - 1 - xb;
          const int r0 = ((int)floorf(t[1]) - 1 - ylo) + sy * ((int)floorf(t[2]) - 1 - zlo);
          const unsigned bits = (1u << (fx0 >> ks)) | (1u << ((fx0 + 3) >> ks));
#pragma unroll
          for (int k = 0; k < 4; ++k)
#pragma unroll
            for (int j = 0; j < 4; ++j) atomicOr(&s_xbits[r0 + j + sy * k], bits);
        }
      }
      __syncthreads();
      // row lengths in whole groups of 4 nodes and their exclusive scan, four
      // rows per thread and pass (rows past nrows stay empty)
      int carry = 0;
#pragma unroll 1
      for (int p0 = 0; p0 < (int)nrows; p0 += 4 * MT) {
        const int q4 = p0 / 4 + threadIdx.x;
        const bool in = q4 < MR / 4;
        int len[4], st[4], run = 0;
        {
          const uint4 m4 = in ? reinterpret_cast<const uint4*>(s_xbits)[q4] : make_uint4(0, 0, 0, 0);
          const unsigned m[4] = {m4.x, m4.y, m4.z, m4.w};
#pragma unroll
          for (int q = 0; q < 4; ++q) {
            const int f = __ffs(m[q]) - 1, l = 31 - __clz(m[q]);   // -1, -1 when empty
            st[q] = xb + (f << ks);
            len[q] = m[q] ? (l - f + 1) << ks : 0;
            run += len[q];
          }
        }
        int incl = run;
#pragma unroll
        for (int o = 1; o < 32; o <<= 1) {
          const int t = __shfl_up_sync(0xffffffffu, incl, o);
          if (lane >= o) incl += t;
        }
        if (lane == 31) s_warp[threadIdx.x >> 5] = incl;
        __syncthreads();
        int pos = carry + incl - run;
#pragma unroll
        for (int k = 0; k < MT / 32; ++k) {
          const int t = s_warp[k];
          if (k < (int)(threadIdx.x >> 5)) pos += t;
          carry += t;
        }
        if (in) {
          int o4[4];
          unsigned short gr[4];
#pragma unroll
          for (int q = 0; q < 4; ++q) {
            o4[q] = 4 * (pos - st[q]);
            gr[q] = (unsigned short)min(pos / 4, 65535);
            pos += len[q];
          }
          reinterpret_cast<int4*>(s_off4)[q4] = make_int4(o4[0], o4[1], o4[2], o4[3]);
          reinterpret_cast<ushort4*>(s_grp)[q4] = make_ushort4(gr[0], gr[1], gr[2], gr[3]);
          if (4 * q4 + 4 >= (int)nrows && 4 * q4 < (int)nrows)   // the end of the last row
            s_grp[4 * q4 + 4] = (unsigned short)min(pos / 4, 65535);
        }
        if (p0 + 4 * MT < (int)nrows) __syncthreads();   // the warp sums are used again
      }
      if (threadIdx.x == 0) s_N = carry;
      __syncthreads();
      N = s_N;
      fit = N <= mn;
      // the groups' global offsets, rows strided over the whole block (row r
      // is (y, z) = (r % sy, r / sy), followed incrementally)
      if (fit) {
        int yy = (int)threadIdx.x % sy, zz = (int)threadIdx.x / sy;
        const int dy = MT % sy, dz = MT / sy;
        for (int r = threadIdx.x; r < (int)nrows; r += MT) {
          const int k0 = s_grp[r], k1 = s_grp[r + 1];
          if (k1 > k0) {
            const int base = (wrap(B.G[2] + zlo + zz, g.n[2]) * g.n[1] +
                              wrap(B.G[1] + ylo + yy, g.n[1])) * g.n[0];
            int xg = wrap(B.G[0] + k0 * 4 - (s_off4[r] >> 2), g.n[0]);
            for (int k = k0; k < k1; ++k) {
              s_gofs[k] = base + xg;
              xg = wrap_pos(xg + 4, g.n[0]);
            }
          }
          yy += dy;
          zz += dz;
          if (yy >= sy) {
            yy -= sy;
            ++zz;
          }
        }
      }
    }
    if (!fit && threadIdx.x == 0) atomicAdd(T.stats, 1);
    __syncthreads();
    if (save) {
      int* hd = cache_tab + (size_t)blockIdx.x * cache_words(shape);
      if (threadIdx.x == 0) {
        hd[0] = xlo;
        hd[1] = ylo;
        hd[2] = zlo;
        hd[3] = sx;
        hd[4] = sy;
        hd[5] = sz;
        hd[6] = N;
        hd[7] = fit ? 1 : 0;
      }
      if (fit) {
        int* dst = hd + 16;
        unsigned short* gg = reinterpret_cast<unsigned short*>(hd + cache_groups_at(shape));
        for (int r = threadIdx.x; r <= sy * sz; r += MT) {
          if (r < sy * sz) dst[r] = s_off4[r];
          gg[r] = s_grp[r];
        }
        dst = hd + cache_offsets_at(shape);
        for (int q = threadIdx.x; q < N / 4; q += MT) dst[q] = s_gofs[q];
      }
    }
  }
  const RowTable RT{s_gofs, g.n[0], vec4};
  const StagedRows SR{dyn, -(ylo + sy * zlo), sy};
  const int ofsA = (int)(reinterpret_cast<unsigned char*>(bufA) - dyn);
  const int ngroups = fit ? N / 4 : 0;
  const bool dbl = 2 * N <= mn;                // two staging buffers
  float* bufB = bufA + mn / 2;

  // ---- the components, one after the other ---------------------------------
  // Velocity: interpolation at the centroid, gradient at the probes.  Where two
  // buffers fit, the components are staged in turn (u -> A, v -> B, w -> A, and
  // with a pressure field p -> B), the next one's copies in flight while the
  // current one is used.  Traction t = (G + G^T) n: component i yields (G n)_i and
  // adds n_i G_i. to G^T n; the pressure jump P = p+ - p- (open) or p (closed).
  // Spread: a component's marker forces are spread as soon as they are known,
  // with the factors of the interpolation, in exact fixed point (one 32-bit
  // word per staged node) in place of the component's staged velocity, and
  // flushed with float4 global atomics.
  if (FIELD && (VEL || FLUSH)) {
    const bool press = PROBE && !PLAIN && pr != nullptr;
    float Pj = 0.f;
    const float cl = area * sc.cl_scale;
    if (VEL && fit) {
      stage_async<MT>(bufA, u, RT, ngroups);
      cp_async_commit();
      if (dbl) stage_async<MT>(bufB, vv, RT, ngroups);
      cp_async_commit();
    }
    // the components in a loop, not unrolled: the unrolled kernel measured
    // slower (instruction fetch stalls)
#pragma unroll 1
    for (int comp = 0; comp < (press ? 4 : 3); ++comp) {
      const float* velc = comp == 0 ? u : (comp == 1 ? vv : (comp == 2 ? w : pr));
      float* buf = (dbl && (comp & 1)) ? bufB : bufA;
      const int obuf = ofsA + ((dbl && (comp & 1)) ? 2 * mn : 0);
      if (VEL && fit) {
        // one later group (the next component) may still be in flight
        if (dbl && (comp < 2 || (comp == 2 && press))) cp_async_wait<1>(); else cp_async_wait<0>();
        __syncthreads();   // every thread's copies of this component have landed
      }
      float Fc = 0.f;      // this component of the marker force
      if (PROBE && !PLAIN && comp == 3) {
        if (mine) {
          // probe pressure p* and the correction h (Du/Dt).n, per side with its
          // own normal: P = p*+ + h a.n (closed), p*+ - p*- + 2 h a.n (open)
          const float an = s_own[12 * MT];
#pragma unroll 1
          for (int l = 0; l < (two ? 2 : 1); ++l) {
            int cc[3];
            float t3[3];
            const float* o = s_own + 3 * l * MT;
            const float t[3] = {o[0], o[MT], o[2 * MT]};
            locate(t, 3, cc, t3);
            DirW X, Y, Z;
            dir_weights(t3[0], sc.mk, X);
            dir_weights(t3[1], sc.mk, Y);
            dir_weights(t3[2], sc.mk, Z);
            const float ps = fit ? mls_value((const float*)nullptr, SR.at(cc, obuf), X, Y, Z)
                                 : value_global<FEW>(pr, g, T.body + s_hdr[0], cc[0], cc[1], cc[2], X, Y, Z);
            Pj += (l == 0 ? 1.f : -1.f) * ps + sc.probe_h * an;
          }
        }
        continue;
      }
      if (PROBE && mine) {
        // open sheet: (tau+ - tau-) . n+
        float gr[3] = {0.f, 0.f, 0.f};
#pragma unroll 1
        for (int l = 0; l < (two ? 2 : 1); ++l) {
          ProbeW P;
          const float* o = s_own + 3 * l * MT;
          const float t[3] = {o[0], o[MT], o[2 * MT]};
          P.prepare(t, comp, sc.mk);
          float q[3];
          if (fit) {
            mls_grad((const float*)nullptr, SR.at(P.cc, obuf), P.X, P.Y, P.Z, q);
          } else {
            const float3 q3 = gradient_global<FEW>(velc, g, T.body + s_hdr[0], P);
            q[0] = q3.x;
            q[1] = q3.y;
            q[2] = q3.z;
          }
#pragma unroll
          for (int j = 0; j < 3; ++j) gr[j] += l == 0 ? q[j] : -q[j];
        }
#pragma unroll
        for (int j = 0; j < 3; ++j) gr[j] *= sc.kg[j];
        const float n[3] = {s_own[6 * MT], s_own[7 * MT], s_own[8 * MT]};
        const float gn = gr[0] * n[0] + gr[1] * n[1] + gr[2] * n[2];
        const float ni = comp == 0 ? n[0] : (comp == 1 ? n[1] : n[2]);
#pragma unroll
        for (int j = 0; j < 3; ++j)
          s_own[(16 + j) * MT] = fmaf(ni, gr[j], s_own[(16 + j) * MT] + (comp == j ? gn : 0.f));
      }
      // the centroid's factors, for the interpolation and the spread (after the
      // probes: what both need does not fit in registers)
      DirW CX, CY, CZ;
      int ccC[3];
      if ((INTERP || FLUSH) && mine) {
        float t3[3];
        if (PROBE) {
#pragma unroll
          for (int d = 0; d < 3; ++d) tc[d] = s_own[(13 + d) * MT];
        }
        locate(tc, comp, ccC, t3);
        dir_weights(t3[0], sc.mk, CX);
        dir_weights(t3[1], sc.mk, CY);
        dir_weights(t3[2], sc.mk, CZ);
      }
      if (mine) {
        if (INTERP) {
          const float Ul = fit ? mls_value((const float*)nullptr, SR.at(ccC, obuf), CX, CY, CZ)
                               : value_global<FEW>(velc, g, T.body + s_hdr[0], ccC[0], ccC[1], ccC[2], CX, CY, CZ);
          const float Vb = PROBE ? s_own[(9 + comp) * MT]
                                 : (comp == 0 ? vb[0] : (comp == 1 ? vb[1] : vb[2]));
          Fc = (Vb - Ul) * sc.inv_dt;
          if (REC && PROBE) s_own[(9 + comp) * MT] = Fc;   // kept for the record
          if (REC && !PROBE) {
            if (comp == 0) vb[0] = Fc;
            if (comp == 1) vb[1] = Fc;
            if (comp == 2) vb[2] = Fc;
          }
          if (U) U[comp * F + gf] = Ul;
          if (Fm) Fm[comp * F + gf] = Fc;
        } else if (FLUSH) {
          Fc = comp == 0 ? vb[0] : (comp == 1 ? vb[1] : vb[2]);
        }
      }
      if (FLUSH) {
        const float coef = mine ? cl * Fc : 0.f;
        float* fc = comp == 0 ? fx : (comp == 1 ? fy : fz);
        if (fit) {
          if (FEW) {
            // (over 256, so that it overflows only where a single one would)
            float ws = fabsf(coef) * 0x1p-8f;
#pragma unroll
            for (int o = 16; o > 0; o >>= 1) ws += __shfl_xor_sync(0xffffffffu, ws, o);
            if (lane == 0) s_bsum[comp][threadIdx.x >> 5] = ws;
          } else {
            // non-negative floats order as their bit patterns, a NaN above all
            const unsigned wm = __reduce_max_sync(0xffffffffu, __float_as_uint(fabsf(coef)));
            if (lane == 0) atomicMax(&s_bmax[comp], wm);
          }
          __syncthreads();   // the bound is known and the staged component used up
          int4* acc4 = reinterpret_cast<int4*>(buf);
          for (int q = threadIdx.x; q < ngroups; q += MT) acc4[q] = make_int4(0, 0, 0, 0);
          __syncthreads();
          float bm = FEW ? 0.f : __uint_as_float(s_bmax[comp]);
          if (FEW) {
#pragma unroll
            for (int k = 0; k < MT / 32; ++k) bm += s_bsum[comp][k];
          }
          bm *= phi_bound_all;
          const bool fin = bm <= 3.0e38f;
          if (!fin && threadIdx.x == 0) atomicOr(T.err, ERR_NONFINITE);
          if (fin && bm > 0.f) {   // uniform over the block
            // scale 2^k such that what a node can take stays below 2^31 (with room for
            // the roundings: 1.001): MT contributions of at most bm, or all the block's
            // contributions, 256 bm.  The sum makes it one to three bits finer at 1.3 %
            // of a full launch, where FEW has idle issue slots and patches of few, large
            // contributions, which the largest one alone scales worst (six drops of 11 to
            // 22 cells: f against float64 3.4e-6 with a bound of 2^30 and the largest,
            // 2.2e-6 now; 3.1e-6 when such patches took the global path)
            constexpr int kTop = !FEW && MT == 128 ? 23 : 22;
            const int k = max(min(kTop - ilogbf(bm * 1.001f), 120), -126);
            if (coef != 0.f)
              mls_spread_fixed(dyn, SR.at(ccC, obuf), CX, CY, CZ, coef * pow2f(k));
            __syncthreads();
            // The fields and the footprint record meet what the clear of this
            // step writes, which may be the grid launched just before this one
            // (this kernel may start while it still runs): wait for that grid
            // to complete (immediate when nothing precedes programmatically).
            asm volatile("griddepcontrol.wait;" ::: "memory");
            const float inv = pow2f(-k);
            for (int q0 = threadIdx.x - lane; q0 < ngroups; q0 += MT) {
              const int q = q0 + lane;
              const int4 a = q < ngroups ? acc4[q] : make_int4(0, 0, 0, 0);
              const bool nz = (a.x | a.y | a.z | a.w) != 0;
              const unsigned bal = __ballot_sync(0xffffffffu, nz);
              if (lane == 0) s_mask[q0 >> 5] |= bal;
              if (!nz) continue;
              const float4 va = make_float4((float)a.x * inv, (float)a.y * inv, (float)a.z * inv,
                                            (float)a.w * inv);
              if (vec4) {
                atomicAdd(reinterpret_cast<float4*>(fc + RT.node(q, 0)), va);
              } else {
#pragma unroll
                for (int jj = 0; jj < 4; ++jj) {
                  const float xq = jj == 0 ? va.x : (jj == 1 ? va.y : (jj == 2 ? va.z : va.w));
                  if (xq != 0.f) atomicAdd(fc + RT.node(q, jj), xq);
                }
              }
            }
          }
        } else {
          asm volatile("griddepcontrol.wait;" ::: "memory");
          if (mine)
            spread_global<FEW>(fc, g, T.body + s_hdr[0], ccC[0], ccC[1], ccC[2], CX, CY, CZ, coef);
        }
      }
      // the next component into the buffer that is free again (with the spread,
      // each thread copies into the groups it has just flushed)
      const int next = comp + (dbl ? 2 : 1);
      if (VEL && fit && next < (press ? 4 : 3)) {
        if (!FLUSH) __syncthreads();
        stage_async<MT>(buf, next == 1 ? vv : (next == 2 ? w : pr), RT, ngroups);
        cp_async_commit();
      }
    }
    if (PROBE && mine) {
      const float s = sc.mu * area;
#pragma unroll
      for (int i = 0; i < 3; ++i) {
        const float t = s * s_own[(16 + i) * MT];
        Fext[i * F + gf] = press ? t - area * Pj * s_own[(6 + i) * MT] : t;
      }
    }
  }

  // ---- records of the tile-owned spread ------------------------------------
  if (REC && !ROWMAP) __syncthreads();   // the header
  if (REC && active) {
    float4 r0 = make_float4(0.f, 0.f, 0.f, __int_as_float(-1));
    float4 r1 = make_float4(0.f, 0.f, 0.f, 0.f);
    if (mine) {
      const float cl = area * sc.cl_scale;
#pragma unroll
      for (int i = 0; i < 3; ++i)
        if (PROBE) {
          vb[i] = s_own[(9 + i) * MT];
          tc[i] = s_own[(13 + i) * MT];
        }
      r0 = make_float4(tc[0], tc[1], tc[2], __int_as_float(s_hdr[0]));
      r1 = make_float4(cl * vb[0], cl * vb[1], cl * vb[2], 0.f);
      int tx[3], ty[3], tz[3];
      const int nx_ = tiles_along(s_hdr[1] + (int)floorf(tc[0]), g.n[0], kTX, tx);
      const int ny_ = tiles_along(s_hdr[2] + (int)floorf(tc[1]), g.n[1], kTY, ty);
      const int nz_ = tiles_along(s_hdr[3] + (int)floorf(tc[2]), g.n[2], kTZ, tz);
      const unsigned m0 = __float_as_uint(fabsf(r1.x)), m1 = __float_as_uint(fabsf(r1.y)),
                     m2 = __float_as_uint(fabsf(r1.z));
      // reductions without a returned value: nothing waits on them
#pragma unroll
      for (int a = 0; a < 3; ++a)
#pragma unroll
        for (int b = 0; b < 3; ++b)
#pragma unroll
          for (int c = 0; c < 3; ++c)
            if (a < nz_ && b < ny_ && c < nx_) {
              const int t = (tz[a] * td.nt[1] + ty[b]) * td.nt[0] + tx[c];
              atomicAdd(td.count + t, 1);
              atomicMax(td.tmax + 4 * (size_t)t, m0);
              atomicMax(td.tmax + 4 * (size_t)t + 1, m1);
              atomicMax(td.tmax + 4 * (size_t)t + 2, m2);
            }
    }
    td.rec[2 * (size_t)gf] = r0;
    td.rec[2 * (size_t)gf + 1] = r1;
  }

  // the body sums and the footprint record meet what the clear writes, too
  asm volatile("griddepcontrol.wait;" ::: "memory");
  if (!FIELD) __syncthreads();   // the header
  if (MEASURE && lane == 0 && (int)(threadIdx.x & ~31) < s_hdr[6]) {
    const int b = s_hdr[0];
    atomicAdd(T.qsum + 2 * b, s_q[0][threadIdx.x >> 5]);
    if (s_hdr[4]) atomicAdd(T.qsum + 2 * b + 1, s_q[1][threadIdx.x >> 5]);
  }
  if (FLUSH && record) {
    // footprint for the next step's clear: per row the x-range of the groups
    // that received a nonzero spread, the bounding box (flag 1) otherwise
    const int gc = s_hdr[5];
    const int rows = sy * sz;
    int count = rows;
    if (fit) {
      // more rows than the record holds: only those that received something,
      // in order (the record does not depend on the blocks' timing)
      const bool compact = rows > kMaxRows;
      int done = 0;
      __syncthreads();   // every warp's bits
      for (int p0 = 0; p0 < rows; p0 += MT) {
        const int r = p0 + threadIdx.x;
        int lo = 0, hi = -1;   // the row's groups
        if (r < rows) {
          lo = s_grp[r];
          hi = s_grp[r + 1] - 1;
        }
        // first set bit at or after lo, last at or before hi, a word at a time
        while (lo <= hi) {
          const unsigned m = s_mask[lo >> 5] >> (lo & 31);
          if (m) {
            lo += __ffs(m) - 1;
            break;
          }
          lo = (lo | 31) + 1;
        }
        while (hi >= lo) {
          const unsigned m = s_mask[hi >> 5] << (31 - (hi & 31));
          if (m) {
            hi -= __clz(m);
            break;
          }
          hi = (hi & ~31) - 1;
        }
        int2 e = make_int2(0, 0);
        if (lo <= hi) {
          const int L = min(4 * (hi - lo + 1), g.n[0]);
          const int x0 = wrap(s_hdr[1] + 4 * lo - (s_off4[r] >> 2), g.n[0]);
          e = make_int2(s_gofs[lo] - x0, x0 | (L << 16));
        }
        int at = r;
        bool put = r < rows;
        if (compact) {
          const unsigned bal = __ballot_sync(0xffffffffu, lo <= hi);
          if (lane == 0) s_warp[threadIdx.x >> 5] = __popc(bal);
          __syncthreads();
          at = done + __popc(bal & ((1u << lane) - 1u));
          for (int k = 0; k < MT / 32; ++k) {
            if (k < (int)(threadIdx.x >> 5)) at += s_warp[k];
            done += s_warp[k];
          }
          __syncthreads();
          put = lo <= hi && at < kMaxRows;
        }
        if (put) T.rowmap[(size_t)gc * kMaxRows + at] = e;
      }
      if (compact) count = done;
    }
    if (threadIdx.x == 0) {
      const bool box = !fit || count > kMaxRows;   // more rows than the record holds: its box
      T.boxes[2 * gc] = make_int4(s_hdr[1] + xlo, s_hdr[2] + ylo, s_hdr[3] + zlo,
                                  box ? 1 : (vec4 ? 2 : 0));
      T.boxes[2 * gc + 1] = make_int4(min(sx, g.n[0]), min(sy, g.n[1]), min(sz, g.n[2]),
                                      box ? 0 : count);
    }
  }
}

// Zero the force fields on the footprint each marker block recorded in its
// last spread: its rows' nonzero x-ranges, or its bounding box when it took
// the global path.  Zeroing more than the footprint is harmless (everything
// nonzero belongs to some recorded footprint), so vector rows are widened to
// whole 32-byte sectors when nx allows, which avoids partial-sector writes
// (widening further to 64 bytes measured slower: more bytes written).
__global__ void __launch_bounds__(256) clear_kernel(DeviceTables T, Grid g, float* __restrict__ fx,
                                                    float* __restrict__ fy, float* __restrict__ fz,
                                                    int vec4, const int4* __restrict__ chunks,
                                                    int4* __restrict__ boxes,
                                                    const int2* __restrict__ rowmap, int max_rows) {
  // the marker kernel launched after this one may start at once: it waits
  // for this grid's completion before it touches what this grid writes
  asm volatile("griddepcontrol.launch_dependents;");
  // the first chunk of each body also zeroes the body's fixed-point sums
  if (threadIdx.x == 0) {
    const int4 ch = chunks[blockIdx.x];
    if (ch.w == 0) {
      T.qsum[2 * ch.x] = 0ull;
      T.qsum[2 * ch.x + 1] = 0ull;
    }
  }
  const int4 lo = boxes[2 * blockIdx.x];
  const int4 sz = boxes[2 * blockIdx.x + 1];
  if (sz.x <= 0 || sz.y <= 0 || sz.z <= 0) return;
  const int nx = g.n[0];
  if (lo.w == 1) {
    // the (y, z) rows of the box, as many lanes to a row as it has float4s (nodes), a
    // power of two; aligned rows are widened to whole float4s.  One block per box: with a
    // warp per row and a node per lane the five boxes of a drop of 30 cells took 80 us,
    // now 27 (58 on rows that are not whole float4s)
    int x0 = wrap(lo.x, nx), L = sz.x;
    if (vec4) {
      L = min((L + (x0 & 3) + 3) & ~3, nx);
      x0 &= ~3;
    }
    const int step = vec4 ? 4 : 1, nq = L / step;
    int W = 32;
    while (W / 2 >= nq) W /= 2;
    const int per = blockDim.x / W, dj = per % sz.y, dk = per / sz.y;
    const long long rows = (long long)sz.y * sz.z;
    const int first = threadIdx.x / W;
    int k = first / sz.y, j = first - k * sz.y;
    for (long long r = first; r < rows; r += per) {
      const size_t base = (size_t)(unsigned)(wrap(lo.z + k, g.n[2]) * g.n[1] + wrap(lo.y + j, g.n[1])) *
                          (unsigned)nx;
      for (int q = threadIdx.x & (W - 1); q < nq; q += W) {
        int xg = x0 + step * q;
        if (xg >= nx) xg -= nx;
        const size_t o = base + xg;
        if (vec4) {
          const float4 z4 = make_float4(0.f, 0.f, 0.f, 0.f);
          *reinterpret_cast<float4*>(fx + o) = z4;
          *reinterpret_cast<float4*>(fy + o) = z4;
          *reinterpret_cast<float4*>(fz + o) = z4;
        } else {
          fx[o] = 0.f;
          fy[o] = 0.f;
          fz[o] = 0.f;
        }
      }
      j += dj;
      k += dk;
      if (j >= sz.y) {
        j -= sz.y;
        ++k;
      }
    }
  } else {
    // float4 stores only for rows recorded in whole float4 groups
    vec4 = vec4 && lo.w == 2;
    const int nrows = sz.w;
    const int2* rm = rowmap + (size_t)blockIdx.x * max_rows;
    const int al = nx % 8 == 0 ? 8 : 4;   // widening, in floats
    // each warp takes 32 rows at a time: one coalesced load of their records,
    // then its groups of `W` lanes clear W rows each, the records passed by
    // shuffles.  Four lanes of float4s: a row's 64 bytes are the common case; with
    // eight, half of the lanes had nothing to store (7.1 -> 4.6 us for one drop,
    // 19 -> 16.6 for 500; 63 us for 1000 drops on 512^3, bound by the writes)
    const int lane = threadIdx.x & 31;
    const int W = vec4 ? 4 : 8, sub = lane & (W - 1), first = lane & ~(W - 1);
    for (int r0 = (threadIdx.x >> 5) * 32; r0 < nrows; r0 += blockDim.x) {
      const int2 mine = r0 + lane < nrows ? rm[r0 + lane] : make_int2(0, 0);
#pragma unroll 2
      for (int j = 0; j < W; ++j) {
        const int src = first + j;
        const int ex = __shfl_sync(0xffffffffu, mine.x, src);
        const int ey = __shfl_sync(0xffffffffu, mine.y, src);
        int L = ey >> 16, x0 = ey & 0xFFFF;  // (row base, first x wrapped | length << 16)
        if (L <= 0) continue;
        if (vec4) {
          L = min((L + (x0 & (al - 1)) + al - 1) & ~(al - 1), nx);
          x0 &= ~(al - 1);
          for (int q = 4 * sub; q < L; q += 4 * W) {
            int xg = x0 + q;
            if (xg >= nx) xg -= nx;
            const size_t o = (size_t)ex + xg;
            const float4 z4 = make_float4(0.f, 0.f, 0.f, 0.f);
            *reinterpret_cast<float4*>(fx + o) = z4;
            *reinterpret_cast<float4*>(fy + o) = z4;
            *reinterpret_cast<float4*>(fz + o) = z4;
          }
        } else {
          for (int q = sub; q < L; q += W) {
            int xg = x0 + q;
            if (xg >= nx) xg -= nx;
            const size_t o = (size_t)ex + xg;
            fx[o] = 0.f;
            fy[o] = 0.f;
            fz[o] = 0.f;
          }
        }
      }
    }
  }
  __syncthreads();
  if (threadIdx.x == 0) boxes[2 * blockIdx.x + 1] = make_int4(0, 0, 0, 0);
}

// (A, V) in float64 and the global-term coefficients from the fixed-point sums
__global__ void measure_finalize_kernel(DeviceTables T, int32_t nb) {
  const int b = blockIdx.x * blockDim.x + threadIdx.x;
  if (b >= nb) return;
  const BodyDev B = T.body[b];
  const unsigned long long qa = T.qsum[2 * b], qv = T.qsum[2 * b + 1];
  T.meas[2 * b] = (double)(long long)qa / (double)B.sA;
  T.meas[2 * b + 1] = B.closed ? (double)(long long)qv / (double)B.sV : 0.0;
  T.coef[b] = body_coef(B, qa, qv);
}

// null (unused) pointers count as aligned
inline bool aligned16(const void* p) { return (reinterpret_cast<uintptr_t>(p) & 15u) == 0; }

template <int MT, bool M, bool I, bool P, bool S, bool R>
cudaError_t launch_mt(ibm_ctx* c, const float* x, const float* v, const float* u, const float* vv,
                      const float* w, const float* pr, const float* accel, float* U, float* Fm,
                      const float* Fm_in, float* Fext, float* fx, float* fy, float* fz,
                      int record, const DeviceTables* tab, int cache, bool pdl) {
  const bool rows = I || P || (S && !R);
  const MarkerShape ms = rows ? c->mshape[P ? 1 : 0] : MarkerShape{0, 0};
  const size_t smem = rows ? marker_smem_bytes(MT, ms, P) : 0;
  const int vec4 = c->vec4 && aligned16(u) && aligned16(vv) && aligned16(w) && aligned16(pr) &&
                   aligned16(fx) && aligned16(fy) && aligned16(fz);
  // pdl: launched as the programmatic dependent of the footprint clear just
  // before it on the stream (it may start once every clear block runs)
  cudaLaunchConfig_t cfg = {};
  cfg.gridDim = dim3((unsigned)c->n_chunks);
  cfg.blockDim = dim3(MT);
  cfg.dynamicSmemBytes = smem;
  cfg.stream = c->stream;
  cudaLaunchAttribute attr[2];
  cfg.attrs = attr;
  cfg.numAttrs = 0;
  if (pdl) {
    attr[cfg.numAttrs].id = cudaLaunchAttributeProgrammaticStreamSerialization;
    attr[cfg.numAttrs++].val.programmaticStreamSerializationAllowed = 1;
  }
  // patches on the global path want an L1 that their blocks' shared memory leaves
  if (rows && c->marker_carveout[P ? 1 : 0]) {
    attr[cfg.numAttrs].id = cudaLaunchAttributePreferredSharedMemoryCarveout;
    attr[cfg.numAttrs++].val.sharedMemCarveout = (unsigned)c->marker_carveout[P ? 1 : 0];
  }
  auto kernel = marker_kernel<MT, M, I, P, S, R, kPlain>;
  if constexpr (P)
    if (pr || c->any_open) kernel = marker_kernel<MT, M, I, P, S, R, kAll>;
  if constexpr (I || P || S)
    if (c->marker_few[P ? 1 : 0]) kernel = marker_kernel<MT, M, I, P, S, R, kFew>;
  return cudaLaunchKernelEx(&cfg, kernel, tab ? *tab : c->d, c->grid,
                            c->sc, (int32_t)c->V, (int32_t)c->F, x, v, u, vv, w, pr, accel, U,
                            Fm, Fm_in, Fext, fx, fy, fz, record, vec4, c->td,
                            c->phi_bound, cache, c->fc_tab, c->fc_face, ms);
}

// the marker kernel for the context's patch size (128 or 256 faces per block)
template <bool M, bool I, bool P, bool S, bool R = false>
cudaError_t launch_t(ibm_ctx* c, const float* x, const float* v, const float* u, const float* vv,
                     const float* w, const float* pr, const float* accel, float* U, float* Fm,
                     const float* Fm_in, float* Fext, float* fx, float* fy, float* fz,
                     int record, const DeviceTables* tab = nullptr, int cache = 0,
                     bool pdl = false) {
  if (c->n_chunks == 0) return cudaSuccess;
  if (c->marker_patch == 128)
    return launch_mt<128, M, I, P, S, R>(c, x, v, u, vv, w, pr, accel, U, Fm, Fm_in, Fext, fx, fy,
                                         fz, record, tab, cache, pdl);
  return launch_mt<kMT, M, I, P, S, R>(c, x, v, u, vv, w, pr, accel, U, Fm, Fm_in, Fext, fx, fy,
                                       fz, record, tab, cache, pdl);
}

}  // namespace

template <int MT, bool M, bool I, bool P, bool S, bool R>
cudaError_t marker_smem_limit() {
  auto set = [](auto kernel) {
    return cudaFuncSetAttribute(kernel, cudaFuncAttributeMaxDynamicSharedMemorySize,
                                marker_smem_max(MT, P));
  };
  cudaError_t e = set(marker_kernel<MT, M, I, P, S, R, kPlain>);
  if constexpr (P)
    if (e == cudaSuccess) e = set(marker_kernel<MT, M, I, P, S, R, kAll>);
  return e == cudaSuccess ? set(marker_kernel<MT, M, I, P, S, R, kFew>) : e;
}

cudaError_t set_marker_smem_limit() {
  cudaError_t e = cudaSuccess;
#define SET(M, I, P, S, R)                                                    \
  if (e == cudaSuccess) e = marker_smem_limit<kMT, M, I, P, S, R>();          \
  if (e == cudaSuccess) e = marker_smem_limit<128, M, I, P, S, R>();
  SET(true, true, true, true, false)
  SET(true, false, true, false, false)
  SET(false, true, true, false, false)
  SET(false, true, false, false, false)
  SET(false, false, true, false, false)
  SET(false, false, false, true, false)
  SET(false, true, false, true, false)
  SET(true, true, true, true, true)
  SET(false, true, false, true, true)
#undef SET
  return e;
}

cudaError_t launch_mls(ibm_ctx* c, const float* x, const float* v, const float* u,
                       const float* vv, const float* w, const float* pr, const float* accel,
                       float* U, float* Fm, const float* Fm_in, float* Fext, float* fx, float* fy,
                       float* fz, bool measure, bool interp, bool probe, bool spread,
                       bool record_box, bool after_clear) {
  const int rb = record_box ? 1 : 0;
#define L(M, I, P, S) \
  launch_t<M, I, P, S>(c, x, v, u, vv, w, pr, accel, U, Fm, Fm_in, Fext, fx, fy, fz, rb)
  if (measure && interp && probe && spread)
    return launch_t<true, true, true, true>(c, x, v, u, vv, w, pr, accel, U, Fm, Fm_in, Fext, fx,
                                            fy, fz, rb, nullptr, 0, after_clear);
  if (measure && !interp && !probe && !spread) return L(true, false, false, false);
  if (measure && !interp && probe && !spread) return L(true, false, true, false);
  if (!measure && interp && probe && !spread) return L(false, true, true, false);
  if (!measure && interp && !probe && !spread) return L(false, true, false, false);
  if (!measure && !interp && probe && !spread) return L(false, false, true, false);
  if (!measure && !interp && !probe && spread) return L(false, false, false, true);
  if (!measure && interp && !probe && spread) return L(false, true, false, true);
#undef L
  return cudaErrorInvalidValue;
}

cudaError_t launch_mls_records(ibm_ctx* c, const float* x, const float* v, const float* u,
                               const float* vv, const float* w, const float* p,
                               const float* accel, const float* Fm_in, float* Fext, bool measure,
                               bool probe) {
  if (measure && probe)   // the step: body sums, interpolation, traction, records
    return launch_t<true, true, true, true, true>(c, x, v, u, vv, w, p, accel, nullptr, nullptr,
                                                  nullptr, Fext, nullptr, nullptr, nullptr, 0);
  if (!measure && !probe && u)   // the coupled forcing: interpolation and records
    return launch_t<false, true, false, true, true>(c, x, v, u, vv, w, nullptr, nullptr, nullptr,
                                                    nullptr, nullptr, nullptr, nullptr, nullptr,
                                                    nullptr, 0);
  if (!measure && !probe && Fm_in)   // given marker forces
    return launch_t<false, false, false, true, true>(c, x, nullptr, nullptr, nullptr, nullptr,
                                                     nullptr, nullptr, nullptr, nullptr, Fm_in,
                                                     nullptr, nullptr, nullptr, nullptr, 0);
  return cudaErrorInvalidValue;
}

cudaError_t zero_body_sums(ibm_ctx* c) {
  if (c->B == 0) return cudaSuccess;
  return cudaMemsetAsync(c->d.qsum, 0, sizeof(unsigned long long) * 2 * c->B, c->stream);
}

cudaError_t launch_measure_finalize(ibm_ctx* c) {
  if (c->B == 0) return cudaSuccess;
  measure_finalize_kernel<<<(unsigned)((c->B + 127) / 128), 128, 0, c->stream>>>(c->d,
                                                                               (int32_t)c->B);
  return cudaGetLastError();
}

cudaError_t launch_clear(ibm_ctx* c, float* fx, float* fy, float* fz) {
  if (c->n_chunks == 0) return cudaSuccess;
  const int vec4 = c->vec4 && aligned16(fx) && aligned16(fy) && aligned16(fz);
  clear_kernel<<<c->n_chunks, 256, 0, c->stream>>>(c->d, c->grid, fx, fy, fz, vec4, c->d.chunks,
                                                  c->d.boxes, c->d.rowmap, kMaxRows);
  return cudaGetLastError();
}

// The coupled forcing of substep `substep` (interpolation of u* and spread
// at the centroids of x): footprints recorded in the flow's own record (the
// step's record is left alone), the previous substep's footprint cleared
// first (substep 0: the caller zeroes the fields), and the face geometry and
// row tables saved in substep 0 and loaded in substeps 1 and 2.
cudaError_t launch_forcing(ibm_ctx* c, int substep, const float* x, const float* xv,
                           const float* u, const float* vv, const float* w, float* fx, float* fy,
                           float* fz) {
  if (c->n_chunks == 0) return cudaSuccess;
  DeviceTables t = c->d;
  t.boxes = c->fc_boxes;
  t.rowmap = c->fc_rowmap;
  if (substep > 0) {
    const int vec4 = c->vec4 && aligned16(fx) && aligned16(fy) && aligned16(fz);
    clear_kernel<<<c->n_chunks, 256, 0, c->stream>>>(t, c->grid, fx, fy, fz, vec4, c->d.chunks,
                                                    t.boxes, t.rowmap, kMaxRows);
    const cudaError_t e = cudaGetLastError();
    if (e != cudaSuccess) return e;
  }
  return launch_t<false, true, false, true>(c, x, xv, u, vv, w, nullptr, nullptr, nullptr, nullptr,
                                            nullptr, nullptr, fx, fy, fz, 1, &t,
                                            substep == 0 ? 1 : 2);
}

}  // namespace ibm
