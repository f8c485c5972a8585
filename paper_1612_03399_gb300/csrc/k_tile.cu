// Tile-owned spreading of the marker forces onto the staggered grid (Sec. 2.2,
// Eq. mls_cl: f_i^k = sum over the markers l whose support holds node k of
// c_l phi_k^l F_i^l), deterministic and without global atomics on the fields.
//
// The marker kernel (record mode) writes one record per marker (centroid in
// cells, c_l F) and counts, per tile of kTX x kTY x kTZ grid nodes, the markers
// whose centroid supports reach it (the union over the three components of the
// 3x3x3 nearest-node supports: nodes f-1 .. f+2 per direction), with the
// largest |c_l F| per component.  Then:
//   tile_scan_kernel    every tile once: reached tiles get a range in the
//                       marker list and are listed, with the tiles the previous
//                       clear-mode call reached and this one does not,
//   tile_fill_kernel    each marker writes its id into the ranges of its tiles,
//   tile_spread_kernel  one block per listed tile and component: every listed
//                       marker adds c_l phi F to the nodes it supports, in exact
//                       fixed point in shared memory (a power-of-two scale per
//                       tile and component, so the sum does not depend on the
//                       order); the tile then stores every 8-node x-segment that
//                       received contributions or that the previous clear-mode
//                       call left nonzero (a bit mask per tile), with plain
//                       stores: each node is written by exactly one block, once.
// A clear-mode call thereby leaves exactly this call's forces in the fields
// (no separate clear, no read of the fields); accumulate mode adds the tile's
// nonzero nodes to the fields' values (read, add, store: still one owner per
// node).  The epoch of clear-mode calls is kept on the device, so a captured
// sequence of steps needs no host state.
#include <cuda_runtime.h>
#include <limits.h>
#include <math.h>

#include <algorithm>

#include "ibm_internal.cuh"
#include "mls_closed_form.cuh"

namespace ibm {
namespace {

// begin a call: the epoch (clear mode), the list length, the pair total, and
// the fixed-point body sums of the marker kernel
__global__ void tile_begin_kernel(TileDev td, unsigned long long* qsum, int nq, int accumulate) {
  const int i = blockIdx.x * blockDim.x + threadIdx.x;
  if (i == 0) {
    if (!accumulate) td.state[TS_EPOCH] += 1;
    td.state[TS_LEN] = 0;
    td.state[TS_PAIRS] = 0;
  }
  if (qsum && i < nq) qsum[i] = 0ull;
}

// block-wide exclusive scan of v (blockDim.x multiple of 32, <= 1024); returns
// the exclusive prefix, *total the block's sum (s_warp: 32 ints of scratch)
__device__ __forceinline__ int block_scan(int v, int* s_warp, int* total) {
  const int lane = threadIdx.x & 31, wid = threadIdx.x >> 5, nw = blockDim.x >> 5;
  int incl = v;
#pragma unroll
  for (int o = 1; o < 32; o <<= 1) {
    const int y = __shfl_up_sync(0xffffffffu, incl, o);
    if (lane >= o) incl += y;
  }
  if (lane == 31) s_warp[wid] = incl;
  __syncthreads();
  if (wid == 0) {
    int w = lane < nw ? s_warp[lane] : 0;
#pragma unroll
    for (int o = 1; o < 32; o <<= 1) {
      const int y = __shfl_up_sync(0xffffffffu, w, o);
      if (lane >= o) w += y;
    }
    if (lane < nw) s_warp[lane] = w;
  }
  __syncthreads();
  const int ex = (wid ? s_warp[wid - 1] : 0) + incl - v;
  *total = s_warp[nw - 1];
  __syncthreads();
  return ex;
}

// every tile once: the tiles that markers reach in this call get a range in
// the marker list and are listed; in clear mode so are the tiles that the
// previous clear-mode call listed and this one does not (their segments are
// zeroed), and the reached tiles take this call's epoch
template <bool CLEAR>
__global__ void __launch_bounds__(1024) tile_scan_kernel(TileDev td) {
  __shared__ int s_warp[32];
  __shared__ int s_pbase, s_lbase;
  const int t = blockIdx.x * blockDim.x + threadIdx.x;
  const bool valid = t < td.n_tiles;
  const int cnt = valid ? td.count[t] : 0;
  bool listed = cnt > 0;
  if (CLEAR && valid) {
    const int e = td.state[TS_EPOCH];
    const int last = td.epoch[t];
    listed = listed || last == e - 1;
    if (cnt > 0) td.epoch[t] = e;
  }
  int ptot, ltot;
  const int pex = block_scan(cnt, s_warp, &ptot);
  const int lex = block_scan(listed ? 1 : 0, s_warp, &ltot);
  if (threadIdx.x == 0) {
    s_pbase = ptot ? atomicAdd(td.state + TS_PAIRS, ptot) : 0;
    s_lbase = ltot ? atomicAdd(td.state + TS_LEN, ltot) : 0;
  }
  __syncthreads();
  if (listed) {
    td.active[0][s_lbase + lex] = t;
    td.off[t] = s_pbase + pex;
    td.cur[t] = s_pbase + pex;
  }
}

// every marker with a record writes its id into the lists of its tiles (the
// same tiles, from the same record, as the marker kernel counted)
__global__ void __launch_bounds__(256) tile_fill_kernel(DeviceTables T, TileDev td, Grid g,
                                                        int32_t F) {
  const int f = blockIdx.x * blockDim.x + threadIdx.x;
  if (f >= F) return;
  const float4 r0 = td.rec[2 * (size_t)f];
  const int b = __float_as_int(r0.w);
  if (b < 0) return;
  const int G0 = __ldg(&T.body[b].G[0]), G1 = __ldg(&T.body[b].G[1]), G2 = __ldg(&T.body[b].G[2]);
  int tx[3], ty[3], tz[3];
  const int nx_ = tiles_along(G0 + (int)floorf(r0.x), g.n[0], kTX, tx);
  const int ny_ = tiles_along(G1 + (int)floorf(r0.y), g.n[1], kTY, ty);
  const int nz_ = tiles_along(G2 + (int)floorf(r0.z), g.n[2], kTZ, tz);
  // the faces of a warp lie close together: one atomic per distinct tile among
  // its lanes, the lanes taking consecutive slots
#pragma unroll 1
  for (int a = 0; a < nz_; ++a)
#pragma unroll 1
    for (int c = 0; c < ny_; ++c)
#pragma unroll 1
      for (int d = 0; d < nx_; ++d) {
        const int t = (tz[a] * td.nt[1] + ty[c]) * td.nt[0] + tx[d];
        const unsigned peers = __match_any_sync(__activemask(), t);
        const int lane = threadIdx.x & 31, lead = __ffs(peers) - 1;
        int base = 0;
        if (lane == lead) base = atomicAdd(td.cur + t, __popc(peers));
        base = __shfl_sync(peers, base, lead);
        td.mlist[base + __popc(peers & ((1u << lane) - 1u))] = f;
      }
}

// One block per listed tile and component (a persistent grid walks the list).
// A thread per listed marker adds c_l phi F to its 27 nodes in exact fixed
// point: q = c_l phi F 2^k, its float value rounded to an integer, split into
// hi = floor(q / 2^16) and lo = q - 2^16 hi in [0, 2^16], each summed with a
// 32-bit shared atomic (lo as unsigned).  With n markers listed and
// |q| <= min(2^38, 2^45 / n_pow2) the hi sums stay below 2^30 and the lo sums
// below 2^32 for n < 2^16; the node's value 2^16 sum(hi) + sum(lo) is exact
// and does not depend on the order.  2^k comes from the tile's largest |c_l F|
// (recorded by the marker kernel) and the bound on |phi|.
//
// The accumulators have two more nodes on every side, so a support that meets
// the tile is added whole, without a test per node; what falls outside is
// another tile's and is dropped.  Only where the period is at most one node
// longer than the tile can such a node be this tile's again: it is then folded
// back.  A component per block keeps the accumulators at 23 KB (eight blocks
// of 128 threads per SM); tiles list about 100 markers.  170 -> 128 us for 320 k
// markers on 256^3 (before: a tile's three components in one block of 256,
// every node tested against the tile and its segment flagged).  Two shared
// atomics per node and the store of a tile's 1024 nodes are what is left.
constexpr int kPX = kTX + 4, kPY = kTY + 4, kPZ = kTZ + 4;
constexpr int kPadNodes = kPX * kPY * kPZ;
template <bool CLEAR>
__global__ void __launch_bounds__(kTileThreads, 8) tile_spread_kernel(
    DeviceTables T, TileDev td, Grid g, MlsK K, float phi_bound, float* __restrict__ fx,
    float* __restrict__ fy, float* __restrict__ fz) {
  __shared__ __align__(16) int s_hi[kPadNodes];
  __shared__ __align__(16) unsigned s_lo[kPadNodes];
  __shared__ uint32_t s_prev[4], s_new[4];
  __shared__ unsigned s_tmax;
  __shared__ int s_m0, s_m1;
  const int lane = threadIdx.x & 31;
  const int L = 3 * td.state[TS_LEN];
  for (int item = blockIdx.x; item < L; item += gridDim.x) {
    const int t = td.active[0][item / 3], i = item % 3;
    const int tx = t % td.nt[0], ty = (t / td.nt[0]) % td.nt[1], tz = t / (td.nt[0] * td.nt[1]);
    const int X0 = tx * kTX, Y0 = ty * kTY, Z0 = tz * kTZ;
    const int ex = min(kTX, g.n[0] - X0), ey = min(kTY, g.n[1] - Y0), ez = min(kTZ, g.n[2] - Z0);
    for (int q = threadIdx.x; q < kPadNodes / 4; q += kTileThreads) {
      reinterpret_cast<int4*>(s_hi)[q] = make_int4(0, 0, 0, 0);
      reinterpret_cast<int4*>(s_lo)[q] = make_int4(0, 0, 0, 0);
    }
    if (threadIdx.x < 4) {
      s_prev[threadIdx.x] = CLEAR ? td.mask[12 * (size_t)t + 4 * i + threadIdx.x] : 0u;
      s_new[threadIdx.x] = 0u;
    }
    if (threadIdx.x == 0) {
      s_m0 = td.off[t];
      s_m1 = td.cur[t];
      if (i == 0) td.count[t] = 0;   // ready for the next call
      s_tmax = td.tmax[4 * (size_t)t + i];
      td.tmax[4 * (size_t)t + i] = 0u;
    }
    __syncthreads();
    const int m0 = s_m0, n = s_m1 - s_m0;
    // scale 2^k with phi_bound * max|c_l F| * 2^k <= qcap
    int np2 = 1;
    while (np2 < n && np2 < (1 << 20)) np2 <<= 1;
    const float qcap = fminf(0x1p38f, __int_as_float((127 + 45) << 23) / (float)np2);
    const float bm = __uint_as_float(s_tmax) * phi_bound;
    float scale = 0.f, inv_scale = 0.f;
    if (bm > 0.f && bm <= 3.0e38f) {
      const int k = max(min(ilogbf(qcap) - (ilogbf(bm) + 1), 120), -120);
      scale = pow2f(k);
      inv_scale = pow2f(-k);
    }
    if (threadIdx.x == 0 && n >= 65536) atomicOr(T.err, ERR_TILE_DENSE);
    for (int q = threadIdx.x; q < n; q += kTileThreads) {
      const int m = td.mlist[m0 + q];
      const float4 r0 = td.rec[2 * (size_t)m];
      const float coef = __ldg(reinterpret_cast<const float*>(td.rec + 2 * (size_t)m + 1) + i) * scale;
      if (coef == 0.f) continue;
      const BodyDev* B = T.body + __float_as_int(r0.w);
      const float tc[3] = {r0.x, r0.y, r0.z};
      const int T0[3] = {X0, Y0, Z0}, EX[3] = {ex, ey, ez};
      float uf[3];
      int l0[3];   // the support's first node, from the padded corner
      bool reach = true;
#pragma unroll
      for (int d = 0; d < 3; ++d) {
        const float uu = tc[d] - (d == i ? 0.f : 0.5f);
        const float cc = floorf(uu + 0.5f);
        uf[d] = uu - cc;
        l0[d] = wrap_any(__ldg(&B->G[d]) + (int)cc - 1 - T0[d] + 2, g.n[d]);
        reach = reach && l0[d] < EX[d] + 2;
      }
      if (!reach) continue;
      DirW X, Y, Z;
      dir_weights(uf[0], K, X);
      dir_weights(uf[1], K, Y);
      dir_weights(uf[2], K, Z);
      const float xb1 = -(X.b0 + X.b2);
      const float ya[3] = {Y.a0, Y.a1, Y.a2}, yb[3] = {Y.b0, -(Y.b0 + Y.b2), Y.b2};
      const float za[3] = {Z.a0 * coef, Z.a1 * coef, Z.a2 * coef};
      const float zb[3] = {Z.b0 * coef, -(Z.b0 + Z.b2) * coef, Z.b2 * coef};
      const int at = (l0[2] * kPY + l0[1]) * kPX + l0[0];
      auto add = [&](int node, float val) {
        val = rintf(val);
        const float hf = floorf(val * (1.f / 65536.f));
        atomicAdd(s_hi + node, (int)hf);
        atomicAdd(s_lo + node, (unsigned)fmaf(-hf, 65536.f, val));
      };
#pragma unroll
      for (int sz = 0; sz < 3; ++sz) {
#pragma unroll
        for (int sy = 0; sy < 3; ++sy) {
          const int r = at + (sz * kPY + sy) * kPX;
          const float t0 = ya[sy] * za[sz], t1 = fmaf(yb[sy], za[sz], ya[sy] * zb[sz]);
          const float d = t0 - t1;
          add(r, fmaf(X.a0, d, -X.b0 * t0));
          add(r + 1, fmaf(X.a1, d, -xb1 * t0));
          add(r + 2, fmaf(X.a2, d, -X.b2 * t0));
        }
      }
    }
    __syncthreads();
    if (g.n[0] - ex < 2 || g.n[1] - ey < 2 || g.n[2] - ez < 2) {
      // nodes beyond the tile that are its own again, one period on
      for (int q = threadIdx.x; q < kPadNodes; q += kTileThreads) {
        const int px = q % kPX - 2, py = (q / kPX) % kPY - 2, pz = q / (kPX * kPY) - 2;
        const int x = wrap_any(px, g.n[0]), y = wrap_any(py, g.n[1]), z = wrap_any(pz, g.n[2]);
        if ((x != px || y != py || z != pz) && x < ex && y < ey && z < ez &&
            (s_hi[q] != 0 || s_lo[q] != 0u)) {
          const int to = ((z + 2) * kPY + y + 2) * kPX + x + 2;
          atomicAdd(s_hi + to, s_hi[q]);
          atomicAdd(s_lo + to, s_lo[q]);
        }
      }
      __syncthreads();
    }
    // segments of 8 nodes, 8 lanes each: stored when they received something or
    // (clear mode) were left nonzero by the last call
    float* fc = i == 0 ? fx : (i == 1 ? fy : fz);
    for (int q = threadIdx.x; q < kTileNodes; q += kTileThreads) {
      const int x = q % kTX, y = (q / kTX) % kTY, z = q / (kTX * kTY), sg = q >> 3;
      const int node = ((z + 2) * kPY + y + 2) * kPX + x + 2;
      const int hi = s_hi[node];
      const unsigned lo = s_lo[node];
      const unsigned got = __ballot_sync(0xffffffffu, (hi | (int)lo) != 0);
      const bool old = CLEAR && ((s_prev[sg >> 5] >> (sg & 31)) & 1u);
      if (!((got >> (lane & ~7)) & 0xffu) && !old) continue;   // whole segments
      const long long S = (long long)hi * 65536ll + (long long)lo;
      const float val =
          fmaf((float)(int)(S >> 32), 4294967296.f, (float)(unsigned)(S & 0xffffffffll)) * inv_scale;
      const bool inside = x < ex && y < ey && z < ez;
      const size_t idx = ((size_t)(Z0 + z) * g.n[1] + (Y0 + y)) * g.n[0] + (X0 + x);
      if (CLEAR) {
        if (inside) fc[idx] = val;
        if (val != 0.f) atomicOr(&s_new[sg >> 5], 1u << (sg & 31));
      } else if (inside && val != 0.f) {
        fc[idx] += val;
      }
    }
    __syncthreads();
    if (CLEAR && threadIdx.x < 4) td.mask[12 * (size_t)t + 4 * i + threadIdx.x] = s_new[threadIdx.x];
  }
}

}  // namespace

cudaError_t tile_spread_occupancy(int* blocks_per_sm) {
  return cudaOccupancyMaxActiveBlocksPerMultiprocessor(blocks_per_sm, tile_spread_kernel<true>,
                                                       kTileThreads, 0);
}

cudaError_t launch_tile_begin(ibm_ctx* c, bool accumulate, bool zero_sums) {
  const int nq = zero_sums ? 2 * (int)c->B : 0;
  const int blocks = (nq + 255) / 256 > 0 ? (nq + 255) / 256 : 1;
  tile_begin_kernel<<<blocks, 256, 0, c->stream>>>(c->td, zero_sums ? c->d.qsum : nullptr, nq,
                                                   accumulate ? 1 : 0);
  return cudaGetLastError();
}

cudaError_t launch_tile_spread(ibm_ctx* c, float* fx, float* fy, float* fz, bool accumulate) {
  if (c->F == 0) return cudaSuccess;
  const unsigned nb = (unsigned)((c->td.n_tiles + 1023) / 1024);
  if (accumulate)
    tile_scan_kernel<false><<<nb, 1024, 0, c->stream>>>(c->td);
  else
    tile_scan_kernel<true><<<nb, 1024, 0, c->stream>>>(c->td);
  cudaError_t e = cudaGetLastError();
  if (e != cudaSuccess) return e;
  tile_fill_kernel<<<(unsigned)((c->F + 255) / 256), 256, 0, c->stream>>>(c->d, c->td, c->grid,
                                                                         (int32_t)c->F);
  e = cudaGetLastError();
  if (e != cudaSuccess) return e;
  if (accumulate)
    tile_spread_kernel<false><<<c->tile_grid, kTileThreads, 0, c->stream>>>(
        c->d, c->td, c->grid, c->sc.mk, c->phi_bound, fx, fy, fz);
  else
    tile_spread_kernel<true><<<c->tile_grid, kTileThreads, 0, c->stream>>>(
        c->d, c->td, c->grid, c->sc.mk, c->phi_bound, fx, fy, fz);
  return cudaGetLastError();
}

}  // namespace ibm
