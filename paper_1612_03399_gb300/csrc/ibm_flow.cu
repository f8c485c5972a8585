// The fluid phase (Sec. 2.1): incompressible Navier-Stokes on the triply
// periodic MAC grid with the three-substep RK3 fractional step.
//
// Per substep l:
//   rhs_kernel      H(u) (divergence form), and R = dt (gamma_l H + rho_l H_prev
//                   - alpha_l grad p + alpha_l nu lap u) for the three
//                   components, one thread per cell computing the u, v and w
//                   nodes of that cell index
//   the factorised Crank-Nicolson solve: the operator
//                   (1 - a d_xx)(1 - a d_yy)(1 - a d_zz), a = alpha_l dt nu / 2,
//                   is inverted in one of three exact ways, picked per substep
//                   at creation:
//     cn_solve_kernel  by short filters: with c = a/h_d^2 the inverse of the
//                   periodic 1-D factor 1 - c (E - 2 + E^-1) is a circulant
//                   whose entries fall off as r^|m|, r < 1 the smaller root
//                   of c r^2 - (1 + 2c) r + c; when its mass beyond |m| = W
//                   (W <= 8) is below 2^-26 in every direction, the three
//                   inverses are applied as separable (2W+1)-tap filters and
//                   u* = u + du is written in the same pass
//     line_x_kernel, line_yz_kernel  by recursions along the lines, for r <= 0.7
//     R2C (batch 3) -> cn_scale_kernel -> C2R, add_kernel (u* = u + du):
//                   otherwise, the operator being diagonal in Fourier space
//   div_kernel      div(u* + s f)
//   (x, y) R2C -> poisson_z_kernel -> C2R: lap(phi) = div / (alpha_l dt), the z
//                   direction by recursions; long or thin domains: R2C ->
//                   poisson_scale_kernel -> C2R in all three
//   project_kernel  u = u* + s f - alpha_l dt grad(phi),
//                   p <- p + phi - a lap(phi)
// The eigenvalues of the periodic second difference, -(4/h^2) sin^2(pi k/n),
// are tabulated per direction in float64 on the host and stored as float.
#include <cuda_runtime.h>
#include <cufft.h>

#include <algorithm>
#include <cmath>
#include <string>
#include <vector>

#include "ibm.h"
#include "ibm_internal.cuh"

struct ibm_flow {
  int device = 0;
  cudaStream_t stream = nullptr;
  int n[3] = {0, 0, 0};
  double L[3] = {0, 0, 0}, h[3] = {0, 0, 0};
  double nu = 0, dt = 0;
  size_t N = 0, NC = 0;         // cells; complex coefficients of one field
  float* H[2] = {nullptr, nullptr};   // [3][N] nonlinear terms, ping-pong
  int hcur = 0;                 // H[hcur] holds the last predictor's H(u)
  int last = -1;                // last predicted substep of the current step
  float* R = nullptr;           // [3][N] right-hand sides, then increments
  float* rp = nullptr;          // [N] divergence, then phi
  cufftComplex* S = nullptr;    // [3][NC] spectra
  float* lam = nullptr;         // [n_x/2 + 1 | n_y | n_z] eigenvalues
  cufftHandle r2c3 = 0, c2r3 = 0, r2c1 = 0, c2r1 = 0;
  bool plans = false;
  // per substep: the real-space solve's half width W (-1: Fourier path) and
  // its taps g[d][|m|] per direction, m = 0..W
  int solve_w[3] = {-1, -1, -1};
  float taps[3][3][9] = {};
  bool z_lines = false;         // the Poisson solve's z direction by recursions,
  float4* zcol = nullptr;       // with their constants per column [ny][nx/2 + 1]
  int rhs_planes = 16;          // planes per thread of the right-hand side kernel
  int solve_planes[3] = {32, 32, 32};   // output planes per block of the real-space solves
  // per substep: solved by recursions along the lines; the powers of r they use
  bool lines[3] = {false, false, false};
  float* pw = nullptr;          // [3][pw_stride]
  size_t pw_stride = 0;
  // phase timing (profiling aid): events at the 12 kernel boundaries of each
  // substep and the 3 of the body update
  bool timing = false;
  cudaEvent_t ev[3][12] = {};
  cudaEvent_t evs[3] = {};
  bool have_sub[3] = {false, false, false};
  bool have_struct = false;
};

namespace ibm {
namespace {

constexpr double kGamma[3] = {8.0 / 15.0, 5.0 / 12.0, 3.0 / 4.0};
constexpr double kRho[3] = {0.0, -17.0 / 60.0, -5.0 / 12.0};

struct FGrid {
  int nx, ny, nz;
  float ih[3], ih2[3];   // 1/h, 1/h^2
};

struct Vec3 {
  float* c[3];
};
struct CVec3 {
  const float* c[3];
};

// offsets of the six periodic neighbours of cell (i, j, k) relative to its
// index (grids below 2^31 cells, checked at creation): one 64-bit base per
// thread and 32-bit offsets instead of a full index per load
struct Nbr {
  int xp, xm, yp, ym, zp, zm;
  __device__ __forceinline__ Nbr(int i, int j, int k, int nx, int ny, int nz) {
    const int sxy = nx * ny;
    xp = i == nx - 1 ? 1 - nx : 1;
    xm = i == 0 ? nx - 1 : -1;
    yp = j == ny - 1 ? (1 - ny) * nx : nx;
    ym = j == 0 ? (ny - 1) * nx : -nx;
    zp = k == nz - 1 ? (1 - nz) * sxy : sxy;
    zm = k == 0 ? (nz - 1) * sxy : -sxy;
  }
};

// H(u) and the predictor's right-hand side at the u, v and w nodes of cell
// index (i, j, k).  Products for the d-derivative of component c are formed
// where the difference needs them: at the cell centres for d = c (mean of the
// two neighbouring c nodes, squared), at the (c, d) edges otherwise (mean of
// u_d along c times mean of u_c along d).
__global__ void __launch_bounds__(256) rhs_kernel(FGrid G, const float* __restrict__ u,
                                                  const float* __restrict__ v,
                                                  const float* __restrict__ w,
                                                  const float* __restrict__ p, CVec3 Hp, Vec3 Ho,
                                                  Vec3 Ro, float gam, float rho, float alpha,
                                                  float nu, float dt) {
  const int i = blockIdx.x * blockDim.x + threadIdx.x;
  const int j = blockIdx.y * blockDim.y + threadIdx.y;
  const int k = blockIdx.z;
  if (i >= G.nx || j >= G.ny) return;
  const Nbr d(i, j, k, G.nx, G.ny, G.nz);
  const size_t o = ((size_t)k * G.ny + j) * G.nx + i;
  const float* up = u + o;
  const float* vp = v + o;
  const float* wp = w + o;
  const float* pp = p + o;
  const float U = __ldg(up), Uip = __ldg(up + d.xp), Uim = __ldg(up + d.xm),
              Ujp = __ldg(up + d.yp), Ujm = __ldg(up + d.ym), Ukp = __ldg(up + d.zp),
              Ukm = __ldg(up + d.zm), Uip_jm = __ldg(up + (d.xp + d.ym)),
              Uip_km = __ldg(up + (d.xp + d.zm));
  const float V = __ldg(vp), Vip = __ldg(vp + d.xp), Vim = __ldg(vp + d.xm),
              Vjp = __ldg(vp + d.yp), Vjm = __ldg(vp + d.ym), Vkp = __ldg(vp + d.zp),
              Vkm = __ldg(vp + d.zm), Vim_jp = __ldg(vp + (d.xm + d.yp)),
              Vjp_km = __ldg(vp + (d.yp + d.zm));
  const float W = __ldg(wp), Wip = __ldg(wp + d.xp), Wim = __ldg(wp + d.xm),
              Wjp = __ldg(wp + d.yp), Wjm = __ldg(wp + d.ym), Wkp = __ldg(wp + d.zp),
              Wkm = __ldg(wp + d.zm), Wim_kp = __ldg(wp + (d.xm + d.zp)),
              Wjm_kp = __ldg(wp + (d.ym + d.zp));
  const float P = __ldg(pp), Pim = __ldg(pp + d.xm), Pjm = __ldg(pp + d.ym),
              Pkm = __ldg(pp + d.zm);
  float H[3];
  {  // u nodes
    const float cp = 0.5f * (U + Uip), cm = 0.5f * (Uim + U);
    const float xx = (cp * cp - cm * cm) * G.ih[0];
    const float yy = (0.5f * (Vjp + Vim_jp) * 0.5f * (Ujp + U) - 0.5f * (V + Vim) * 0.5f * (U + Ujm)) * G.ih[1];
    const float zz = (0.5f * (Wkp + Wim_kp) * 0.5f * (Ukp + U) - 0.5f * (W + Wim) * 0.5f * (U + Ukm)) * G.ih[2];
    H[0] = -(xx + yy + zz);
  }
  {  // v nodes
    const float xx = (0.5f * (Uip + Uip_jm) * 0.5f * (Vip + V) - 0.5f * (U + Ujm) * 0.5f * (V + Vim)) * G.ih[0];
    const float cp = 0.5f * (V + Vjp), cm = 0.5f * (Vjm + V);
    const float yy = (cp * cp - cm * cm) * G.ih[1];
    const float zz = (0.5f * (Wkp + Wjm_kp) * 0.5f * (Vkp + V) - 0.5f * (W + Wjm) * 0.5f * (V + Vkm)) * G.ih[2];
    H[1] = -(xx + yy + zz);
  }
  {  // w nodes
    const float xx = (0.5f * (Uip + Uip_km) * 0.5f * (Wip + W) - 0.5f * (U + Ukm) * 0.5f * (W + Wim)) * G.ih[0];
    const float yy = (0.5f * (Vjp + Vjp_km) * 0.5f * (Wjp + W) - 0.5f * (V + Vkm) * 0.5f * (W + Wjm)) * G.ih[1];
    const float cp = 0.5f * (W + Wkp), cm = 0.5f * (Wkm + W);
    const float zz = (cp * cp - cm * cm) * G.ih[2];
    H[2] = -(xx + yy + zz);
  }
  const float Gp[3] = {(P - Pim) * G.ih[0], (P - Pjm) * G.ih[1], (P - Pkm) * G.ih[2]};
  const float Lu[3] = {
      (Uip - 2.f * U + Uim) * G.ih2[0] + (Ujp - 2.f * U + Ujm) * G.ih2[1] + (Ukp - 2.f * U + Ukm) * G.ih2[2],
      (Vip - 2.f * V + Vim) * G.ih2[0] + (Vjp - 2.f * V + Vjm) * G.ih2[1] + (Vkp - 2.f * V + Vkm) * G.ih2[2],
      (Wip - 2.f * W + Wim) * G.ih2[0] + (Wjp - 2.f * W + Wjm) * G.ih2[1] + (Wkp - 2.f * W + Wkm) * G.ih2[2]};
#pragma unroll
  for (int c = 0; c < 3; ++c) {
    float r = gam * H[c] - alpha * Gp[c] + alpha * nu * Lu[c];
    if (Hp.c[c] != nullptr) r += rho * __ldg(Hp.c[c] + o);
    Ho.c[c][o] = H[c];
    Ro.c[c][o] = dt * r;
  }
}

// Spectra are [batch][nz][ny][nx/2+1]: one warp-wide row of x coefficients
// per threadIdx.y, rows (j, k) grid-strided over blockIdx.x, the batch in
// blockIdx.y (one division per row, none per coefficient).
constexpr int kRowThreads = 32, kRowsPerBlock = 8;

// times norm / prod_d (1 - a lam_d)
__global__ void __launch_bounds__(kRowThreads * kRowsPerBlock)
    cn_scale_kernel(cufftComplex* __restrict__ S, int nxh, int ny, int nz,
                    const float* __restrict__ lam, float a, float norm) {
  const float* lx = lam;
  const float* ly = lam + nxh;
  const float* lz = ly + ny;
  cufftComplex* Sb = S + (size_t)blockIdx.y * nz * ny * nxh;
  for (int r = blockIdx.x * kRowsPerBlock + threadIdx.y; r < ny * nz;
       r += gridDim.x * kRowsPerBlock) {
    const int k = r / ny, j = r - k * ny;
    const float dyz = norm / ((1.f - a * __ldg(ly + j)) * (1.f - a * __ldg(lz + k)));
    cufftComplex* row = Sb + (size_t)r * nxh;
    for (int i = threadIdx.x; i < nxh; i += kRowThreads) {
      const float s = dyz / (1.f - a * __ldg(lx + i));
      cufftComplex c = row[i];
      c.x *= s;
      c.y *= s;
      row[i] = c;
    }
  }
}

// spectrum of div / (alpha dt): times scale / (lam_x + lam_y + lam_z), mean 0
__global__ void __launch_bounds__(kRowThreads * kRowsPerBlock)
    poisson_scale_kernel(cufftComplex* __restrict__ S, int nxh, int ny, int nz,
                         const float* __restrict__ lam, float scale) {
  const float* lx = lam;
  const float* ly = lam + nxh;
  const float* lz = ly + ny;
  for (int r = blockIdx.x * kRowsPerBlock + threadIdx.y; r < ny * nz;
       r += gridDim.x * kRowsPerBlock) {
    const int k = r / ny, j = r - k * ny;
    const float lyz = __ldg(ly + j) + __ldg(lz + k);
    cufftComplex* row = S + (size_t)r * nxh;
    for (int i = threadIdx.x; i < nxh; i += kRowThreads) {
      const float l = __ldg(lx + i) + lyz;
      const float s = (r == 0 && i == 0) ? 0.f : scale / l;
      cufftComplex c = row[i];
      c.x *= s;
      c.y *= s;
      row[i] = c;
    }
  }
}

// The Poisson solve's z direction without transforms: after the (x, y) transforms
// each column (k_x, k_y) is a periodic tridiagonal system,
//   (2 + d - E - E^-1) phi = -h_z^2 f,  d = -h_z^2 (lam_x + lam_y) > 0,
// and 2 + d - E - E^-1 = (1 - r E^-1)(1 - r E)/r with, s = sqrt(d)/2 and
// t = sqrt(1 + s^2), r = 1/(s + t)^2: one recursion up the column and one down.
// Its constants come from a table in float64, each in the form that keeps it
// to rounding: rho = 1 - r = 2s/(s + t) for the recursions (r near 1 for the long
// waves), -h_z^2 r for the result (r near h_x^2/(8 h_z^2) for the short ones on
// cells stretched in z), r^k from exp(-2k asinh(s)).  A recursion adds the small
// f - rho y to y and carries what the addition loses, so a long wave's sum over a
// column does not gather rounding.  A thread holds a segment of at most kZSeg
// entries in registers and runs it twice, first from zero for its end, then from
// the value that enters it: the segments' ends combined, the column closing on
// itself (the sum over a turn / (1 - r^n)).
// Column (0, 0), d = 0, is summed twice in float64 by one warp; its mean is 0.
// What bounds it: HBM, 16 bytes per coefficient once; two z transforms with the
// scaling between them moved three times that: 256^3 65 -> 29 us,
// 200 x 180 x 144 29 -> 12.
constexpr int kZSeg = 16, kZMax = 512;   // entries of a segment, of a column (32 segments)

struct ZLine {   // y <- f + (1 - rho) y; c: what y is too large by
  float2 y = {0.f, 0.f}, c = {0.f, 0.f};
  __device__ __forceinline__ void add(float& v, float& e, float f, float rho) {
    const float inc = fmaf(-rho, v, f) - e, n = v + inc;
    e = (n - v) - inc;
    v = n;
  }
  __device__ __forceinline__ float2 step(float2 f, float rho) {
    add(y.x, c.x, f.x, rho);
    add(y.y, c.y, f.y, rho);
    return y;
  }
};
__device__ __forceinline__ float2 axpy2(float a, float2 x, float2 y) {
  return make_float2(fmaf(a, x.x, y.x), fmaf(a, x.y, y.y));
}

// per column (rho, -h_z^2 r, r^base, 1/(1 - r^n_z)), base the shorter segments' length
__global__ void poisson_z_table_kernel(float4* __restrict__ table, int nx, int ny, int nz, int base,
                                       double hx, double hy, double hz) {
  const int nxh = nx / 2 + 1, col = blockIdx.x * blockDim.x + threadIdx.x;
  if (col >= nxh * ny) return;
  const int j = col / nxh;
  const double kx = hz / hx * sinpi((double)(col - j * nxh) / nx), ky = hz / hy * sinpi((double)j / ny);
  const double s = sqrt(kx * kx + ky * ky), q = 1.0 / (s + sqrt(1.0 + s * s)), theta = 2.0 * asinh(s);
  table[col] = make_float4((float)(2.0 * s * q), (float)(-hz * hz * q * q), (float)exp(-theta * base),
                           col ? (float)(-1.0 / expm1(-theta * nz)) : 0.f);
}

__device__ __noinline__ void poisson_z_mean_column(cufftComplex* __restrict__ S, size_t M, int n,
                                                   double h2, double scale) {
  const int lane = threadIdx.x;
  const int i0 = (int)((long long)n * lane / 32), i1 = (int)((long long)n * (lane + 1) / 32);
  auto sum = [](double v) {
    for (int o = 16; o > 0; o >>= 1) v += __shfl_xor_sync(0xffffffffu, v, o);
    return v;
  };
  auto before = [lane](double v) {   // the sum over the lanes before this one
    double t = v;
    for (int o = 1; o < 32; o <<= 1) {
      const double w = __shfl_up_sync(0xffffffffu, t, o);
      if (lane >= o) t += w;
    }
    return t - v;
  };
  // phi_{k+1} - phi_k = c + g_k, g_k the sum of the mean-free f up to k, c such
  // that a turn adds up to nothing
  double a = 0.0;
  for (int i = i0; i < i1; ++i) a += S[i * M].x;
  const double mean = sum(a) / n;
  double g = before(a - mean * (i1 - i0)), t = 0.0;
  const double g0 = g;
  for (int i = i0; i < i1; ++i) t += (g += S[i * M].x - mean);
  const double c = -sum(t) / n;
  double p = before(t + c * (i1 - i0)), q = 0.0;
  const double p0 = p;
  g = g0;
  for (int i = i0; i < i1; ++i) {
    q += p;
    p += c + (g += S[i * M].x - mean);
  }
  const double pm = sum(q) / n;
  p = p0;
  g = g0;
  for (int i = i0; i < i1; ++i) {
    const double f = S[i * M].x - mean;
    S[i * M] = make_cuComplex((float)(h2 * scale * (p - pm)), 0.f);
    p += c + (g += f);
  }
}

// 32 columns per block, segment threadIdx.y (the first block: column (0, 0));
// scale: what the forward and inverse (x, y) transforms and the time step leave to
// divide by
__global__ void __launch_bounds__(32 * (kZMax / kZSeg))
    poisson_z_kernel(cufftComplex* __restrict__ S, int nxh, int ny, int nz,
                     const float4* __restrict__ table, double h2, double scale) {
  __shared__ float2 ends[2][kZMax / kZSeg][32];
  const int M = nxh * ny;
  if (blockIdx.x == 0) {
    if (threadIdx.y == 0) poisson_z_mean_column(S, (size_t)M, nz, h2, scale);
    return;
  }
  const int col = (int)(blockIdx.x - 1) * 32 + threadIdx.x, lane = threadIdx.x;
  const bool in = col > 0 && col < M;
  const int g = threadIdx.y, segs = blockDim.y, n = nz;
  // the first n mod segs segments are one longer
  const int base = n / segs, rem = n - base * segs;
  const int k0 = g * base + min(g, rem), len = base + (g < rem ? 1 : 0);
  float2* at = reinterpret_cast<float2*>(S) + (size_t)k0 * M + col;
  const float4 k = in ? __ldg(table + col) : make_float4(1.f, 0.f, 0.f, 0.f);
  float2 f[kZSeg];
#pragma unroll
  for (int i = 0; i < kZSeg; ++i)
    f[i] = in && i < len ? at[(size_t)i * M] : make_float2(0.f, 0.f);
  const float rho = k.x, turn = k.z, turn1 = fmaf(-turn, rho, turn), close = k.w;   // r^base, r^(base+1)
  auto across = [&](int h) { return h < rem ? turn1 : turn; };
  {
    ZLine a;
#pragma unroll
    for (int i = 0; i < kZSeg; ++i)
      if (i < len) a.step(f[i], rho);
    ends[0][g][lane] = a.y;
  }
  __syncthreads();
  {
    ZLine a;
    for (int h = 0; h < segs; ++h) a.y = axpy2(across(h), a.y, ends[0][h][lane]);
    a.y = make_float2(close * a.y.x, close * a.y.y);
    for (int h = 0; h < g; ++h) a.y = axpy2(across(h), a.y, ends[0][h][lane]);
#pragma unroll
    for (int i = 0; i < kZSeg; ++i)
      if (i < len) f[i] = a.step(f[i], rho);
  }
  {
    ZLine a;
#pragma unroll
    for (int i = kZSeg - 1; i >= 0; --i)
      if (i < len) a.step(f[i], rho);
    ends[1][g][lane] = a.y;
  }
  __syncthreads();
  ZLine a;
  for (int h = segs - 1; h >= 0; --h) a.y = axpy2(across(h), a.y, ends[1][h][lane]);
  a.y = make_float2(close * a.y.x, close * a.y.y);
  for (int h = segs - 1; h > g; --h) a.y = axpy2(across(h), a.y, ends[1][h][lane]);
  const float s = k.y * (float)scale;
#pragma unroll
  for (int i = kZSeg - 1; i >= 0; --i)
    if (i < len) {
      const float2 x = a.step(f[i], rho);
      if (in) at[(size_t)i * M] = make_float2(s * x.x, s * x.y);
    }
}

// u_c += du_c, du = [3][N]; the component in blockIdx.y
__global__ void add_kernel(Vec3 u, const float* __restrict__ du, size_t N) {
  const int c = blockIdx.y;
  float* uc = c == 0 ? u.c[0] : (c == 1 ? u.c[1] : u.c[2]);
  const float* dc = du + (size_t)c * N;
  for (size_t q = blockIdx.x * (size_t)blockDim.x + threadIdx.x; q < N;
       q += (size_t)gridDim.x * blockDim.x)
    uc[q] += __ldg(dc + q);
}

// div(u* + s f) at the cell centres
__global__ void __launch_bounds__(256) div_kernel(FGrid G, CVec3 u, CVec3 f, float s,
                                                  float* __restrict__ out) {
  const int i = blockIdx.x * blockDim.x + threadIdx.x;
  const int j = blockIdx.y * blockDim.y + threadIdx.y;
  const int k = blockIdx.z;
  if (i >= G.nx || j >= G.ny) return;
  const Nbr nb(i, j, k, G.nx, G.ny, G.nz);
  const size_t o = ((size_t)k * G.ny + j) * G.nx + i;
  const size_t oi = o + nb.xp, oj = o + nb.yp, ok = o + nb.zp;
  float d = (__ldg(u.c[0] + oi) - __ldg(u.c[0] + o)) * G.ih[0] +
            (__ldg(u.c[1] + oj) - __ldg(u.c[1] + o)) * G.ih[1] +
            (__ldg(u.c[2] + ok) - __ldg(u.c[2] + o)) * G.ih[2];
  if (f.c[0] != nullptr) {
    d += s * ((__ldg(f.c[0] + oi) - __ldg(f.c[0] + o)) * G.ih[0] +
              (__ldg(f.c[1] + oj) - __ldg(f.c[1] + o)) * G.ih[1] +
              (__ldg(f.c[2] + ok) - __ldg(f.c[2] + o)) * G.ih[2]);
  }
  out[o] = d;
}

// u = u* + s f - alpha dt grad(phi); p <- p + phi - a lap(phi)
__global__ void __launch_bounds__(256) project_kernel(FGrid G, Vec3 u, float* __restrict__ p,
                                                      const float* __restrict__ phi, CVec3 f,
                                                      float s, float adt, float a) {
  const int i = blockIdx.x * blockDim.x + threadIdx.x;
  const int j = blockIdx.y * blockDim.y + threadIdx.y;
  const int k = blockIdx.z;
  if (i >= G.nx || j >= G.ny) return;
  const Nbr nb(i, j, k, G.nx, G.ny, G.nz);
  const size_t o = ((size_t)k * G.ny + j) * G.nx + i;
  const float* fp = phi + o;
  const float F = __ldg(fp);
  const float Fim = __ldg(fp + nb.xm), Fip = __ldg(fp + nb.xp);
  const float Fjm = __ldg(fp + nb.ym), Fjp = __ldg(fp + nb.yp);
  const float Fkm = __ldg(fp + nb.zm), Fkp = __ldg(fp + nb.zp);
  const float g[3] = {(F - Fim) * G.ih[0], (F - Fjm) * G.ih[1], (F - Fkm) * G.ih[2]};
#pragma unroll
  for (int c = 0; c < 3; ++c) {
    float val = u.c[c][o] - adt * g[c];
    if (f.c[0] != nullptr) val += s * __ldg(f.c[c] + o);
    u.c[c][o] = val;
  }
  const float lap = (Fip - 2.f * F + Fim) * G.ih2[0] + (Fjp - 2.f * F + Fjm) * G.ih2[1] +
                    (Fkp - 2.f * F + Fkm) * G.ih2[2];
  p[o] += F - a * lap;
}

// ---- four cells in x per thread --------------------------------------------
// For grids of whole float4 rows (nx % 4 == 0, 16-byte aligned fields); the
// one-cell kernels above serve the rest.  A plane's quads are numbered through
// its rows, so ragged row lengths leave no idle threads.  Measured on 256^3
// (us; one cell per thread before): right-hand side 206 -> 156 (127 in substep
// 0), divergence 108 -> 69, projection 176 -> 115, at 5.6 .. 7.0 TB/s of what they
// cannot do without; on 200 x 180 x 144: 72 -> 52, 25 -> 10, 54 -> 29.
constexpr int kQuadThreads = 256;

struct Quad {          // offsets of a quad's neighbours relative to its first cell
  int o, xm, xp, yp, ym;   // in-plane offset; the cells before and after; the rows j +- 1
  __device__ __forceinline__ Quad(int q, int nx, int ny) {
    const int nx4 = nx >> 2, j = q / nx4, i = 4 * (q - j * nx4);
    o = j * nx + i;
    xm = i == 0 ? nx - 1 : -1;
    xp = i + 4 == nx ? 4 - nx : 4;
    yp = j == ny - 1 ? (1 - ny) * nx : nx;
    ym = j == 0 ? (ny - 1) * nx : -nx;
  }
};
__device__ __forceinline__ void ld4(float* d, const float* p) {
  const float4 t = __ldg(reinterpret_cast<const float4*>(p));
  d[0] = t.x;
  d[1] = t.y;
  d[2] = t.z;
  d[3] = t.w;
}
__device__ __forceinline__ void st4(float* p, const float* s) {
  *reinterpret_cast<float4*>(p) = make_float4(s[0], s[1], s[2], s[3]);
}

// H(u) and the predictor's right-hand side as rhs_kernel, a thread walking a
// column of quads over `planes` planes: of the plane above it loads each
// field once and keeps what the next step needs of this plane in registers,
// and the products on the (x, y), (x, z) and (y, z) edges serve both
// components they appear in.  11 float4 and 9 single loads per four cells
// instead of 34 loads per cell: rhs_kernel was bound by the issue of loads
// and index arithmetic (80 G cells/s whether its fields came from L2 or HBM).
template <bool PREV>
__global__ void __launch_bounds__(kQuadThreads, 2)
    rhs4_kernel(FGrid G, const float* __restrict__ u, const float* __restrict__ v,
                const float* __restrict__ w, const float* __restrict__ p,
                const float* __restrict__ Hp, float* __restrict__ Ho, float* __restrict__ Ro,
                float gam, float rho, float alpha, float nu, float dt, int planes) {
  const int q = blockIdx.x * kQuadThreads + threadIdx.x;
  const int plane = G.nx * G.ny;
  if (q >= plane / 4) return;
  const size_t N = (size_t)plane * G.nz;
  const Quad Q(q, G.nx, G.ny);
  const int k0 = blockIdx.y * planes, k1 = min(k0 + planes, G.nz);
  const int oym = Q.o + Q.ym, oyp = Q.o + Q.yp;
  // u, v, w of this plane with both x neighbours: index 1 is the quad's first cell
  float U[6], V[6], W[6], Ukm[5], Vkm[4], Vjpkm[4], Wkm[4], Wjm[4], Pkm[4];
  {
    const size_t c = (size_t)k0 * plane, m = (size_t)(k0 == 0 ? G.nz - 1 : k0 - 1) * plane;
    ld4(U + 1, u + c + Q.o);
    U[0] = __ldg(u + c + Q.o + Q.xm);
    U[5] = __ldg(u + c + Q.o + Q.xp);
    ld4(V + 1, v + c + Q.o);
    V[0] = __ldg(v + c + Q.o + Q.xm);
    V[5] = __ldg(v + c + Q.o + Q.xp);
    ld4(W + 1, w + c + Q.o);
    W[0] = __ldg(w + c + Q.o + Q.xm);
    W[5] = __ldg(w + c + Q.o + Q.xp);
    ld4(Ukm, u + m + Q.o);
    Ukm[4] = __ldg(u + m + Q.o + Q.xp);
    ld4(Vkm, v + m + Q.o);
    ld4(Vjpkm, v + m + oyp);
    ld4(Wkm, w + m + Q.o);
    ld4(Wjm, w + c + oym);
    ld4(Pkm, p + m + Q.o);
  }
#pragma unroll 1
  for (int k = k0; k < k1; ++k) {
    const size_t c = (size_t)k * plane, n = (size_t)(k + 1 == G.nz ? 0 : k + 1) * plane;
    float Un[6], Vn[6], Wn[6], Wjmn[4], Ujp[4], Ujm[5], Vjp[5], Vjm[4], Wjp[4], P[5], Pjm[4];
    ld4(Un + 1, u + n + Q.o);
    Un[0] = __ldg(u + n + Q.o + Q.xm);
    Un[5] = __ldg(u + n + Q.o + Q.xp);
    ld4(Vn + 1, v + n + Q.o);
    Vn[0] = __ldg(v + n + Q.o + Q.xm);
    Vn[5] = __ldg(v + n + Q.o + Q.xp);
    ld4(Wn + 1, w + n + Q.o);
    Wn[0] = __ldg(w + n + Q.o + Q.xm);
    Wn[5] = __ldg(w + n + Q.o + Q.xp);
    ld4(Wjmn, w + n + oym);
    ld4(Ujp, u + c + oyp);
    ld4(Ujm, u + c + oym);
    Ujm[4] = __ldg(u + c + oym + Q.xp);
    ld4(Vjp + 1, v + c + oyp);
    Vjp[0] = __ldg(v + c + oyp + Q.xm);
    ld4(Vjm, v + c + oym);
    ld4(Wjp, w + c + oyp);
    ld4(P + 1, p + c + Q.o);
    P[0] = __ldg(p + c + Q.o + Q.xm);
    ld4(Pjm, p + c + oym);
    float xy[5], xz[5], uu[5];   // four times the products at this quad's edges and centres
#pragma unroll
    for (int e = 0; e < 5; ++e) {
      const float vs = V[e] + V[e + 1], ws = W[e] + W[e + 1], us = U[e] + U[e + 1];
      xy[e] = (Ujm[e] + U[e + 1]) * vs;
      xz[e] = (Ukm[e] + U[e + 1]) * ws;
      uu[e] = us * us;
    }
    const float qx = 0.25f * G.ih[0], qy = 0.25f * G.ih[1], qz = 0.25f * G.ih[2];
    float H[4], R[4];
    auto put = [&](int comp, const float (&Hv)[4], const float (&Rv)[4]) {
      const size_t at = comp * N + c + Q.o;
      float r[4];
      float h4[4] = {0.f, 0.f, 0.f, 0.f};
      if (PREV) ld4(h4, Hp + at);
#pragma unroll
      for (int e = 0; e < 4; ++e) r[e] = dt * (PREV ? fmaf(rho, h4[e], Rv[e]) : Rv[e]);
      st4(Ho + at, Hv);
      st4(Ro + at, r);
    };
    const float an = alpha * nu;
    // u nodes
#pragma unroll
    for (int e = 0; e < 4; ++e) {
      const float C = U[e + 1];
      const float yy = (Ujp[e] + C) * (Vjp[e] + Vjp[e + 1]) - xy[e];
      const float zz = (Un[e + 1] + C) * (Wn[e] + Wn[e + 1]) - xz[e];
      H[e] = -(qx * (uu[e + 1] - uu[e]) + qy * yy + qz * zz);
      const float L = (U[e + 2] - 2.f * C + U[e]) * G.ih2[0] + (Ujp[e] - 2.f * C + Ujm[e]) * G.ih2[1] +
                      (Un[e + 1] - 2.f * C + Ukm[e]) * G.ih2[2];
      R[e] = gam * H[e] - alpha * ((P[e + 1] - P[e]) * G.ih[0]) + an * L;
    }
    put(0, H, R);
    // v nodes; the (y, z) edge products
    float yz[4], yzn[4];
#pragma unroll
    for (int e = 0; e < 4; ++e) {
      const float C = V[e + 1];
      yz[e] = (Vkm[e] + C) * (Wjm[e] + W[e + 1]);
      yzn[e] = (Vn[e + 1] + C) * (Wjmn[e] + Wn[e + 1]);
      const float sp = C + Vjp[e + 1], sm = Vjm[e] + C;
      H[e] = -(qx * (xy[e + 1] - xy[e]) + qy * (sp * sp - sm * sm) + qz * (yzn[e] - yz[e]));
      const float L = (V[e + 2] - 2.f * C + V[e]) * G.ih2[0] +
                      (Vjp[e + 1] - 2.f * C + Vjm[e]) * G.ih2[1] +
                      (Vn[e + 1] - 2.f * C + Vkm[e]) * G.ih2[2];
      R[e] = gam * H[e] - alpha * ((P[e + 1] - Pjm[e]) * G.ih[1]) + an * L;
    }
    put(1, H, R);
    // w nodes
#pragma unroll
    for (int e = 0; e < 4; ++e) {
      const float C = W[e + 1];
      const float yy = (Vjpkm[e] + Vjp[e + 1]) * (C + Wjp[e]) - yz[e];
      const float sp = C + Wn[e + 1], sm = Wkm[e] + C;
      H[e] = -(qx * (xz[e + 1] - xz[e]) + qy * yy + qz * (sp * sp - sm * sm));
      const float L = (W[e + 2] - 2.f * C + W[e]) * G.ih2[0] + (Wjp[e] - 2.f * C + Wjm[e]) * G.ih2[1] +
                      (Wn[e + 1] - 2.f * C + Wkm[e]) * G.ih2[2];
      R[e] = gam * H[e] - alpha * ((P[e + 1] - Pkm[e]) * G.ih[2]) + an * L;
    }
    put(2, H, R);
#pragma unroll
    for (int e = 0; e < 4; ++e) {
      Ukm[e] = U[e + 1];
      Vkm[e] = V[e + 1];
      Vjpkm[e] = Vjp[e + 1];
      Wkm[e] = W[e + 1];
      Wjm[e] = Wjmn[e];
      Pkm[e] = P[e + 1];
    }
    Ukm[4] = U[5];
#pragma unroll
    for (int e = 0; e < 6; ++e) {
      U[e] = Un[e];
      V[e] = Vn[e];
      W[e] = Wn[e];
    }
  }
}

// div(u* + s f) as div_kernel
template <bool FORCED>
__global__ void __launch_bounds__(kQuadThreads) div4_kernel(FGrid G, CVec3 u, CVec3 f, float s,
                                                            float* __restrict__ out) {
  const int q = blockIdx.x * kQuadThreads + threadIdx.x;
  const int plane = G.nx * G.ny;
  if (q >= plane / 4) return;
  const Quad Q(q, G.nx, G.ny);
  const int k = blockIdx.y;
  const size_t o = (size_t)k * plane + Q.o;
  const size_t on = (size_t)(k + 1 == G.nz ? 0 : k + 1) * plane + Q.o;
  float a[5], b[4], bp[4], c[4], cp[4], d[4];
  ld4(a, u.c[0] + o);
  a[4] = __ldg(u.c[0] + o + Q.xp);
  ld4(b, u.c[1] + o);
  ld4(bp, u.c[1] + o + Q.yp);
  ld4(c, u.c[2] + o);
  ld4(cp, u.c[2] + on);
  if (FORCED) {
    float fa[5], fb[4], fbp[4], fc[4], fcp[4];
    ld4(fa, f.c[0] + o);
    fa[4] = __ldg(f.c[0] + o + Q.xp);
    ld4(fb, f.c[1] + o);
    ld4(fbp, f.c[1] + o + Q.yp);
    ld4(fc, f.c[2] + o);
    ld4(fcp, f.c[2] + on);
#pragma unroll
    for (int e = 0; e < 4; ++e)
      d[e] = s * ((fa[e + 1] - fa[e]) * G.ih[0] + (fbp[e] - fb[e]) * G.ih[1] +
                  (fcp[e] - fc[e]) * G.ih[2]);
  }
#pragma unroll
  for (int e = 0; e < 4; ++e) {
    const float t = (a[e + 1] - a[e]) * G.ih[0] + (bp[e] - b[e]) * G.ih[1] + (cp[e] - c[e]) * G.ih[2];
    d[e] = FORCED ? t + d[e] : t;
  }
  st4(out + o, d);
}

// u = u* + s f - alpha dt grad(phi); p <- p + phi - a lap(phi), as project_kernel
template <bool FORCED>
__global__ void __launch_bounds__(kQuadThreads)
    project4_kernel(FGrid G, Vec3 u, float* __restrict__ p, const float* __restrict__ phi, CVec3 f,
                    float s, float adt, float a) {
  const int q = blockIdx.x * kQuadThreads + threadIdx.x;
  const int plane = G.nx * G.ny;
  if (q >= plane / 4) return;
  const Quad Q(q, G.nx, G.ny);
  const int k = blockIdx.y;
  const size_t o = (size_t)k * plane + Q.o;
  const size_t on = (size_t)(k + 1 == G.nz ? 0 : k + 1) * plane + Q.o;
  const size_t om = (size_t)(k == 0 ? G.nz - 1 : k - 1) * plane + Q.o;
  float F[6], Fjm[4], Fjp[4], Fkm[4], Fkp[4], val[4], fr[4];
  ld4(F + 1, phi + o);
  F[0] = __ldg(phi + o + Q.xm);
  F[5] = __ldg(phi + o + Q.xp);
  ld4(Fjm, phi + o + Q.ym);
  ld4(Fjp, phi + o + Q.yp);
  ld4(Fkm, phi + om);
  ld4(Fkp, phi + on);
#pragma unroll
  for (int c = 0; c < 3; ++c) {
    const float4 t = *reinterpret_cast<const float4*>(u.c[c] + o);
    const float us[4] = {t.x, t.y, t.z, t.w};
    if (FORCED) ld4(fr, f.c[c] + o);
#pragma unroll
    for (int e = 0; e < 4; ++e) {
      const float lo = c == 0 ? F[e] : (c == 1 ? Fjm[e] : Fkm[e]);
      val[e] = us[e] - adt * ((F[e + 1] - lo) * G.ih[c]);
      if (FORCED) val[e] += s * fr[e];
    }
    st4(u.c[c] + o, val);
  }
  const float4 t = *reinterpret_cast<const float4*>(p + o);
  const float ps[4] = {t.x, t.y, t.z, t.w};
#pragma unroll
  for (int e = 0; e < 4; ++e) {
    const float C = F[e + 1];
    const float lap = (F[e + 2] - 2.f * C + F[e]) * G.ih2[0] + (Fjp[e] - 2.f * C + Fjm[e]) * G.ih2[1] +
                      (Fkp[e] - 2.f * C + Fkm[e]) * G.ih2[2];
    val[e] = ps[e] + (C - a * lap);
  }
  st4(p + o, val);
}

// asynchronous 4- and 16-byte global -> shared copies
__device__ __forceinline__ void cp_async4(float* sdst, const float* gsrc) {
  const unsigned d = (unsigned)__cvta_generic_to_shared(sdst);
  asm volatile("cp.async.ca.shared.global [%0], [%1], 4;\n" ::"r"(d), "l"(gsrc) : "memory");
}
__device__ __forceinline__ void cp_async16(float* sdst, const float* gsrc) {
  const unsigned d = (unsigned)__cvta_generic_to_shared(sdst);
  asm volatile("cp.async.cg.shared.global [%0], [%1], 16;\n" ::"r"(d), "l"(gsrc) : "memory");
}
__device__ __forceinline__ void cp_async_commit() { asm volatile("cp.async.commit_group;\n" ::: "memory"); }
template <int N>
__device__ __forceinline__ void cp_async_wait() {
  asm volatile("cp.async.wait_group %0;\n" ::"n"(N) : "memory");
}

// The real-space factorised solve fused with u* = u + du.  A block owns a
// 32 x 32 tile of (x, y) outputs of one component over `planes` planes; it
// walks the planes + 2W that feed them (periodic wrap in every direction), each
// staged with its x and y halo by asynchronous copies two planes ahead.  Per
// plane the y filter, in packed two-lane float arithmetic, two rows of a quad of
// x per thread, into a second buffer; from there each thread filters its own
// quad in x and keeps the result in a register ring of 2W + 1 planes, whose z
// filter gives the output W planes back.  Taps are symmetric: g[d][|m|].
// What bounds it: instruction issue first (three filters of 2W + 1 taps; 95
// instructions an output with x filtered first, 4-byte copies and a ring that
// moved by one place a plane).  With y first, the ring's places fixed by
// unrolling the walk 2W + 1 times and V4 (rows of whole float4s: 16-byte copies,
// loads and stores; other rows and alignments go word by word) it is 38, and the
// shared-memory pipe (70 %) and the barrier a plane remain.  256^3, 600 MB in
// 90 us at the copy rate: W = 3 172 -> 130 us, W = 4 208 -> 136; 200 x 180 x 144,
// W = 7: 144 -> 90; 64^3: 26 -> 8; word by word on 255 x 256 x 256 186 -> 161 and
// 222 -> 178.
constexpr int kSolveT = 32, kMaxSolveW = 8;

struct SolveTaps {
  float g[3][kMaxSolveW + 1];
};
static_assert(sizeof(ibm_flow::taps[0]) == sizeof(SolveTaps), "tap table layout");

__device__ __forceinline__ float2 f2(float a) { return make_float2(a, a); }

__host__ __device__ constexpr int solve_halo(int W) { return W <= 4 ? 4 : 8; }   // staged columns beside the tile
__host__ __device__ constexpr int solve_blocks(int W) { return W <= 4 ? 3 : 2; } // resident blocks per SM
constexpr size_t solve_smem(int W) {
  return sizeof(float) * (size_t)(kSolveT + 2 * solve_halo(W)) * (3 * (kSolveT + 2 * W) + 2 * kSolveT);
}

template <int W, bool V4>
__global__ void __launch_bounds__(256, solve_blocks(W)) cn_solve_kernel(
    FGrid G, const float* __restrict__ R, Vec3 u, SolveTaps T, int planes) {
  constexpr int HX = solve_halo(W), AX = kSolveT + 2 * HX, QX = AX / 4, AY = kSolveT + 2 * W;
  constexpr int NB = 3, RW = 2 * W + 1;
  constexpr int CX = V4 ? QX : kSolveT + 2 * W;      // staged per row: quads, or single columns
  constexpr int SLOTS = (AY * CX + 255) / 256;
  // A[NB][AY][AX] raw planes with halo, Y[2][32][AX] y-filtered rows
  extern __shared__ __align__(16) float smem[];
  float* const A = smem;
  float* const Y = smem + NB * AY * AX;
  const int tid = threadIdx.x;
  const int nx = G.nx, ny = G.ny, nz = G.nz;
  const int ntx = (nx + kSolveT - 1) / kSolveT;
  const int x0 = (int)(blockIdx.y % ntx) * kSolveT, y0 = (int)(blockIdx.y / ntx) * kSolveT;
  const int k0 = (int)blockIdx.x * planes;
  const int nk = min(planes, nz - k0), nq = nk + 2 * W;
  const size_t plane = (size_t)nx * ny;
  const int c = blockIdx.z;
  const float* Rc = R + (size_t)c * plane * nz;
  float* uc = c == 0 ? u.c[0] : (c == 1 ? u.c[1] : u.c[2]);
  // staging slots: wrapped in-plane offset (-1 past the tile)
  int off[SLOTS];
  short sdst[SLOTS];
#pragma unroll
  for (int s = 0; s < SLOTS; ++s) {
    const int q = tid + 256 * s;
    off[s] = -1;
    sdst[s] = 0;
    if (q < AY * CX) {
      const int r = q / CX, cc = q - r * CX;
      const int xr = V4 ? 4 * cc - HX : cc - W;      // whole quads: x0 and nx are multiples of 4
      const int xg = ((x0 + xr) % nx + nx) % nx, yg = ((y0 - W + r) % ny + ny) % ny;
      off[s] = yg * nx + xg;
      sdst[s] = (short)(r * AX + HX + xr);
    }
  }
  auto stage = [&](int q, int b) {
    int k = k0 - W + q;
    k = k < 0 ? k + nz : (k >= nz ? k - nz : k);
    const float* src = Rc + (size_t)k * plane;
    float* dst = A + b * (AY * AX);
#pragma unroll
    for (int s = 0; s < SLOTS; ++s) {
      if (off[s] < 0) continue;
      if (V4)
        cp_async16(dst + sdst[s], src + off[s]);
      else
        cp_async4(dst + sdst[s], src + off[s]);
    }
    cp_async_commit();
  };
  // y filter: a quad of x in two rows; the first 128 threads take eight quads of
  // a row pair each eight (no bank conflicts), the next the quads left over
  constexpr int QR = QX - 8;
  const int yr = 2 * (tid < 128 ? tid >> 3 : (tid - 128) / QR);
  const int yc = 4 * (tid < 128 ? tid & 7 : 8 + (tid - 128) % QR);
  auto yfilter = [&](int b, int t) {
    if (tid >= 16 * QX) return;
    const float* a = A + b * (AY * AX) + yr * AX + yc;
    float2 o[2][2];
#pragma unroll
    for (int i = 0; i < RW + 1; ++i) {
      const float4 v = *reinterpret_cast<const float4*>(a + i * AX);
      const float2 lo = make_float2(v.x, v.y), hi = make_float2(v.z, v.w);
#pragma unroll
      for (int j = 0; j < 2; ++j) {
        if (i - j < 0 || i - j >= RW) continue;
        const float2 g = f2(T.g[1][i - j < W ? W - i + j : i - j - W]);
        o[j][0] = i == j ? __fmul2_rn(g, lo) : __ffma2_rn(g, lo, o[j][0]);
        o[j][1] = i == j ? __fmul2_rn(g, hi) : __ffma2_rn(g, hi, o[j][1]);
      }
    }
#pragma unroll
    for (int j = 0; j < 2; ++j)
      *reinterpret_cast<float4*>(Y + (t * kSolveT + yr + j) * AX + yc) =
          make_float4(o[j][0].x, o[j][0].y, o[j][1].x, o[j][1].y);
  };
  // outputs: columns ox .. ox + 3 of row oy
  const int lx = 4 * (tid & 7), ly = tid >> 3;
  const int ox = x0 + lx, oy = y0 + ly;
  const bool mine = oy < ny && ox < nx;
  const size_t oo = (size_t)oy * nx + ox;
  float2 ring[RW][2];
#pragma unroll
  for (int m = 0; m < RW; ++m) ring[m][0] = ring[m][1] = make_float2(0.f, 0.f);

  // one barrier per plane: between two of them the x and z filters of plane q
  // and the y filter of plane q + 1
  stage(0, 0);
  if (nq > 1) {
    stage(1, 1);
    cp_async_wait<1>();
  } else {
    cp_async_wait<0>();
  }
  __syncthreads();
  if (nq > 2) stage(2, 2);
  yfilter(0, 0);
  int b = 0;   // the buffer of plane q
  // u of the output plane: V4 loads it a plane ahead (137 -> 130 us; without V4
  // the registers are better spent on the offsets)
  float un[4] = {0.f, 0.f, 0.f, 0.f};
  auto load_u = [&](int ko) {
    const float* ul = uc + (size_t)(k0 + ko) * plane + oo;
    if (V4) {
      const float4 t = *reinterpret_cast<const float4*>(ul);
      un[0] = t.x; un[1] = t.y; un[2] = t.z; un[3] = t.w;
    } else {
#pragma unroll
      for (int j = 0; j < 4; ++j)
        if (ox + j < nx) un[j] = ul[j];
    }
  };
  if (V4 && W == 0 && mine) load_u(0);
  for (int q0 = 0; q0 < nq; q0 += RW) {
#pragma unroll
    for (int s = 0; s < RW; ++s) {
      const int q = q0 + s;
      if (q >= nq) break;
      if (q + 2 < nq)
        cp_async_wait<1>();
      else
        cp_async_wait<0>();
      // Y[q & 1] complete and plane q + 1 visible; every thread is past the y
      // filter of plane q (its buffer is free) and the x filter of plane q - 1
      // (Y[(q + 1) & 1] is free)
      __syncthreads();
      const int ko = q - 2 * W;
      const float uu[4] = {un[0], un[1], un[2], un[3]};
      if (mine && (V4 ? ko >= -1 && q + 1 < nq : ko >= 0)) load_u(V4 ? ko + 1 : ko);
      if (q + 3 < nq) stage(q + 3, b);
      b = b == NB - 1 ? 0 : b + 1;
      if (q + 1 < nq) yfilter(b, (q + 1) & 1);
      // x filter of the thread's quad: even distances on aligned pairs
      {
        float win[4 + 2 * HX];
        const float* yq = Y + ((q & 1) * kSolveT + ly) * AX + lx;
#pragma unroll
        for (int v = 0; v < 1 + HX / 2; ++v) {
          const float4 t = *reinterpret_cast<const float4*>(yq + 4 * v);
          win[4 * v] = t.x;
          win[4 * v + 1] = t.y;
          win[4 * v + 2] = t.z;
          win[4 * v + 3] = t.w;
        }
        float2 o[2];
#pragma unroll
        for (int j = 0; j < 2; ++j) {
          const int w0 = HX + 2 * j;
          o[j] = __fmul2_rn(f2(T.g[0][0]), make_float2(win[w0], win[w0 + 1]));
#pragma unroll
          for (int m = 2; m <= W; m += 2) {
            o[j] = __ffma2_rn(f2(T.g[0][m]), make_float2(win[w0 - m], win[w0 - m + 1]), o[j]);
            o[j] = __ffma2_rn(f2(T.g[0][m]), make_float2(win[w0 + m], win[w0 + m + 1]), o[j]);
          }
#pragma unroll
          for (int m = 1; m <= W; m += 2) {
            o[j].x = fmaf(T.g[0][m], win[w0 - m], o[j].x);
            o[j].y = fmaf(T.g[0][m], win[w0 + 1 - m], o[j].y);
            o[j].x = fmaf(T.g[0][m], win[w0 + m], o[j].x);
            o[j].y = fmaf(T.g[0][m], win[w0 + 1 + m], o[j].y);
          }
          ring[s][j] = o[j];
        }
      }
      if (ko >= 0 && mine) {   // z filter: the newest plane is place s, the centre W before it
        float2 r[2];
#pragma unroll
        for (int j = 0; j < 2; ++j) {
          r[j] = V4 ? make_float2(uu[2 * j], uu[2 * j + 1]) : make_float2(un[2 * j], un[2 * j + 1]);
          float2 d = __fmul2_rn(f2(T.g[2][0]), ring[(s + RW - W) % RW][j]);
#pragma unroll
          for (int m = 1; m <= W; ++m)
            d = __ffma2_rn(f2(T.g[2][m]),
                           __fadd2_rn(ring[(s + RW - W - m) % RW][j], ring[(s + RW - W + m) % RW][j]),
                           d);
          r[j] = __fadd2_rn(r[j], d);
        }
        float* uo = uc + (size_t)(k0 + ko) * plane + oo;
        if (V4) {
          *reinterpret_cast<float4*>(uo) = make_float4(r[0].x, r[0].y, r[1].x, r[1].y);
        } else {
          const float o[4] = {r[0].x, r[0].y, r[1].x, r[1].y};
#pragma unroll
          for (int j = 0; j < 4; ++j)
            if (ox + j < nx) uo[j] = o[j];
        }
      }
    }
  }
}

// ---- the factorised solve by recursions along the lines ---------------------
// 1 - c (E - 2 + E^-1) = (c/r) (1 - r E^-1)(1 - r E), r < 1 the smaller root of
// c r^2 - (1 + 2c) r + c = 0, so its periodic inverse is a first-order recursion
// up every line and one down, times r/c.  A line is cut into kSegs segments that
// run from zero; the values that enter them follow from the segments' ends (the
// line closes on itself: the sum over a turn divided by 1 - r^n), and reach the
// i-th entry of a segment times r^(i+1).  Exact to rounding for any line; the
// sums grow by 1/(1 - r) at most before the scaling takes it back.
// A block holds 32 lines in shared memory, kSegs threads to a line; three passes
// (z, y, x) move 84 N bytes, the last adds to u.  Replaces the transforms where
// 17 taps are not enough: on 200 x 180 x 144 a substep's forward and inverse
// transforms of three fields, the scaling and the add took 324 us, the passes
// take 42 + 32 + 52 us; the error of u* against float64 is 0.6 of the transforms'
// (r = 0.35 .. 0.7).
constexpr int kSegs = 8;
constexpr int kMaxLine = 1600;          // entries of a line that fit shared memory

struct LineSolve {
  float r, q, close;   // r, r/c, 1 / (1 - r^n)
  const float* pw;     // r^k, k = 0 .. ceil(n / kSegs)
};

// one line per lane (stride `pitch` between its entries in s), segment threadIdx.y;
// `in(i)` gives entry i, `out(i, x)` takes the solution
template <class In, class Out>
__device__ __forceinline__ void solve_lines(float* s, int pitch, int n, const LineSolve& L,
                                            float (*ends)[2][32], In in, Out out) {
  const int lane = threadIdx.x, g = threadIdx.y;
  const int i0 = n * g / kSegs, len = n * (g + 1) / kSegs - i0;
  float* p = s + i0 * pitch;
  float y = 0.f;
#pragma unroll 4
  for (int i = 0; i < len; ++i) {
    y = fmaf(L.r, y, in(i0 + i));
    p[i * pitch] = y;
  }
  ends[g][0][lane] = y;
  __syncthreads();
  float c = 0.f;
#pragma unroll
  for (int h = 0; h < kSegs; ++h)
    c = fmaf(__ldg(L.pw + (n * (h + 1) / kSegs - n * h / kSegs)), c, ends[h][0][lane]);
  c *= L.close;                       // what enters entry 0 from the line's end
  for (int h = 0; h < g; ++h)
    c = fmaf(__ldg(L.pw + (n * (h + 1) / kSegs - n * h / kSegs)), c, ends[h][0][lane]);
  float x = 0.f;
#pragma unroll 4
  for (int i = len - 1; i >= 0; --i) {
    x = fmaf(L.r, x, L.q * fmaf(c, __ldg(L.pw + i + 1), p[i * pitch]));
    p[i * pitch] = x;
  }
  ends[g][1][lane] = x;
  __syncthreads();
  c = 0.f;
#pragma unroll
  for (int h = kSegs - 1; h >= 0; --h)
    c = fmaf(__ldg(L.pw + (n * (h + 1) / kSegs - n * h / kSegs)), c, ends[h][1][lane]);
  c *= L.close;
  for (int h = kSegs - 1; h > g; --h)
    c = fmaf(__ldg(L.pw + (n * (h + 1) / kSegs - n * h / kSegs)), c, ends[h][1][lane]);
#pragma unroll 4
  for (int i = 0; i < len; ++i) out(i0 + i, fmaf(c, __ldg(L.pw + len - i), p[i * pitch]));
}

// x lines, 32 rows per block: the last pass, added to u
__global__ void __launch_bounds__(32 * kSegs) line_x_kernel(FGrid G, const float* __restrict__ R,
                                                            Vec3 u, LineSolve L) {
  extern __shared__ __align__(16) float smem[];
  __shared__ float ends[kSegs][2][32];
  const int n = G.nx, pitch = n | 1;               // odd: no bank conflicts down the rows
  const int rows = G.ny * G.nz, r0 = 32 * blockIdx.x, nr = min(32, rows - r0);
  const float* f = R + ((size_t)blockIdx.y * rows + r0) * n;
  float* uc = (blockIdx.y == 0 ? u.c[0] : (blockIdx.y == 1 ? u.c[1] : u.c[2])) + (size_t)r0 * n;
  for (int k = threadIdx.y; k < nr; k += kSegs)
    for (int i = threadIdx.x; i < n; i += 32) smem[k * pitch + i] = f[k * n + i];
  __syncthreads();
  float* s = smem + threadIdx.x * pitch;
  solve_lines(s, 1, n, L, ends, [&](int i) { return s[i]; }, [&](int i, float x) { s[i] = x; });
  __syncthreads();
  for (int k = threadIdx.y; k < nr; k += kSegs)
    for (int i = threadIdx.x; i < n; i += 32) uc[k * n + i] += smem[k * pitch + i];
}

// y or z lines, in place in R: 32 neighbouring x per block, the other direction
// in blockIdx.y, the component in blockIdx.z
template <bool Z>
__global__ void __launch_bounds__(32 * kSegs) line_yz_kernel(FGrid G, float* __restrict__ R,
                                                             LineSolve L) {
  extern __shared__ __align__(16) float smem[];
  __shared__ float ends[kSegs][2][32];
  const size_t plane = (size_t)G.nx * G.ny, stride = Z ? plane : (size_t)G.nx;
  const int n = Z ? G.nz : G.ny, x = 32 * blockIdx.x + threadIdx.x;
  const bool in_row = x < G.nx;
  float* f = R + blockIdx.z * plane * G.nz + blockIdx.y * (Z ? (size_t)G.nx : plane) + x;
  solve_lines(
      smem + threadIdx.x, 32, n, L, ends,
      [&](int i) { return in_row ? f[i * stride] : 0.f; },
      [&](int i, float v) {
        if (in_row) f[i * stride] = v;
      });
}

FGrid fgrid(const ibm_flow* fl);

// every given field 16-byte aligned (null: not used) and rows of whole float4s
template <class... P>
bool quads(const ibm_flow* fl, P... f) {
  const uintptr_t bits = (reinterpret_cast<uintptr_t>(f) | ...);
  return fl->n[0] % 4 == 0 && (bits & 15u) == 0;
}
cudaError_t launch_cn_solve(const ibm_flow* fl, int l, float* u, float* v, float* w,
                            cudaStream_t s) {
  const FGrid G = fgrid(fl);
  SolveTaps T;
  for (int d = 0; d < 3; ++d)
    for (int m = 0; m <= kMaxSolveW; ++m) T.g[d][m] = fl->taps[l][d][m];
  const int planes = fl->solve_planes[l];
  const unsigned tiles = (unsigned)(((fl->n[0] + kSolveT - 1) / kSolveT) *
                                    ((fl->n[1] + kSolveT - 1) / kSolveT));
  const dim3 grid((unsigned)((fl->n[2] + planes - 1) / planes), tiles, 3), block(256);
  const Vec3 U{{u, v, w}};
  const bool v4 = quads(fl, u, v, w);
  switch (fl->solve_w[l]) {
#define IBM_SOLVE_CASE(WW)                                                            \
  case WW:                                                                            \
    (v4 ? cn_solve_kernel<WW, true> : cn_solve_kernel<WW, false>)<<<grid, block, solve_smem(WW), s>>>( \
        G, fl->R, U, T, planes);                                                      \
    break;
    IBM_SOLVE_CASE(0) IBM_SOLVE_CASE(1) IBM_SOLVE_CASE(2) IBM_SOLVE_CASE(3) IBM_SOLVE_CASE(4)
    IBM_SOLVE_CASE(5) IBM_SOLVE_CASE(6) IBM_SOLVE_CASE(7) IBM_SOLVE_CASE(8)
#undef IBM_SOLVE_CASE
    default: return cudaErrorInvalidValue;
  }
  return cudaGetLastError();
}

// The recursions' constants for c = a / h^2, and the powers of r a segment needs.
double line_root(double c) { return 2.0 * c / (1.0 + 2.0 * c + std::sqrt(1.0 + 4.0 * c)); }
LineSolve line_solve(double c, int n, const float* pw) {
  const double r = line_root(c);
  return {(float)r, (float)(2.0 / (1.0 + 2.0 * c + std::sqrt(1.0 + 4.0 * c))),
          (float)(1.0 / (1.0 - std::pow(r, n))), pw};
}
int line_powers(int n) { return (n + kSegs - 1) / kSegs + 2; }

cudaError_t launch_lines(const ibm_flow* fl, int l, float* u, float* v, float* w, cudaStream_t s) {
  const FGrid G = fgrid(fl);
  const double a = (kGamma[l] + kRho[l]) * fl->dt * fl->nu / 2.0;
  LineSolve L[3];
  const float* pw = fl->pw + (size_t)l * fl->pw_stride;
  for (int d = 0; d < 3; ++d) {
    L[d] = line_solve(a / (fl->h[d] * fl->h[d]), fl->n[d], pw);
    pw += line_powers(fl->n[d]);
  }
  const dim3 block(32, kSegs);
  const unsigned nx32 = (unsigned)((G.nx + 31) / 32);
  const int rows = G.ny * G.nz;
  line_yz_kernel<true><<<dim3(nx32, (unsigned)G.ny, 3), block, 32 * sizeof(float) * G.nz, s>>>(
      G, fl->R, L[2]);
  line_yz_kernel<false><<<dim3(nx32, (unsigned)G.nz, 3), block, 32 * sizeof(float) * G.ny, s>>>(
      G, fl->R, L[1]);
  line_x_kernel<<<dim3((unsigned)((rows + 31) / 32), 3), block, 32 * sizeof(float) * (G.nx | 1), s>>>(
      G, fl->R, Vec3{{u, v, w}}, L[0]);
  return cudaGetLastError();
}

// The recursions take a substep instead of the transforms while r <= 0.7 (their
// rounding, about 2/(1 - r) units per direction, is then that of a transform)
// and lines fit shared memory.  Where 17 taps or fewer do, the fused filters
// stay: W = 7 on 200 x 180 x 144 takes 90 us.  Long lines leave few blocks per SM
// (one from 880 entries on), so the gain shrinks: a whole predictor, transforms
// against lines, us: 200 x 180 x 144 384, 179; 512 x 256 x 128 879, 554; 128 x 256 x 512
// 879, 498; 900 x 128 x 96 704, 595; 96 x 1600 x 64 881, 464; 1600 x 96 x 64 564, 539;
// 1597 x 96 x 64 1131, 560; only x lines of 1000 to 1024, where the transforms are at
// their best, lose: 1024 x 256 x 64 808, 848.
bool use_lines(const ibm_flow* fl, int l) {
  if (fl->solve_w[l] >= 0) return false;
  const double a = (kGamma[l] + kRho[l]) * fl->dt * fl->nu / 2.0;
  for (int d = 0; d < 3; ++d)
    if (fl->n[d] > kMaxLine || line_root(a / (fl->h[d] * fl->h[d])) > 0.7) return false;
  return fl->n[1] <= 65535 && fl->n[2] <= 65535;   // the launches' grid.y
}

// The Poisson solve takes the z direction by recursions where a column fits a
// block's registers and its slowest recursion dies down to e^-4 within a turn
// (the larger of L_x, L_y at most 1.57 L_z): past that the closing of the column
// amplifies its rounding.  Errors against float64 relative to the transforms', on
// 9 x 5 x 15 .. 128^3 and cells 1 : 1 : 0.65 .. 1 : 1 : 16: p 0.3 .. 1.0, u 0.6 .. 1.0;
// beyond the line, at L_x = 4 L_z, p up to 1.2 (a float32 restatement).
bool use_z_lines(const ibm_flow* fl) {
  if (fl->n[2] > kZMax || (long long)(fl->n[0] / 2 + 1) * fl->n[1] > 0x7fffffffll - 32) return false;
  double least = 1e300;
  for (int d = 0; d < 2; ++d)
    if (fl->n[d] > 1) {
      const double k = 2.0 / fl->h[d] * std::sin(3.14159265358979323846 / fl->n[d]);
      least = std::min(least, 2.0 * std::asinh(0.5 * fl->h[2] * k));
    }
  return least * fl->n[2] >= 4.0;
}

int z_segments(const ibm_flow* fl) { return (fl->n[2] + kZSeg - 1) / kZSeg; }

cudaError_t set_up_z_lines(ibm_flow* fl) {
  fl->z_lines = use_z_lines(fl);
  if (!fl->z_lines) return cudaSuccess;
  const int M = (fl->n[0] / 2 + 1) * fl->n[1];
  const cudaError_t e = cudaMalloc(&fl->zcol, sizeof(float4) * (size_t)M);
  if (e != cudaSuccess) return e;
  poisson_z_table_kernel<<<(unsigned)((M + 127) / 128), 128>>>(
      fl->zcol, fl->n[0], fl->n[1], fl->n[2], fl->n[2] / z_segments(fl), fl->h[0], fl->h[1], fl->h[2]);
  return cudaGetLastError();
}

// device table of the powers, and the kernels' shared memory
cudaError_t set_up_lines(ibm_flow* fl) {
  bool any = false;
  for (int l = 0; l < 3; ++l) any = (fl->lines[l] = use_lines(fl, l)) || any;
  if (!any) return cudaSuccess;
  fl->pw_stride = 0;
  for (int d = 0; d < 3; ++d) fl->pw_stride += line_powers(fl->n[d]);
  std::vector<float> pw;
  for (int l = 0; l < 3; ++l) {
    const double a = (kGamma[l] + kRho[l]) * fl->dt * fl->nu / 2.0;
    for (int d = 0; d < 3; ++d) {
      const double r = line_root(a / (fl->h[d] * fl->h[d]));
      for (int k = 0; k < line_powers(fl->n[d]); ++k) pw.push_back((float)std::pow(r, k));
    }
  }
  cudaError_t e = cudaMalloc(&fl->pw, pw.size() * sizeof(float));
  if (e == cudaSuccess)
    e = cudaMemcpy(fl->pw, pw.data(), pw.size() * sizeof(float), cudaMemcpyHostToDevice);
  const size_t most = 32 * sizeof(float) * (size_t)(std::max({fl->n[0], fl->n[1], fl->n[2]}) | 1);
  if (e == cudaSuccess) e = allow_smem(line_x_kernel, most);
  for (auto k : {line_yz_kernel<false>, line_yz_kernel<true>})
    if (e == cudaSuccess) e = allow_smem(k, most);
  return e;
}

FGrid fgrid(const ibm_flow* fl) {
  FGrid G;
  G.nx = fl->n[0];
  G.ny = fl->n[1];
  G.nz = fl->n[2];
  for (int d = 0; d < 3; ++d) {
    G.ih[d] = (float)(1.0 / fl->h[d]);
    G.ih2[d] = (float)(1.0 / (fl->h[d] * fl->h[d]));
  }
  return G;
}

dim3 cell_grid(const ibm_flow* fl) {
  return dim3((unsigned)((fl->n[0] + 31) / 32), (unsigned)((fl->n[1] + 7) / 8), (unsigned)fl->n[2]);
}

// blocks of the quad kernels: a plane's quads, and `planes` planes per block
dim3 quad_grid(const ibm_flow* fl, int planes) {
  const int nq = fl->n[0] / 4 * fl->n[1];
  return dim3((unsigned)((nq + kQuadThreads - 1) / kQuadThreads),
              (unsigned)((fl->n[2] + planes - 1) / planes));
}

// Planes per thread of rhs4_kernel: the whole waves of blocks (two fit on an
// SM) times a column's length, the first plane's extra loads counted as one and
// a half planes (200 x 180 x 144: 9 planes, 1.9 waves, instead of 1.07 with 16)
int rhs_planes(const ibm_flow* fl, int n_sm) {
  const long nb = (fl->n[0] / 4 * fl->n[1] + kQuadThreads - 1) / kQuadThreads;
  int best = 1;
  double least = 1e300;
  for (int z = 4; z <= 32; ++z) {
    const long blocks = nb * ((fl->n[2] + z - 1) / z), waves = (blocks + 2 * n_sm - 1) / (2 * n_sm);
    const double cost = waves * (std::min(z, fl->n[2]) + 1.5);
    if (cost < least) {
      least = cost;
      best = z;
    }
  }
  return best;
}

// Output planes per block of cn_solve_kernel<W>: the whole waves of blocks times
// the planes a block walks (its 2W planes of halo, and two to fill the pipeline)
int solve_planes(const ibm_flow* fl, int W, int n_sm) {
  const long tiles = 3l * ((fl->n[0] + kSolveT - 1) / kSolveT) * ((fl->n[1] + kSolveT - 1) / kSolveT);
  const long slots = (long)solve_blocks(W) * n_sm;
  int best = fl->n[2];
  double least = 1e300;
  for (int parts = 1; parts <= std::max(1, fl->n[2] / 8); ++parts) {
    const int z = (fl->n[2] + parts - 1) / parts;
    const long blocks = tiles * ((fl->n[2] + z - 1) / z);
    const double cost = (double)((blocks + slots - 1) / slots) * (z + 2 * W + 2);
    if (cost < least) {
      least = cost;
      best = z;
    }
  }
  return best;
}

// blocks for the row kernels: enough rows in flight, at most one pass over them
unsigned row_blocks(const ibm_flow* fl) {
  const int rows = fl->n[1] * fl->n[2];
  const int b = (rows + kRowsPerBlock - 1) / kRowsPerBlock;
  return (unsigned)(b < 152 * 32 ? b : 152 * 32);
}

unsigned flat_blocks(size_t total) {
  const size_t b = (total + 255) / 256;
  return (unsigned)(b < (size_t)152 * 16 ? (b > 0 ? b : 1) : (size_t)152 * 16);
}

cudaError_t fft_status(cufftResult r) {
  return r == CUFFT_SUCCESS ? cudaSuccess : cudaErrorUnknown;
}

cudaError_t set_plan_streams(ibm_flow* fl, cudaStream_t s) {
  for (cufftHandle h : {fl->r2c3, fl->c2r3, fl->r2c1, fl->c2r1})
    if (cufftSetStream(h, s) != CUFFT_SUCCESS) return cudaErrorUnknown;
  return cudaSuccess;
}

void release(ibm_flow* fl) {
  if (fl->plans) {
    cufftDestroy(fl->r2c3);
    cufftDestroy(fl->c2r3);
    cufftDestroy(fl->r2c1);
    cufftDestroy(fl->c2r1);
  }
  for (void* q : {(void*)fl->H[0], (void*)fl->H[1], (void*)fl->R, (void*)fl->rp, (void*)fl->S,
                  (void*)fl->lam, (void*)fl->pw, (void*)fl->zcol})
    if (q) cudaFree(q);
  for (auto& row : fl->ev)
    for (cudaEvent_t& ev : row)
      if (ev) cudaEventDestroy(ev);
  for (cudaEvent_t& ev : fl->evs)
    if (ev) cudaEventDestroy(ev);
}

// Entries g_m, m = 0..kMaxSolveW, of the inverse of the periodic n-point
// operator 1 - c (E - 2 + E^-1): its eigenvalues are 1 + 4c sin^2(pi k/n), so
// g_m = (1/n) sum_k cos(2 pi k m/n) / (1 + 4c sin^2(pi k/n))  (float64).
// They are positive and sum to 1 over a period.
void inverse_taps(double cc, int n, double* g) {
  for (int m = 0; m <= kMaxSolveW; ++m) {
    double acc = 0.0;
    for (int k = 0; k < n; ++k) {
      const double sn = std::sin(M_PI * k / n);
      acc += std::cos(2.0 * M_PI * (double)k * m / n) / (1.0 + 4.0 * cc * sn * sn);
    }
    g[m] = acc / n;
  }
}

// Picks each substep's solve: the smallest W <= kMaxSolveW with the mass of the
// entries beyond |m| = W below 2^-26 in every direction and 2W + 1 <= n_d in every
// direction (short filters), else W = -1 (line recursions or transforms; also for
// planes of more than 65535 tiles).
void choose_solves(ibm_flow* fl) {
  const long tiles = (long)((fl->n[0] + kSolveT - 1) / kSolveT) * ((fl->n[1] + kSolveT - 1) / kSolveT);
  for (int l = 0; l < 3; ++l) {
    if (tiles > 65535) {   // the launch's grid.y
      fl->solve_w[l] = -1;
      continue;
    }
    const double a = (kGamma[l] + kRho[l]) * fl->dt * fl->nu / 2.0;
    int wl = 0;
    double g[3][kMaxSolveW + 1];
    for (int d = 0; d < 3 && wl >= 0; ++d) {
      inverse_taps(a / (fl->h[d] * fl->h[d]), fl->n[d], g[d]);
      int wd = -1;
      double inner = g[d][0];
      for (int w = 0; w <= kMaxSolveW && 2 * w + 1 <= fl->n[d]; ++w) {
        if (w > 0) inner += 2.0 * g[d][w];
        if (1.0 - inner <= std::ldexp(1.0, -26)) {
          wd = w;
          break;
        }
      }
      wl = wd < 0 ? -1 : std::max(wl, wd);
    }
    // every direction is filtered with the largest W: a short period that its own
    // width already covers would count entries twice, and the walk wrap past it
    for (int d = 0; d < 3; ++d)
      if (2 * wl + 1 > fl->n[d]) wl = -1;
    fl->solve_w[l] = wl;
    for (int d = 0; d < 3; ++d)
      for (int m = 0; m <= kMaxSolveW; ++m)
        fl->taps[l][d][m] = wl >= 0 && m <= wl ? (float)g[d][m] : 0.f;
  }
}

ibm_status flow_err(ibm_status s, const std::string& m) {
  set_global_error(m);
  return s;
}

}  // namespace

// record boundary k of substep l (k = 0..11) when phase timing is on
cudaError_t flow_mark(ibm_flow* fl, int l, int k, cudaStream_t s) {
  if (!fl->timing) return cudaSuccess;
  return cudaEventRecord(fl->ev[l][k], s);
}

// record boundary k (0..2) of the body update: its start, after the marker
// kernel (body sums and probe traction), after the force kernel
cudaError_t flow_mark_struct(ibm_flow* fl, int k, cudaStream_t s) {
  if (!fl->timing) return cudaSuccess;
  const cudaError_t e = cudaEventRecord(fl->evs[k], s);
  if (e == cudaSuccess && k == 2) fl->have_struct = true;
  return e;
}

cudaError_t flow_predict(ibm_flow* fl, int l, float* u, float* v, float* w, const float* p,
                         cudaStream_t s) {
  const FGrid G = fgrid(fl);
  const float dt = (float)fl->dt, nu = (float)fl->nu;
  const double alpha = kGamma[l] + kRho[l];
  CVec3 Hp{{nullptr, nullptr, nullptr}};
  if (kRho[l] != 0.0)
    for (int c = 0; c < 3; ++c) Hp.c[c] = fl->H[fl->hcur] + c * fl->N;
  float* Hn = fl->H[fl->hcur ^ 1];
  const Vec3 Ho{{Hn, Hn + fl->N, Hn + 2 * fl->N}};
  const Vec3 Ro{{fl->R, fl->R + fl->N, fl->R + 2 * fl->N}};
  cudaError_t e = set_plan_streams(fl, s);
  if (e != cudaSuccess) return e;
  e = flow_mark(fl, l, 0, s);
  if (e != cudaSuccess) return e;
  if (quads(fl, u, v, w, p)) {
    auto kernel = Hp.c[0] ? rhs4_kernel<true> : rhs4_kernel<false>;
    kernel<<<quad_grid(fl, fl->rhs_planes), kQuadThreads, 0, s>>>(
        G, u, v, w, p, Hp.c[0], Hn, fl->R, (float)kGamma[l], (float)kRho[l], (float)alpha, nu, dt,
        fl->rhs_planes);
  } else {
    rhs_kernel<<<cell_grid(fl), dim3(32, 8), 0, s>>>(G, u, v, w, p, Hp, Ho, Ro, (float)kGamma[l],
                                                       (float)kRho[l], (float)alpha, nu, dt);
  }
  e = cudaGetLastError();
  if (e == cudaSuccess) e = flow_mark(fl, l, 1, s);
  const bool lines = fl->lines[l], fourier = fl->solve_w[l] < 0 && !lines;
  // real-space path: the three Fourier phases stay empty
  if (e == cudaSuccess && fourier) e = fft_status(cufftExecR2C(fl->r2c3, fl->R, fl->S));
  if (e == cudaSuccess) e = flow_mark(fl, l, 2, s);
  if (e == cudaSuccess && fourier) {
    const int nxh = fl->n[0] / 2 + 1;
    cn_scale_kernel<<<dim3(row_blocks(fl), 3), dim3(kRowThreads, kRowsPerBlock), 0, s>>>(
        fl->S, nxh, fl->n[1], fl->n[2], fl->lam, (float)(alpha * fl->dt * fl->nu / 2.0),
        (float)(1.0 / (double)fl->N));
    e = cudaGetLastError();
  }
  if (e == cudaSuccess) e = flow_mark(fl, l, 3, s);
  if (e == cudaSuccess && fourier) e = fft_status(cufftExecC2R(fl->c2r3, fl->S, fl->R));
  if (e == cudaSuccess) e = flow_mark(fl, l, 4, s);
  if (e == cudaSuccess && fourier) {
    add_kernel<<<dim3(flat_blocks(fl->N), 3), 256, 0, s>>>(Vec3{{u, v, w}}, fl->R, fl->N);
    e = cudaGetLastError();
  } else if (e == cudaSuccess) {
    e = lines ? launch_lines(fl, l, u, v, w, s) : launch_cn_solve(fl, l, u, v, w, s);
  }
  if (e == cudaSuccess) e = flow_mark(fl, l, 5, s);
  if (e == cudaSuccess) {
    fl->hcur ^= 1;
    fl->last = l;
  }
  return e;
}

cudaError_t flow_project(ibm_flow* fl, int l, float* u, float* v, float* w, float* p,
                         const float* fx, const float* fy, const float* fz, float fscale,
                         cudaStream_t s) {
  const FGrid G = fgrid(fl);
  const double alpha = kGamma[l] + kRho[l];
  const CVec3 f{{fx, fy, fz}};
  cudaError_t e = set_plan_streams(fl, s);
  if (e != cudaSuccess) return e;
  e = flow_mark(fl, l, 6, s);
  if (e != cudaSuccess) return e;
  const bool q4 = quads(fl, u, v, w, p, fx, fy, fz);
  if (q4) {
    auto kernel = fx ? div4_kernel<true> : div4_kernel<false>;
    kernel<<<quad_grid(fl, 1), kQuadThreads, 0, s>>>(G, CVec3{{u, v, w}}, f, fscale, fl->rp);
  } else {
    div_kernel<<<cell_grid(fl), dim3(32, 8), 0, s>>>(G, CVec3{{u, v, w}}, f, fscale, fl->rp);
  }
  e = cudaGetLastError();
  if (e == cudaSuccess) e = flow_mark(fl, l, 7, s);
  if (e == cudaSuccess) e = fft_status(cufftExecR2C(fl->r2c1, fl->rp, fl->S));
  if (e == cudaSuccess) e = flow_mark(fl, l, 8, s);
  if (e == cudaSuccess) {
    const int nxh = fl->n[0] / 2 + 1;
    if (fl->z_lines) {
      const dim3 block(32, (unsigned)z_segments(fl));
      poisson_z_kernel<<<(unsigned)((nxh * fl->n[1] + 31) / 32) + 1, block, 0, s>>>(
          fl->S, nxh, fl->n[1], fl->n[2], fl->zcol, fl->h[2] * fl->h[2],
          1.0 / ((double)fl->n[0] * fl->n[1] * alpha * fl->dt));
    } else {
      poisson_scale_kernel<<<row_blocks(fl), dim3(kRowThreads, kRowsPerBlock), 0, s>>>(
          fl->S, nxh, fl->n[1], fl->n[2], fl->lam, (float)(1.0 / ((double)fl->N * alpha * fl->dt)));
    }
    e = cudaGetLastError();
  }
  if (e == cudaSuccess) e = flow_mark(fl, l, 9, s);
  if (e == cudaSuccess) e = fft_status(cufftExecC2R(fl->c2r1, fl->S, fl->rp));
  if (e == cudaSuccess) e = flow_mark(fl, l, 10, s);
  if (e == cudaSuccess) {
    const float adt = (float)(alpha * fl->dt), a = (float)(alpha * fl->dt * fl->nu / 2.0);
    if (q4) {
      auto kernel = fx ? project4_kernel<true> : project4_kernel<false>;
      kernel<<<quad_grid(fl, 1), kQuadThreads, 0, s>>>(G, Vec3{{u, v, w}}, p, fl->rp, f, fscale,
                                                       adt, a);
    } else {
      project_kernel<<<cell_grid(fl), dim3(32, 8), 0, s>>>(G, Vec3{{u, v, w}}, p, fl->rp, f, fscale,
                                                           adt, a);
    }
    e = cudaGetLastError();
  }
  if (e == cudaSuccess) e = flow_mark(fl, l, 11, s);
  if (e == cudaSuccess && fl->timing) fl->have_sub[l] = true;
  return e;
}

bool flow_matches(const ibm_flow* fl, const ibm_grid_desc& g, double dt, double mu) {
  for (int d = 0; d < 3; ++d)
    if (g.n[d] != fl->n[d] || std::fabs(g.L[d] - fl->L[d]) > 1e-12 * std::fabs(fl->L[d]))
      return false;
  return std::fabs(dt - fl->dt) <= 1e-12 * fl->dt && std::fabs(mu - fl->nu) <= 1e-12 * (1.0 + fl->nu);
}

cudaStream_t flow_stream(const ibm_flow* fl) { return fl->stream; }
int flow_device(const ibm_flow* fl) { return fl->device; }
size_t flow_cells(const ibm_flow* fl) { return fl->N; }

}  // namespace ibm

using ibm::flow_err;

extern "C" ibm_status ibm_flow_create(const ibm_grid_desc* grid, double nu, double dt,
                                      ibm_flow** out) {
  if (out) *out = nullptr;
  if (!grid || !out) return flow_err(IBM_ERR_INVALID_ARG, "ibm_flow_create: null argument");
  for (int d = 0; d < 3; ++d)
    if (grid->n[d] < 4 || !(grid->L[d] > 0.0) || !std::isfinite(grid->L[d]))
      return flow_err(IBM_ERR_INVALID_ARG, "ibm_flow_create: grid needs n >= 4 and L > 0");
  if ((double)grid->n[0] * grid->n[1] * grid->n[2] >= 2147483648.0)
    return flow_err(IBM_ERR_UNSUPPORTED, "ibm_flow_create: grids of 2^31 cells or more");
  if (grid->n[2] > 65535 || (grid->n[1] + 7) / 8 > 65535)
    return flow_err(IBM_ERR_UNSUPPORTED, "ibm_flow_create: n_z above 65535 or n_y above 524280");
  if (!(nu >= 0.0) || !std::isfinite(nu) || !(dt > 0.0) || !std::isfinite(dt))
    return flow_err(IBM_ERR_INVALID_ARG, "ibm_flow_create: needs nu >= 0 and dt > 0");
  ibm_flow* fl = new ibm_flow();
  cudaGetDevice(&fl->device);
  for (int d = 0; d < 3; ++d) {
    fl->n[d] = grid->n[d];
    fl->L[d] = grid->L[d];
    fl->h[d] = grid->L[d] / grid->n[d];
  }
  fl->nu = nu;
  fl->dt = dt;
  ibm::choose_solves(fl);
  int n_sm = 0;
  if (cudaDeviceGetAttribute(&n_sm, cudaDevAttrMultiProcessorCount, fl->device) == cudaSuccess) {
    fl->rhs_planes = ibm::rhs_planes(fl, std::max(n_sm, 1));
    for (int l = 0; l < 3; ++l)
      if (fl->solve_w[l] >= 0) fl->solve_planes[l] = ibm::solve_planes(fl, fl->solve_w[l], std::max(n_sm, 1));
  }
  const int nx = fl->n[0], ny = fl->n[1], nz = fl->n[2], nxh = nx / 2 + 1;
  fl->N = (size_t)nx * ny * nz;
  fl->NC = (size_t)nxh * ny * nz;
  cudaError_t e = cudaSuccess;
  e = ibm::set_up_lines(fl);
  if (e == cudaSuccess) e = ibm::set_up_z_lines(fl);
  for (int b = 0; b < 2 && e == cudaSuccess; ++b) e = cudaMalloc(&fl->H[b], 3 * fl->N * sizeof(float));
  if (e == cudaSuccess) e = cudaMalloc(&fl->R, 3 * fl->N * sizeof(float));
  if (e == cudaSuccess) e = cudaMalloc(&fl->rp, fl->N * sizeof(float));
  if (e == cudaSuccess) e = cudaMalloc(&fl->S, 3 * fl->NC * sizeof(cufftComplex));
  if (e == cudaSuccess) e = cudaMalloc(&fl->lam, (size_t)(nxh + ny + nz) * sizeof(float));
  if (e == cudaSuccess) {
    std::vector<float> lam;
    const int m[3] = {nxh, ny, nz};
    for (int d = 0; d < 3; ++d)
      for (int q = 0; q < m[d]; ++q) {
        const double s = std::sin(M_PI * q / fl->n[d]);
        lam.push_back((float)(-(4.0 / (fl->h[d] * fl->h[d])) * s * s));
      }
    e = cudaMemcpy(fl->lam, lam.data(), lam.size() * sizeof(float), cudaMemcpyHostToDevice);
  }
  // the tables are there whichever stream the flow runs on
  if (e == cudaSuccess) e = cudaStreamSynchronize(nullptr);
  if (e != cudaSuccess) {
    ibm::release(fl);
    delete fl;
    cudaGetLastError();
    return flow_err(e == cudaErrorMemoryAllocation ? IBM_ERR_OOM : IBM_ERR_CUDA,
                    std::string("ibm_flow_create: ") + cudaGetErrorString(e));
  }
  int dims[3] = {nz, ny, nx};
  cufftResult r = cufftPlanMany(&fl->r2c3, 3, dims, nullptr, 1, 0, nullptr, 1, 0, CUFFT_R2C, 3);
  bool ok = r == CUFFT_SUCCESS;
  if (ok) ok = cufftPlanMany(&fl->c2r3, 3, dims, nullptr, 1, 0, nullptr, 1, 0, CUFFT_C2R, 3) == CUFFT_SUCCESS;
  // the Poisson solve's: all three directions, or (x, y) of every plane
  const int rank = fl->z_lines ? 2 : 3, batch = fl->z_lines ? nz : 1;
  int* pd = dims + 3 - rank;
  if (ok) ok = cufftPlanMany(&fl->r2c1, rank, pd, nullptr, 1, 0, nullptr, 1, 0, CUFFT_R2C, batch) == CUFFT_SUCCESS;
  if (ok) ok = cufftPlanMany(&fl->c2r1, rank, pd, nullptr, 1, 0, nullptr, 1, 0, CUFFT_C2R, batch) == CUFFT_SUCCESS;
  if (!ok) {
    // plans created so far are destroyed individually
    for (cufftHandle h : {fl->r2c3, fl->c2r3, fl->r2c1, fl->c2r1})
      if (h) cufftDestroy(h);
    fl->plans = false;
    ibm::release(fl);
    delete fl;
    return flow_err(IBM_ERR_CUDA, "ibm_flow_create: cuFFT plan creation failed");
  }
  fl->plans = true;
  *out = fl;
  return IBM_OK;
}

extern "C" ibm_status ibm_flow_solve_width(const ibm_flow* fl, int32_t substep, int32_t* width) {
  if (!fl || !width) return flow_err(IBM_ERR_INVALID_ARG, "ibm_flow_solve_width: null argument");
  if (substep < 0 || substep > 2)
    return flow_err(IBM_ERR_INVALID_ARG, "ibm_flow_solve_width: substep must be 0, 1 or 2");
  *width = fl->solve_w[substep];
  return IBM_OK;
}

extern "C" ibm_status ibm_flow_set_stream(ibm_flow* fl, void* stream) {
  if (!fl) return flow_err(IBM_ERR_INVALID_ARG, "ibm_flow_set_stream: null flow");
  fl->stream = static_cast<cudaStream_t>(stream);
  return IBM_OK;
}

extern "C" void ibm_flow_destroy(ibm_flow* fl) {
  if (!fl) return;
  cudaSetDevice(fl->device);
  // coupled steps run on a context's stream: wait for all work on the device
  cudaDeviceSynchronize();
  ibm::release(fl);
  delete fl;
}

extern "C" ibm_status ibm_flow_predict(ibm_flow* fl, int32_t substep, float* u, float* v,
                                       float* w, const float* p) {
  if (!fl || !u || !v || !w || !p) return flow_err(IBM_ERR_INVALID_ARG, "ibm_flow_predict: null argument");
  if (substep < 0 || substep > 2)
    return flow_err(IBM_ERR_INVALID_ARG, "ibm_flow_predict: substep must be 0, 1 or 2");
  if (substep > 0 && fl->last != substep - 1)
    return flow_err(IBM_ERR_INVALID_ARG, "ibm_flow_predict: substeps must run in order");
  cudaSetDevice(fl->device);
  const cudaError_t e = ibm::flow_predict(fl, substep, u, v, w, p, fl->stream);
  if (e != cudaSuccess)
    return flow_err(IBM_ERR_CUDA, std::string("ibm_flow_predict: ") + cudaGetErrorString(e));
  return IBM_OK;
}

extern "C" ibm_status ibm_flow_project(ibm_flow* fl, int32_t substep, float* u, float* v,
                                       float* w, float* p, const float* fx, const float* fy,
                                       const float* fz, float f_scale) {
  if (!fl || !u || !v || !w || !p) return flow_err(IBM_ERR_INVALID_ARG, "ibm_flow_project: null argument");
  if (substep < 0 || substep > 2)
    return flow_err(IBM_ERR_INVALID_ARG, "ibm_flow_project: substep must be 0, 1 or 2");
  const bool any = fx || fy || fz;
  if (any && !(fx && fy && fz))
    return flow_err(IBM_ERR_INVALID_ARG, "ibm_flow_project: give all three force fields or none");
  cudaSetDevice(fl->device);
  const cudaError_t e = ibm::flow_project(fl, substep, u, v, w, p, fx, fy, fz, f_scale, fl->stream);
  if (e != cudaSuccess)
    return flow_err(IBM_ERR_CUDA, std::string("ibm_flow_project: ") + cudaGetErrorString(e));
  return IBM_OK;
}

extern "C" ibm_status ibm_flow_set_phase_timing(ibm_flow* fl, int32_t on) {
  if (!fl) return flow_err(IBM_ERR_INVALID_ARG, "ibm_flow_set_phase_timing: null flow");
  cudaSetDevice(fl->device);
  if (on && !fl->ev[0][0]) {
    for (auto& row : fl->ev)
      for (cudaEvent_t& ev : row) {
        const cudaError_t e = cudaEventCreate(&ev);
        if (e != cudaSuccess)
          return flow_err(IBM_ERR_CUDA, std::string("cudaEventCreate: ") + cudaGetErrorString(e));
      }
    for (cudaEvent_t& ev : fl->evs) {
      const cudaError_t e = cudaEventCreate(&ev);
      if (e != cudaSuccess)
        return flow_err(IBM_ERR_CUDA, std::string("cudaEventCreate: ") + cudaGetErrorString(e));
    }
  }
  fl->timing = on != 0;
  for (bool& b : fl->have_sub) b = false;
  fl->have_struct = false;
  return IBM_OK;
}

extern "C" ibm_status ibm_flow_get_phase_times(ibm_flow* fl, float* ms) {
  if (!fl || !ms) return flow_err(IBM_ERR_INVALID_ARG, "ibm_flow_get_phase_times: null argument");
  for (bool b : fl->have_sub)
    if (!b)
      return flow_err(IBM_ERR_INVALID_ARG,
                      "ibm_flow_get_phase_times: no timed substep 0, 1 and 2 recorded");
  cudaSetDevice(fl->device);
  cudaError_t e = cudaEventSynchronize(fl->ev[2][11]);
  for (int k = 0; k < 11; ++k) {
    ms[k] = 0.f;
    for (int l = 0; l < 3 && e == cudaSuccess; ++l) {
      float t = 0.f;
      e = cudaEventElapsedTime(&t, fl->ev[l][k], fl->ev[l][k + 1]);
      ms[k] += t;
    }
  }
  ms[11] = ms[12] = 0.f;
  if (e == cudaSuccess && fl->have_struct) {
    e = cudaEventSynchronize(fl->evs[2]);
    if (e == cudaSuccess) e = cudaEventElapsedTime(&ms[11], fl->evs[0], fl->evs[1]);
    if (e == cudaSuccess) e = cudaEventElapsedTime(&ms[12], fl->evs[1], fl->evs[2]);
  }
  if (e != cudaSuccess)
    return flow_err(IBM_ERR_CUDA, std::string("ibm_flow_get_phase_times: ") + cudaGetErrorString(e));
  return IBM_OK;
}
