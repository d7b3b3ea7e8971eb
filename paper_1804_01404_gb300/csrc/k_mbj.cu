// TB-mBJ exchange potential (xc = 3; Sec. 4.1 names the Becke-Johnson potential and its
// Tran-Blaha variant as options besides the LDA).  Published forms, per spin channel of the
// spin-unpolarised system (rho_s = rho/2, t_s = tau~/2):
//   D   = 2 t_s - |grad rho_s|^2 / (4 rho_s)              (curvature of the Fermi hole)
//   Q   = (lap rho_s - 2 gamma D) / 6,  gamma = 0.8
//   x   : x exp(-2x/3) / (x - 2) = (2/3) pi^(2/3) rho_s^(5/3) / Q      (Becke-Roussel hole)
//   b   = (x^3 exp(-x) / (8 pi rho_s))^(1/3)
//   v_BR = -(1/b) (1 - exp(-x) - x exp(-x) / 2)
//   v_x = c v_BR + (3c - 2) (1/pi) sqrt(5/12) sqrt(2 t_s / rho_s)
//   c   = alpha + beta sqrt(g), g = (1/Omega) int |grad rho| / rho,  alpha = -0.012, beta = 1.023
// tau~ = tau - |j|^2 / (2 rho) is the kinetic energy density of the time-dependent orbitals with
// the current's share removed (unchanged by a uniform A'), tau = sum_k w_k sum_n |(D1 + i k) u|^2,
// j = sum_k w_k sum_n 2 Im(conj(u) (D1 + i k) u).  Derivatives are the 8th-order central
// differences of the orbital stencil (periodic wrap, or zero outside an isolated box).  Points with
// rho <= 1e-10 get no mBJ potential.
//
// Launches: k_tau (partial sums of rho, tau, j over chunks of orbitals, one thread per grid point; k_tau_seg: one
// thread per two x-adjacent points of four planes of FP32 grids with an even nx), k_mbj_x (folds the chunks,
// differentiates rho, solves the Becke-Roussel equation, and with c fixed adds v_x to V, else leaves its two
// parts and sums g) and, with c from g, k_mbj_apply.
#include <cuda_runtime.h>

#include <algorithm>

#include "grid_sum.cuh"
#include "tdks_internal.h"

namespace tdks {

namespace {

constexpr int kMbjThreads = 128;          // k_tau, a group of k_tau_seg
constexpr int kTauGroups = 3;             // k_tau_seg: orbital groups of a CTA (its registers fill an SM)
constexpr int kTauSeg = 4;                // k_tau_seg: planes of a thread
constexpr int kTauChain = 16;             // k_tau_seg: orbitals of a register sum
constexpr size_t kTauSmem = sizeof(float) * kTauGroups * 10 * kTauSeg * kMbjThreads;
constexpr int kBrPoints = 64;             // k_mbj_x: points of a CTA, four threads each
constexpr double kPi23 = 2.14502939711102560008;   // pi^(2/3)
constexpr double kPi = 3.14159265358979323846;
constexpr double kRhoMin = 1e-10;
constexpr double kGamma = 0.8, kAlpha = -0.012, kBeta = 1.023;

struct Fd {   // the stencil's difference coefficients (kFD1, kFD2), passed by value
  double d1[4], d2[5];
};

template <typename T>
struct D1h {  // first-derivative coefficients FD1[m] / h_a in the orbitals' precision, formed on the host
  T c[3][4];
};

struct Nbr {   // linear indices of the 4 neighbours per side along each axis (-1: outside the box)
  int p[3][4], m[3][4];
};

__device__ __forceinline__ Nbr neighbours(int ix, int iy, int iz, int nx, int ny, int nz, int periodic) {
  Nbr b;
  const int n[3] = {nx, ny, nz}, i[3] = {ix, iy, iz};
#pragma unroll
  for (int a = 0; a < 3; ++a) {
#pragma unroll
    for (int m = 1; m <= 4; ++m) {
      int jp = i[a] + m, jm = i[a] - m;
      bool op = true, om = true;
      if (periodic) {
        jp = jp >= n[a] ? jp - n[a] : jp;       // n >= 4: one wrap suffices
        jm = jm < 0 ? jm + n[a] : jm;
      } else {
        op = jp < n[a];
        om = jm >= 0;
      }
      int cp[3] = {ix, iy, iz}, cm[3] = {ix, iy, iz};
      cp[a] = jp;
      cm[a] = jm;
      b.p[a][m - 1] = op ? (cp[2] * ny + cp[1]) * nx + cp[0] : -1;
      b.m[a][m - 1] = om ? (cm[2] * ny + cm[1]) * nx + cm[0] : -1;
    }
  }
  return b;
}

template <typename V>
__device__ __forceinline__ V ld_or_zero(const V* f, int i) {
  return i >= 0 ? f[i] : V{};
}

// part[(chunk * 5 + c) * npts + p], c = rho, tau, j_x, j_y, j_z, over the orbitals of one chunk.
template <typename T>
__global__ void __launch_bounds__(kMbjThreads) k_tau(const typename Cplx<T>::type* __restrict__ u, int nk, int norb,
                                                    int nx, int ny, int nz, int periodic,
                                                    const double* __restrict__ kpts, const double* __restrict__ kw,
                                                    D1h<T> d1, int ochunk, double* __restrict__ part) {
  using C = typename Cplx<T>::type;
  const int npts = nx * ny * nz;
  const int p = blockIdx.x * blockDim.x + threadIdx.x;
  if (p >= npts) return;
  const int ix = p % nx, iy = (p / nx) % ny, iz = p / (nx * ny);
  const Nbr nb = neighbours(ix, iy, iz, nx, ny, nz, periodic);
  const int o0 = blockIdx.y * ochunk, o1 = min(o0 + ochunk, nk * norb);
  T acc[5] = {0, 0, 0, 0, 0};
  // the orbitals of one k at a time: unweighted sums over them, weighted once per k (the weight and
  // wave vector are converted once per k -- FP64 -> FP32 conversions run on the slow FP64 pipe), and
  // a branch-free inner loop whose loads the compiler can overlap across orbitals
  for (int o = o0; o < o1;) {
    const int k = o / norb;
    const int oe = min(o1, (k + 1) * norb);
    const T q[3] = {(T)kpts[3 * k], (T)kpts[3 * k + 1], (T)kpts[3 * k + 2]};
    T sk[5] = {0, 0, 0, 0, 0};
#pragma unroll 2
    for (; o < oe; ++o) {
      const C* f = u + (size_t)o * npts;
      const C c0 = f[p];
      sk[0] += c0.x * c0.x + c0.y * c0.y;
#pragma unroll
      for (int a = 0; a < 3; ++a) {
        C g = C{-q[a] * c0.y, q[a] * c0.x};                             // i q u
#pragma unroll
        for (int m = 0; m < 4; ++m) {
          const C fp = ld_or_zero(f, nb.p[a][m]), fm = ld_or_zero(f, nb.m[a][m]);
          g.x += d1.c[a][m] * (fp.x - fm.x);
          g.y += d1.c[a][m] * (fp.y - fm.y);
        }
        sk[1] += g.x * g.x + g.y * g.y;
        sk[2 + a] += c0.x * g.y - c0.y * g.x;                           // Im(conj(u) g)
      }
    }
    const T w = (T)(2.0 * kw[k]);
    acc[0] += w * sk[0];
    acc[1] += T(0.5) * w * sk[1];
#pragma unroll
    for (int c = 2; c < 5; ++c) acc[c] += w * sk[c];
  }
#pragma unroll
  for (int c = 0; c < 5; ++c) part[((size_t)blockIdx.y * 5 + c) * npts + p] = (double)acc[c];
}

// k_tau for FP32 grids with an even nx: a thread takes two x-adjacent points (x even) of kTauSeg planes.  A point
// pair is one 16-byte load; the pairs of the planes z0 - 4 .. z0 + 7 of a column are loaded once, so a pair costs 15
// loads instead of 50 for its two points.  One thread per pair (21 loads, any z) was bound by L2: a CTA's 256
// points lie in one or two planes, and each orbital's eight planes around them came from L2 again for every CTA,
// 13 times the orbital; the CTAs here cover four planes, 3 times.  The kTauGroups groups of a CTA take different
// orbitals of the chunk and are added in shared memory, so that few chunks (FP64 folds) fill the SMs.  An FP32 sum in
// registers ends after kTauChain orbitals and is added to the thread's in shared memory: one chain over a group's
// 68 orbitals (1024 of 30^3) left the potential 1.3e-8 from FP64, sums by k-point 1.1e-8, this 0.7e-8.
// 20^3, 1024 orbitals: 107 us before, 70 here (42 % of the issue slots; what is left is the latency of L2).
// With an even nx a neighbour pair is wholly inside or wholly outside an isolated box.
__device__ __forceinline__ float4 ld4_or_zero(const float2* f, int i) {
  return i >= 0 ? __ldg(reinterpret_cast<const float4*>(f + i)) : make_float4(0.f, 0.f, 0.f, 0.f);
}

__global__ void __launch_bounds__(kMbjThreads* kTauGroups, 1) k_tau_seg(const float2* __restrict__ u, int nk, int norb,
                                                                      int nx, int ny, int nz, int periodic,
                                                                      const double* __restrict__ kpts,
                                                                      const double* __restrict__ kw, D1h<float> d1,
                                                                      int ochunk, double* __restrict__ part) {
  constexpr int L = kTauSeg;
  extern __shared__ float tau_smem[];              // [kTauGroups][10 L][kMbjThreads] sums of a thread
  const int npts = nx * ny * nz, nxh = nx / 2, nxy = nx * ny, ncol = nxh * ny;
  const int grp = threadIdx.x / kMbjThreads, lt = threadIdx.x - grp * kMbjThreads;
  const int t = blockIdx.x * kMbjThreads + lt;
  const int seg = t / ncol, col = t - seg * ncol, z0 = seg * L;
  const bool in = z0 < nz;
  const int iy = col / nxh, ix = 2 * (col - iy * nxh), pxy = iy * nx + ix;
  int ox[4], oy[8], oz[L + 8];                     // in-plane offsets of pairs, plane offsets (-1: outside the box)
  const int dxs[4] = {-4, -2, 2, 4};
#pragma unroll
  for (int j = 0; j < 4; ++j) {
    int jx = ix + dxs[j];
    const bool inx = periodic || (jx >= 0 && jx < nx);
    jx = jx < 0 ? jx + nx : (jx >= nx ? jx - nx : jx);
    ox[j] = inx ? iy * nx + jx : -1;
  }
#pragma unroll
  for (int j = 0; j < 8; ++j) {
    const int m = 1 + (j >> 1);
    int jy = (j & 1) ? iy - m : iy + m;
    const bool iny = periodic || (jy >= 0 && jy < ny);
    jy = jy < 0 ? jy + ny : (jy >= ny ? jy - ny : jy);
    oy[j] = iny ? jy * nx + ix : -1;
  }
#pragma unroll
  for (int j = 0; j < L + 8; ++j) {
    int jz = z0 + j - 4;
    const bool inz = in && (periodic ? jz < nz + 4 : jz >= 0 && jz < nz);   // (of a partial segment: nothing beyond)
    jz = jz < 0 ? jz + nz : (jz >= nz ? jz - nz : jz);
    oz[j] = inz ? jz * nxy + pxy : -1;
  }
  const int c0 = blockIdx.y * ochunk, c1 = min(c0 + ochunk, nk * norb), gl = (max(c1 - c0, 0) + kTauGroups - 1) / kTauGroups;
  const int o0 = c0 + grp * gl, o1 = in ? min(o0 + gl, c1) : o0;
  float* mine = tau_smem + grp * 10 * L * kMbjThreads + lt;
  float acc[L][2][5];
#pragma unroll
  for (int i = 0; i < 10 * L; ++i) {
    acc[i / 10][i / 5 % 2][i % 5] = 0.f;
    mine[i * kMbjThreads] = 0.f;
  }
  auto flush = [&]() {                             // a chain of FP32 sums ends
#pragma unroll
    for (int i = 0; i < 10 * L; ++i) {
      mine[i * kMbjThreads] += acc[i / 10][i / 5 % 2][i % 5];
      acc[i / 10][i / 5 % 2][i % 5] = 0.f;
    }
  };
  int chain = 0;
  for (int o = o0; o < o1; ++o) {
    // (weighted orbital by orbital; the conversions of the weight and the wave vector are once per k)
    const int k = o / norb;
    const float q[3] = {(float)kpts[3 * k], (float)kpts[3 * k + 1], (float)kpts[3 * k + 2]};
    const float w2 = (float)(2.0 * kw[k]);
    const int oe = min(o1, (k + 1) * norb);
#pragma unroll 1
    for (; o < oe; ++o) {
      if (++chain > kTauChain) {
        flush();
        chain = 1;
      }
      const float2* f = u + (size_t)o * npts;
      float4 w[L + 8];
#pragma unroll
      for (int j = 0; j < L + 8; ++j) w[j] = ld4_or_zero(f, oz[j]);
#pragma unroll
      for (int zz = 0; zz < L; ++zz) {
        if (zz > 0 && z0 + zz >= nz) break;
        const float2* fz = f + (size_t)(z0 + zz) * nxy;
        float4 X[4], Y[8];
#pragma unroll
        for (int j = 0; j < 4; ++j) X[j] = ld4_or_zero(fz, ox[j]);
#pragma unroll
        for (int j = 0; j < 8; ++j) Y[j] = ld4_or_zero(fz, oy[j]);
        auto lo = [](float4 v) { return make_float2(v.x, v.y); };
        auto hi = [](float4 v) { return make_float2(v.z, v.w); };
        const float2 lo_c = lo(w[zz + 4]), hi_c = hi(w[zz + 4]);
        // x +- m of point A (x) and B (x + 1), m = 1..4
        const float2 axp[4] = {hi_c, lo(X[2]), hi(X[2]), lo(X[3])}, axm[4] = {hi(X[1]), lo(X[1]), hi(X[0]), lo(X[0])};
        const float2 bxp[4] = {lo(X[2]), hi(X[2]), lo(X[3]), hi(X[3])}, bxm[4] = {lo_c, hi(X[1]), lo(X[1]), hi(X[0])};
#pragma unroll
        for (int pt = 0; pt < 2; ++pt) {
          const float2 c = pt == 0 ? lo_c : hi_c;
          float tau = 0.f;
          acc[zz][pt][0] += w2 * (c.x * c.x + c.y * c.y);
#pragma unroll
          for (int a = 0; a < 3; ++a) {
            float2 g = make_float2(-q[a] * c.y, q[a] * c.x);              // i q u
#pragma unroll
            for (int m = 0; m < 4; ++m) {
              float2 fp, fm;
              if (a == 0) { fp = pt == 0 ? axp[m] : bxp[m]; fm = pt == 0 ? axm[m] : bxm[m]; }
              else if (a == 1) { fp = pt == 0 ? lo(Y[2 * m]) : hi(Y[2 * m]); fm = pt == 0 ? lo(Y[2 * m + 1]) : hi(Y[2 * m + 1]); }
              else { fp = pt == 0 ? lo(w[zz + 5 + m]) : hi(w[zz + 5 + m]); fm = pt == 0 ? lo(w[zz + 3 - m]) : hi(w[zz + 3 - m]); }
              g.x += d1.c[a][m] * (fp.x - fm.x);
              g.y += d1.c[a][m] * (fp.y - fm.y);
            }
            tau += g.x * g.x + g.y * g.y;
            acc[zz][pt][2 + a] += w2 * (c.x * g.y - c.y * g.x);             // Im(conj(u) g)
          }
          acc[zz][pt][1] += 0.5f * w2 * tau;
        }
      }
    }
    --o;
  }
  flush();
  __syncthreads();
  if (grp > 0 || !in) return;
#pragma unroll
  for (int i = 0; i < 10 * L; i += 5) {
    const int zz = i / 10, pt = i / 5 % 2;
    if (z0 + zz >= nz) break;
#pragma unroll
    for (int c = 0; c < 5; ++c) {
      double v = (double)mine[(i + c) * kMbjThreads];
#pragma unroll
      for (int g = 1; g < kTauGroups; ++g) v += (double)mine[(g * 10 * L + i + c) * kMbjThreads];
      part[((size_t)blockIdx.y * 5 + c) * npts + (size_t)(z0 + zz) * nxy + pxy + pt] = v;
    }
  }
}

// first derivative squared and second derivative of rho along one axis (i of n points, stride) at p
__device__ __forceinline__ void rho_axis(const double* __restrict__ rho, int p, int i, int n, int stride, int periodic,
                                         double h, const Fd& fd, double* g2, double* lap) {
  double d = 0.0, s = fd.d2[0] * rho[p];
#pragma unroll
  for (int m = 1; m <= 4; ++m) {
    int up = m, dn = -m;
    bool iu = true, id = true;
    if (periodic) {
      up -= i + up >= n ? n : 0;
      dn += i + dn < 0 ? n : 0;
    } else {
      iu = i + up < n;
      id = i + dn >= 0;
    }
    const double fp = iu ? rho[p + up * stride] : 0.0, fm = id ? rho[p + dn * stride] : 0.0;
    d += fd.d1[m - 1] * (fp - fm);
    s += fd.d2[m] * (fp + fm);
  }
  d /= h;
  *g2 = d * d;
  *lap = s / (h * h);
}

// H(x) = x exp(-2x/3) - y (x - 2): the Becke-Roussel equation times (x - 2), one root per branch
__device__ __forceinline__ double br_h(double x, double y) { return x * exp(-2.0 * x / 3.0) - y * (x - 2.0); }

__device__ __forceinline__ float br_hf(float x, float y) { return x * __expf(-2.0f * x / 3.0f) - y * (x - 2.0f); }

// Root x of x exp(-2x/3)/(x-2) = y: y < 0 in (0, 2) (H(0) = 2y < 0 < H(2)), y > 0 in (2, hi)
// (H(2) > 0 > H(hi)).  The bracket is narrowed by bisection in FP32 (26 steps; FP64 arithmetic runs
// at a small fraction of the FP32 rate on this GPU) and widened by a relative 1e-5 to cover the
// FP32 rounding of H; FP64 Newton steps kept inside it then reach full precision.  Where y is
// outside the FP32 range, or the widened bracket does not keep the signs of H, the bisection runs
// in FP64 (34 steps) on the whole branch.
__device__ double br_root(double y) {
  double neg = 0.0, pos = 0.0;        // H(neg) < 0 < H(pos)
  bool have = false;
  const double ay = fabs(y);
  if (ay > 1e-30 && ay < 1e30) {
    const float yf = (float)y;
    float nf, pf;
    if (yf < 0.0f) {
      nf = 0.0f;
      pf = 2.0f;
    } else {
      pf = 2.0f;
      nf = 4.0f;
      while (br_hf(nf, yf) > 0.0f && nf < 256.0f) nf *= 2.0f;   // y > 1e-30: the root is below 160
    }
    for (int it = 0; it < 26; ++it) {
      const float mid = 0.5f * (nf + pf);
      if (br_hf(mid, yf) < 0.0f) nf = mid; else pf = mid;
    }
    const double a = fmin((double)nf, (double)pf), b = fmax((double)nf, (double)pf);
    const double pad = 1e-5 * b;
    neg = y < 0.0 ? fmax(a - pad, 0.0) : b + pad;
    pos = y < 0.0 ? fmin(b + pad, 2.0) : fmax(a - pad, 2.0);
    have = br_h(neg, y) < 0.0 && br_h(pos, y) > 0.0;
  }
  if (!have) {
    if (y < 0.0) {
      neg = 0.0;
      pos = 2.0;
    } else {
      pos = 2.0;
      neg = 4.0;
      while (br_h(neg, y) > 0.0 && neg < 4096.0) neg *= 2.0;   // exp(-2x/3) underflows long before 4096
    }
    for (int it = 0; it < 34; ++it) {
      const double mid = 0.5 * (neg + pos);
      if (br_h(mid, y) < 0.0) neg = mid; else pos = mid;
    }
  }
  double x = 0.5 * (neg + pos);
  const double lo = fmin(neg, pos), hi = fmax(neg, pos);
  for (int it = 0; it < 5; ++it) {   // Newton, kept inside [lo, hi] (the root may sit at an end, x = 2)
    const double e = exp(-2.0 * x / 3.0);
    const double f = x * e - y * (x - 2.0), df = e * (1.0 - 2.0 * x / 3.0) - y;
    if (df == 0.0) break;
    const double xn = x - f / df;
    if (!(xn >= lo && xn <= hi)) break;
    const bool done = fabs(xn - x) <= 1e-9 * x;       // quadratic convergence: x is exact to rounding
    x = xn;
    if (done) break;
  }
  return x;
}

// v_x^mBJ(rho, grad rho, lap rho, tau~) = c A + (3c - 2) B: with c = c_fixed > 0 added to V, else A and B of a point
// go to its first two entries of part and the last CTA writes c = alpha + beta sqrt(g) to *c_out.  Bound by the chain
// of FP64 instructions of a point (70 cycles each, one warp per scheduler), so its independent parts run on four
// threads: a quarter of the chunks each, and an axis of the derivatives for the first three.  Newton stops
// when it has converged (two steps instead of five), and g no longer differentiates rho in a launch of its own.
// 20^3, 19 chunks: 36 us and 10 for g before, 35 and 3.5 for k_mbj_apply here (about 400 FP64 instructions a point).
__global__ void __launch_bounds__(4 * kBrPoints) k_mbj_x(const double* __restrict__ rho, double* __restrict__ part,
                                                       int nchunk, int nx, int ny, int nz, int periodic, double hx,
                                                       double hy, double hz, Fd fd, double c_fixed, double* partials,
                                                       unsigned* ticket, double* c_out, double* __restrict__ V) {
  __shared__ double s_fold[4][5][kBrPoints], s_der[3][2][kBrPoints], tot[1];
  const int npts = nx * ny * nz, lp = threadIdx.x % kBrPoints, quarter = threadIdx.x / kBrPoints;
  double sum[1] = {0.0};
  for (int base = blockIdx.x * kBrPoints; base < npts; base += gridDim.x * kBrPoints) {
    const int p = base + lp;
    const double r0 = p < npts ? rho[p] : 0.0;
    const bool on = r0 > kRhoMin;
    if (on) {
      // tau~ from the orbitals' chunks (their own rho for the current's share)
      double s[5] = {0, 0, 0, 0, 0};
#pragma unroll 4
      for (int ch = quarter; ch < nchunk; ch += 4)
#pragma unroll
        for (int c = 0; c < 5; ++c) s[c] += part[((size_t)ch * 5 + c) * npts + p];
#pragma unroll
      for (int c = 0; c < 5; ++c) s_fold[quarter][c][lp] = s[c];
      if (quarter < 3) {
        const int r = p / nx, x = p - r * nx, z = r / ny, y = r - z * ny;
        const int i = quarter == 0 ? x : quarter == 1 ? y : z, n = quarter == 0 ? nx : quarter == 1 ? ny : nz;
        rho_axis(rho, p, i, n, quarter == 0 ? 1 : quarter == 1 ? nx : nx * ny, periodic,
                 quarter == 0 ? hx : quarter == 1 ? hy : hz, fd, &s_der[quarter][0][lp], &s_der[quarter][1][lp]);
      }
    }
    __syncthreads();
    if (on && quarter == 0) {
      double s[5];
#pragma unroll
      for (int c = 0; c < 5; ++c) s[c] = (s_fold[0][c][lp] + s_fold[1][c][lp]) + (s_fold[2][c][lp] + s_fold[3][c][lp]);
      const double g2 = s_der[0][0][lp] + s_der[1][0][lp] + s_der[2][0][lp];
      const double lap = s_der[0][1][lp] + s_der[1][1][lp] + s_der[2][1][lp];
      double tt = 0.0;
      if (s[0] > 0.0) tt = fmax(s[1] - (s[2] * s[2] + s[3] * s[3] + s[4] * s[4]) / (2.0 * s[0]), 0.0);
      const double rs = 0.5 * r0, ts = 0.5 * tt, gs2 = 0.25 * g2;
      const double D = 2.0 * ts - gs2 / (4.0 * rs);
      const double Q = (0.5 * lap - 2.0 * kGamma * D) / 6.0;
      const double K = (2.0 / 3.0) * kPi23 * rs * cbrt(rs * rs);            // (2/3) pi^(2/3) rho_s^(5/3)
      const double x = Q != 0.0 ? br_root(K / Q) : 2.0;
      const double ex = exp(-x);
      const double b = cbrt(x * x * x * ex / (8.0 * kPi * rs));
      const double A = -(1.0 - ex - 0.5 * x * ex) / b, B = sqrt(5.0 / 12.0) / kPi * sqrt(2.0 * ts / rs);
      if (c_fixed > 0.0) {
        V[p] += c_fixed * A + (3.0 * c_fixed - 2.0) * B;
      } else {
        part[p] = A;
        part[(size_t)npts + p] = B;
        sum[0] += sqrt(g2) / r0;
      }
    }
    __syncthreads();
  }
  if (c_fixed > 0.0) return;
  if (grid_sum<1>(sum, partials, ticket, tot) && threadIdx.x == 0) *c_out = kAlpha + kBeta * sqrt(tot[0] / npts);
}

// V += c A + (3c - 2) B of k_mbj_x
__global__ void __launch_bounds__(128) k_mbj_apply(const double* __restrict__ rho, const double* __restrict__ part,
                                                 int npts, const double* __restrict__ c_dev, double* __restrict__ V) {
  const int p = blockIdx.x * blockDim.x + threadIdx.x;
  if (p >= npts || !(rho[p] > kRhoMin)) return;
  const double c = *c_dev;
  V[p] += c * part[p] + (3.0 * c - 2.0) * part[(size_t)npts + p];
}

}  // namespace

// whether k_tau_seg takes the grid
template <typename T>
static bool tau_seg(const int n[3]) { return sizeof(T) == 4 && n[0] % 2 == 0; }

static long long tau_ctas(const int n[3], bool seg) {
  const long long items = seg ? (long long)(n[0] / 2) * n[1] * ((n[2] + kTauSeg - 1) / kTauSeg) : (long long)n[0] * n[1] * n[2];
  return (items + kMbjThreads - 1) / kMbjThreads;
}

// chunks of orbitals for the tau kernels: one wave of CTAs of points x chunks, one per SM (k_tau_seg, whose
// registers fill it) or about 8 (k_tau)
int mbj_chunks(const int n[3], int norb_tot, bool f32) {
  const bool seg = f32 && tau_seg<float>(n);
  long long ch = (seg ? 152LL : 152LL * 8) / tau_ctas(n, seg);
  if (ch > norb_tot) ch = norb_tot;
  return ch < 1 ? 1 : (int)ch;
}

template <typename T>
cudaError_t launch_mbj(const typename Cplx<T>::type* u, int nk, int norb, const int n[3], int periodic,
                       const double h[3], const double* kpts, const double* kw, const double* rho, double c_fixed,
                       double* part, int nchunk, double* partials, unsigned* ticket, double* c_dev, double* V,
                       cudaStream_t s, int* nlaunch) {
  const int npts = n[0] * n[1] * n[2];
  const int norb_tot = nk * norb;
  const int ochunk = (norb_tot + nchunk - 1) / nchunk;
  const bool seg = tau_seg<T>(n) && (reinterpret_cast<size_t>(u) & 15) == 0;   // (16-byte loads)
  const dim3 grid((unsigned)tau_ctas(n, seg), nchunk);
  Fd fd;
  for (int m = 0; m < 4; ++m) fd.d1[m] = kFD1[m];
  for (int m = 0; m < 5; ++m) fd.d2[m] = kFD2[m];
  D1h<T> d1;
  for (int a = 0; a < 3; ++a)
    for (int m = 0; m < 4; ++m) d1.c[a][m] = (T)(kFD1[m] / h[a]);
  if constexpr (sizeof(T) == 4) {
    if (seg) {
      const cudaError_t es = cudaFuncSetAttribute(k_tau_seg, cudaFuncAttributeMaxDynamicSharedMemorySize, (int)kTauSmem);
      if (es != cudaSuccess) return es;
      k_tau_seg<<<grid, kMbjThreads * kTauGroups, kTauSmem, s>>>(u, nk, norb, n[0], n[1], n[2], periodic, kpts, kw, d1, ochunk,
                                                                 part);
    }
  }
  if (!seg)
    k_tau<T><<<grid, kMbjThreads, 0, s>>>(u, nk, norb, n[0], n[1], n[2], periodic, kpts, kw, d1, ochunk, part);
  cudaError_t e = cudaGetLastError();
  if (e != cudaSuccess) return e;
  const int bx = std::min(304, (npts + kBrPoints - 1) / kBrPoints);
  k_mbj_x<<<bx, 4 * kBrPoints, 0, s>>>(rho, part, nchunk, n[0], n[1], n[2], periodic, h[0], h[1], h[2], fd, c_fixed,
                                       partials, ticket, c_dev, V);
  e = cudaGetLastError();
  int nl = 2;
  if (e == cudaSuccess && !(c_fixed > 0.0)) {
    k_mbj_apply<<<(npts + 127) / 128, 128, 0, s>>>(rho, part, npts, c_dev, V);
    e = cudaGetLastError();
    nl = 3;
  }
  if (nlaunch) *nlaunch = nl;
  return e;
}

template cudaError_t launch_mbj<float>(const float2*, int, int, const int*, int, const double*, const double*,
                                       const double*, const double*, double, double*, int, double*, unsigned*, double*,
                                       double*, cudaStream_t, int*);
template cudaError_t launch_mbj<double>(const double2*, int, int, const int*, int, const double*, const double*,
                                        const double*, const double*, double, double*, int, double*, unsigned*,
                                        double*, double*, cudaStream_t, int*);

}  // namespace tdks
