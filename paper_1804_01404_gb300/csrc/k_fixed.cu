// Taylor launches of FP64 orbitals in 64-bit fixed point.
//
// FP64 arithmetic is the bound of the FP64 cell kernels: one DFMA holds a scheduler of this GPU for 70
// cycles, an integer instruction for 1 to 4 (measured with chains of each).  Here an orbital is propagated
// as 64-bit integers, X = round(u 2^s), with s chosen from the largest |Re u|, |Im u| of the orbital so that
// |X| < 2^59; the last bit is 2^-59 of that maximum, finer than the FP64 rounding of every value within 64
// times of it.  Values, differences and products:
//   * X = h 2^31 + l with |l| <= 2^30 (two 32-bit digits; sums and differences of neighbours are digit
//     sums without carries);
//   * the 8th-order weights are small integers over a common denominator (D2: 8064, -1008, 128, -9 over
//     5040 with centre -14350; D1: 672, -168, 32, -3 over 840), so the weighted sums are exact;
//   * each axis sum is then multiplied once by a 57-bit coefficient dt/(2 h^2) ... as digits
//     c = (ch 2^28 + cl) 2^-57: three multiply-adds into accumulators shared by all terms of the point.
// A stage takes about 800 instructions per 32 points (multiply-adds at a quarter rate bound it: 64 % of the heavy FMA
// pipe) against 7000 cycles for its 100 FP64 instructions.  One Taylor step of 1024 orbitals of 20^3: 7.00 ms in
// FP64, 1.48 here (the launch 1.47, with the orbital written, the density and the current 1.85); of 8 orbitals of 16^3:
// 500 us and 48 (the launch 36, and 51).  Error of one step against 113-bit arithmetic, l2 over an orbital, 20^3 and
// 16^3: 5.3e-17 and 5.9e-17 relative (the rounding of the result to FP64); the FP64 kernel 1.0e-16 and 6.2e-17; the
// largest error at any point is also the smaller of the two on seven grids.  The unit is one for a whole orbital, so
// that single values below 2^-6 of the largest are less exact than in FP64, by 2^6 at the limit of kFxRange.  The density
// is right to FP64 rounding of the values at every point; the current is 9e-18 of the density off on average (36 steps of
// six cells), the FP64 kernel's 1.1e-17.
//
// An orbital is spread over a cluster of 1, 2, 4 or 8 CTAs, each owning a slab of planes in three
// shared-memory copies (psi and two Horner vectors); the four planes above and below a slab are read from
// the neighbours' shared memory.  So the copies always fit, few orbitals still use many SMs, and a stage
// takes two cluster barriers: after the local pass (with the partial projections, which every CTA sends to
// every other) and after the nonlocal scatter.
//
// Ranges: |X| < 2^60 after every stage, checked at every point; an orbital that leaves it (an unstable
// step), holds a non-finite value, decays into a vacuum (kFxRange), or meets a potential or a wave vector outside
// the range of the coefficients writes nothing but its flag, and the FP64 kernel propagates it (launched after this one;
// its CTAs return at once for the others: 3 us for 8 orbitals, 6 us for 1024).
#include <cuda_runtime.h>

#include <cmath>
#include <cstdint>

#include "fixed.h"
#include "warp_sum.cuh"

namespace tdks {

namespace {

constexpr int kFxThreads = 512;
constexpr int kFxStaticReserve = 4 * 1024;
// Orbitals with a block of 4 x 4 x 4 points all 2^12 below their largest value go to the FP64 kernel: they decay
// into a vacuum, where an FP64 stencil is right to 2^-53 of its own neighbours and a unit here is 2^-59 of the
// largest value anywhere.  Down to 2^-12 a unit changes the exchange potential (the cube root of |u|^2) by less than
// 2^-55 of the largest; low-pass orbitals of 9^3 to 20^3 cells and boxes have blocks of 2^-2 to 2^-9.
constexpr int kFxRange = 12;

using ll = long long;

__device__ __forceinline__ ll mw(int a, int b, ll c) { return (ll)a * b + c; }

// digits of a 64-bit value: x = h 2^31 + l, l in [-2^30, 2^30)
__device__ __forceinline__ int2 digits31(ll x) {
  const int l = ((int)((unsigned)x << 1)) >> 1;
  return make_int2((int)((x - l) >> 31), l);
}
__device__ __forceinline__ ll join31(int h, int l) { return ((ll)h << 31) + l; }
// digits of a coefficient: c = h 2^28 + l, l in [-2^27, 2^27)
__host__ __device__ inline int2 digits28(ll c) {
  const ll h = (c + (1LL << 27)) >> 28;
  return int2{(int)h, (int)(c - (h << 28))};
}
// x >> SH (rounded) in digits of 27 bits, for products that are summed over many points
template <int SH>
__device__ __forceinline__ int2 digits27(ll x) {
  const ll y = (x + (1 << (SH - 1))) >> SH;
  const int l = ((int)((unsigned)y << 5)) >> 5;
  return make_int2((int)((y - l) >> 27), l);
}

// Sum of products p c, p = ph 2^31 + pl, c = ch 2^28 + cl: the product of the low digits (below the last
// bit of the result after the shift by 57) is left out.
struct Acc3 {
  ll a1 = 0, a2 = 1LL << 25, a3 = 1LL << 28;     // half a unit each: the shifts of value57 round
  __device__ __forceinline__ void add(int ph, int pl, int2 c) {
    a1 = mw(ph, c.x, a1);
    a2 = mw(ph, c.y, a2);
    a3 = mw(pl, c.x, a3);
  }
  __device__ __forceinline__ void add64(ll z, int2 c) { add((int)(z >> 31), (int)(z & 0x7fffffff), c); }
  __device__ __forceinline__ ll value57() const { return (a1 << 2) + (a2 >> 26) + (a3 >> 29); }
};

// ... with the low product, for the projectors' coarser coefficients
struct Acc4 {
  ll a1 = 0, a2 = 0, a3 = 0, a4 = 0;
  __device__ __forceinline__ void add(int ph, int pl, int ch, int cl) {
    a1 = mw(ph, ch, a1);
    a2 = mw(ph, cl, a2);
    a3 = mw(pl, ch, a3);
    a4 = mw(pl, cl, a4);
  }
  // 31 < sh < 59.  Rounded: every lane of every CTA gives one value of a projection, and 256 floors of its three lower
  // sums were a bias of 400 units, 3e-17 of the density in the current.
  __device__ __forceinline__ ll value(int sh) const {
    const ll t = a2 + ((a3 + (a4 >> 28)) >> 3);
    return (a1 << (59 - sh)) + ((t + (1LL << (sh - 32))) >> (sh - 31));
  }
};

// FP64 -> fixed point for a largest exponent field e: values below 2^(e - 1022) become |X| < 2^59
__device__ __forceinline__ ll to_fixed(double v, int e) {
  const int hi = __double2hiint(v), ef = (hi >> 20) & 0x7ff;
  ll m = ((ll)((hi & 0xfffff) | 0x100000) << 32) | (unsigned)__double2loint(v);
  if (ef == 0) m = 0;
  const int sh = 6 - (e - ef);
  ll r;
  if (sh >= 0) r = m << sh;
  else {
    const int k = min(-sh, 60);
    r = (m + (1LL << (k - 1))) >> k;
  }
  return hi < 0 ? -r : r;
}
__device__ __forceinline__ double to_double(ll x, int s) {   // x 2^-s
  if (x == 0) return 0.0;
  const double d = __ll2double_rn(x);
  return __hiloint2double(__double2hiint(d) - s * (1 << 20), __double2loint(d));
}
__device__ __forceinline__ double pow2d(int k) { return __hiloint2double((1023 + k) << 20, 0); }

// t / m of a Taylor stage (m = 4, 3, 2, 1), rounded
__device__ __forceinline__ ll div_stage(ll t, int m, int2 third) {
  if (m == 4) return (t + 2) >> 2;
  if (m == 2) return (t + 1) >> 1;
  if (m == 1) return t;
  Acc3 a;
  a.add64(t, third);
  return a.value57();
}

__device__ __forceinline__ unsigned smem_addr(const void* p) { return (unsigned)__cvta_generic_to_shared(p); }
__device__ __forceinline__ unsigned cluster_rank() { unsigned r; asm volatile("mov.u32 %0, %%cluster_ctarank;" : "=r"(r)); return r; }
__device__ __forceinline__ unsigned map_cta(unsigned addr, unsigned rank) {
  unsigned r;
  asm volatile("mapa.shared::cluster.u32 %0, %1, %2;" : "=r"(r) : "r"(addr), "r"(rank));
  return r;
}
__device__ __forceinline__ void cluster_sync() {
  asm volatile("barrier.cluster.arrive.release.aligned;\nbarrier.cluster.wait.acquire.aligned;" ::: "memory");
}
__device__ __forceinline__ int4 ld_cluster(unsigned addr) {
  int4 v;
  asm volatile("ld.shared::cluster.v4.s32 {%0, %1, %2, %3}, [%4];" : "=r"(v.x), "=r"(v.y), "=r"(v.z), "=r"(v.w) : "r"(addr) : "memory");
  return v;
}
__device__ __forceinline__ void st_cluster64(unsigned addr, ll v) {
  asm volatile("st.shared::cluster.s64 [%0], %1;" ::"r"(addr), "l"(v) : "memory");
}
__device__ __forceinline__ void st_cluster32(unsigned addr, unsigned v) {
  asm volatile("st.shared::cluster.u32 [%0], %1;" ::"r"(addr), "r"(v) : "memory");
}
__device__ __forceinline__ int4 isum(int4 a, int4 b) { return make_int4(a.x + b.x, a.y + b.y, a.z + b.z, a.w + b.w); }


// Weighted sums of the neighbour pairs of one point, per part: the weights come from the argument block
// (constant bank), which keeps every product one multiply-add (a literal power of two becomes four shifts
// and adds).
struct LapSum {
  ll h0 = 0, l0 = 0, h1 = 0, l1 = 0;
  __device__ __forceinline__ void add(int4 p, int4 q, int w) {
    h0 = mw(p.x + q.x, w, h0);
    l0 = mw(p.y + q.y, w, l0);
    h1 = mw(p.z + q.z, w, h1);
    l1 = mw(p.w + q.w, w, l1);
  }
  __device__ __forceinline__ void get(ll v[2]) const {      // sum w2 (u+ + u-) >> 15
    v[0] = (h0 << 16) + (l0 >> 15);
    v[1] = (h1 << 16) + (l1 >> 15);
  }
};
struct DerSum {
  ll h0 = 0, l0 = 0, h1 = 0, l1 = 0;
  __device__ __forceinline__ void add(int4 p, int4 q, int w) {
    h0 = mw(p.z - q.z, w, h0);
    l0 = mw(p.w - q.w, w, l0);
    h1 = mw(q.x - p.x, w, h1);
    l1 = mw(q.y - p.y, w, l1);
  }
  // (sum w1 (u+ - u-).im, sum w1 (u- - u+).re) >> 11, the two parts of -i q D1 u
  __device__ __forceinline__ void get(ll v[2]) const {
    v[0] = (h0 << 20) + (l0 >> 11);
    v[1] = (h1 << 20) + (l1 >> 11);
  }
};

// x >> 4 (rounded, |x| < 2^60) in digits of 28 bits: 56 bits of an orbital's largest value.  Rounding half up lifts
// the mean by half a unit of x, which for the derivative sums meets the half unit their floor (DerSum::get) took.
__device__ __forceinline__ int2 digits28s(ll x) {
  const ll y = (x + 8) >> 4;
  const int l = ((int)((unsigned)y << 4)) >> 4;
  return make_int2((int)((y - l) >> 28), l);
}
// Sums over points of |u|^2 and Im(conj(u) D1_a u), of u >> 4 and the scaled D1 >> 4, as the three sums of digit
// products: 2^56 v[0] + 2^28 v[1] + v[2] (the norm's middle one twice).  A product of digits is below 2^56 and a point
// adds at most four, so that 32 points of a thread stay in 64 bits; parts() then carries, and the sums over
// threads are exact.
struct ObsAcc {
  ll n[3] = {0, 0, 0}, j[3][3] = {{0, 0, 0}, {0, 0, 0}, {0, 0, 0}};
  __device__ __forceinline__ void norm(int2 ux, int2 uy) {
    n[0] = mw(ux.x, ux.x, mw(uy.x, uy.x, n[0]));
    n[1] = mw(ux.x, ux.y, mw(uy.x, uy.y, n[1]));
    n[2] = mw(ux.y, ux.y, mw(uy.y, uy.y, n[2]));
  }
  __device__ __forceinline__ void cur(int a, int2 ux, int2 uy, const ll der[2]) {
    const int2 d0 = digits28s(der[0]), d1 = digits28s(der[1]);
    j[a][0] = mw(ux.x, d0.x, mw(uy.x, d1.x, j[a][0]));
    j[a][1] = mw(ux.x, d0.y, mw(ux.y, d0.x, mw(uy.x, d1.y, mw(uy.y, d1.x, j[a][1]))));
    j[a][2] = mw(ux.y, d0.y, mw(uy.y, d1.y, j[a][2]));
  }
  // 2^56 v0 + 2^28 v1 + v2 = 2^84 t[0] + 2^56 t[1] + 2^28 t[2] + t[3], 0 <= t[1], t[2], t[3] < 2^28
  static __device__ __forceinline__ void parts(ll v0, ll v1, ll v2, ll* t) {
    const ll mask = (1 << 28) - 1;
    t[3] = v2 & mask;
    v1 += v2 >> 28;
    t[2] = v1 & mask;
    v0 += v1 >> 28;
    t[1] = v0 & mask;
    t[0] = v0 >> 28;
  }
};

}  // namespace

// Potential digits dt V (|dt V| < 1; a value outside flags its cell, whose orbitals then return before their first
// stage), phase factors exp(i q.d) of every (cell, k) and
// sphere entry: q = k + A' of the step (ph) and of its observables (pho, nullable).  One launch before
// the orbitals: 7 us of sincos for 64 k and 1018 entries, which each of the norb orbitals of a k would
// otherwise repeat (32 k cycles each).
__global__ void __launch_bounds__(128) k_fx_prep(FxArgs a) {
  const ll nv = (ll)a.npts * (a.vstride ? a.ncell : 1);
  const ll nph = (ll)a.nk * a.nsph * (a.phstride ? a.ncell : 1);
  const ll tot = nv + nph * (a.obs && a.natom ? 2 : 1);
  for (ll i = (ll)blockIdx.x * blockDim.x + threadIdx.x; i < tot; i += (ll)gridDim.x * blockDim.x) {
    if (i < nv) {
      const double v = a.V64[i] * a.dt;
      const bool in = fabs(v) < 1.0;
      a.V[i] = in ? digits28(__double2ll_rn(v * 144115188075855872.0)) : make_int2(0, 0);
      if (!in) a.vbad[a.vstride ? i / a.npts : 0] = 1;
      continue;
    }
    ll j = i - nv;
    const bool ob = j >= nph;
    if (ob) j -= nph;
    const int e = (int)(j % a.nsph);
    const int kk = (int)(j / a.nsph), cell = kk / a.nk, k = kk - cell * a.nk;
    const double* ac = ob ? a.Ap_obs_cell : a.Ap_cell;
    double arg = 0.0;
#pragma unroll
    for (int d = 0; d < 3; ++d) {
      const double A = ac ? ac[3 * cell + d] : (ob ? a.Ap_obs[d] : a.Ap[d]);
      arg += (a.kpts[3 * k + d] + A) * a.sph_d[3 * e + d];
    }
    double s, c;
    sincos(arg, &s, &c);
    const int2 dc = digits28(__double2ll_rn(c * 144115188075855872.0));
    const int2 ds = digits28(__double2ll_rn(s * 144115188075855872.0));
    (ob ? a.pho : a.ph)[j] = make_int4(dc.x, dc.y, ds.x, ds.y);
  }
}

namespace {

// Partial projections of this CTA's planes, one warp per (atom, moment): part[job * 8 + 2 p + (0: Re, 1: Im)]
// = sum_i beta_ip d_i^(j) ph_i v_i 2^(Kb - 4 - sN) over the slab's sphere points, sent to CTA `dst` (all:
// every CTA of the cluster).  NJ = 4: moments 1, d_x, d_y, d_z (the displacements scaled by 2^(Kd - 57)).
template <int NJ>
__device__ __forceinline__ void fx_project(const FxArgs& a, const int4* cur, int pbase, const int4* ph, ll* part, int rank,
                                           int ncta, bool all) {
  const int lane = threadIdx.x & 31, warp = threadIdx.x >> 5, nw = blockDim.x >> 5;
  const int jobs = a.natom * NJ;
  for (int job = warp; job < jobs; job += nw) {
    const int at = job / NJ, j = job - at * NJ;
    const int2 r = a.ent_rng[rank * a.natom + at];
    Acc4 acc[8];
    for (int i = r.x + lane; i < r.y; i += 32) {
      const int4 u = cur[a.sph_sidx[i] - pbase];
      const int4 f = ph[i];
      const int2 fc = make_int2(f.x, f.y), fs = make_int2(f.z, f.w);
      Acc3 tr, ti;
      tr.add(u.x, u.y, fc);
      tr.add(-u.z, -u.w, fs);
      ti.add(u.x, u.y, fs);
      ti.add(u.z, u.w, fc);
      ll re = tr.value57(), im = ti.value57();
      if (NJ > 1 && j > 0) {
        const int2 dd = a.sph_dfx[3 * i + j - 1];
        Acc3 dr, di;
        dr.add64(re, dd);
        di.add64(im, dd);
        re = dr.value57();
        im = di.value57();
      }
      const int2 pr = digits31((re + 8) >> 4), pi = digits31((im + 8) >> 4);
      const int4 b01 = a.beta[2 * i], b23 = a.beta[2 * i + 1];
      acc[0].add(pr.x, pr.y, b01.x, b01.y);
      acc[1].add(pi.x, pi.y, b01.x, b01.y);
      acc[2].add(pr.x, pr.y, b01.z, b01.w);
      acc[3].add(pi.x, pi.y, b01.z, b01.w);
      acc[4].add(pr.x, pr.y, b23.x, b23.y);
      acc[5].add(pi.x, pi.y, b23.x, b23.y);
      acc[6].add(pr.x, pr.y, b23.z, b23.w);
      acc[7].add(pi.x, pi.y, b23.z, b23.w);
    }
    ll v[8];
#pragma unroll
    for (int q = 0; q < 8; ++q) v[q] = acc[q].value(a.sN);
    const ll t = warp_split_sum<8>(v);             // lane L: total of value L >> 2
    if ((lane & 3) == 0) {
      const unsigned loc = smem_addr(part + (size_t)rank * jobs * 8 + job * 8 + (lane >> 2));
      for (int c = 0; c < (all ? ncta : 1); ++c) st_cluster64(map_cta(loc, c), t);
    }
  }
}

// J_nl of the orbital from the cluster's partial moments (CTA 0): sum over atoms and projectors of
// 2 E_p Im(conj(b^(d)) c) dV^2; warp d takes the component d.
__device__ __forceinline__ void fx_nonlocal_current(const FxArgs& a, const ll* part, int ncta, int s, double* jnl) {
  const int lane = threadIdx.x & 31, d = threadIdx.x >> 5;
  if (d >= 3) return;
  const int jobs = a.natom * 4;
  double sum = 0.0;
  for (int ap = lane; ap < jobs; ap += 32) {
    const int at = ap >> 2, p = ap & 3;
    ll v[4] = {0, 0, 0, 0};
    for (int r = 0; r < ncta; ++r) {
      const ll* pc = part + (size_t)r * jobs * 8 + (size_t)(at * 4) * 8 + 2 * p;
      v[0] += pc[0];
      v[1] += pc[1];
      v[2] += pc[8 * (d + 1)];
      v[3] += pc[8 * (d + 1) + 1];
    }
    const double im = (double)v[2] * (double)v[1] - (double)v[3] * (double)v[0];
    sum += im * a.jfac[at * 4 + p];
  }
#pragma unroll
  for (int o = 16; o > 0; o >>= 1) sum += __shfl_xor_sync(0xffffffffu, sum, o);
  if (lane == 0) {
    const double f = pow2d(-s);
    jnl[d] = sum * f * f;
  }
}

}  // namespace

// OBS: 0 none, 1 norm and current of the propagated orbital, 2 of the input orbital (periodic cells).
// ISO: equal spacings, the neighbours of all axes enter one Laplacian sum.  ZL: planes of a column segment.
template <bool PER, int OBS, bool ISO, int ZL>
__global__ void __launch_bounds__(kFxThreads, 1) k_cell_fx(FxArgs a) {
  extern __shared__ __align__(16) unsigned char fx_smem[];
  __shared__ unsigned s_max[8], s_min[8], s_flag[8];
  __shared__ unsigned s_wmax[kFxThreads / 32];
  __shared__ int2 s_cd[3], s_diag;
  __shared__ int s_cbad;
  __shared__ double s_qo[3], s_jnl[3], s_obs[8][4];
  __shared__ ll s_red[kFxThreads / 32][16];
  const int tid = threadIdx.x, lane = tid & 31, warp = tid >> 5;
  const int ncta = a.ncta, rank = ncta > 1 ? (int)cluster_rank() : 0;
  // every CTA of the cluster has started before the first write to its shared memory (waited for below)
  if (ncta > 1) asm volatile("barrier.cluster.arrive.release.aligned;" ::: "memory");
  const int orb = blockIdx.x / ncta;
  const int nxy = a.nx * a.ny, ps = a.pstride;
  const int zbeg = min(a.nz, rank * a.zl), zend = min(a.nz, zbeg + a.zl);
  const int pbase = rank * a.zl * ps, slab = a.zl * ps;
  int4* buf = reinterpret_cast<int4*>(fx_smem);
  ll* part = reinterpret_cast<ll*>(buf + 3 * slab);
  ll* parto = part + (size_t)ncta * a.natom * 8;
  int4* ec = reinterpret_cast<int4*>(parto + (OBS ? (size_t)ncta * a.natom * 32 : 0));
  unsigned* paddr = reinterpret_cast<unsigned*>(ec + a.natom * 4);   // [nz + 8] planes -4 .. nz + 3
  const int cell = orb / (a.nk * a.norb);
  const int k = (orb - cell * a.nk * a.norb) / a.norb;
  const double2* psi = a.psi_in + (size_t)orb * a.npts;
  const int2* Vc = a.V + (size_t)cell * a.vstride;
  const int4* ph = a.ph + (size_t)cell * a.phstride + (size_t)k * a.nsph;
  const int4* pho = OBS ? a.pho + (size_t)cell * a.phstride + (size_t)k * a.nsph : nullptr;
  const int2 third = digits28(48038396025285291LL);

  // the slab as FP64 into the first copy, its largest exponent, a copy for a fallback (predicted steps)
  const int vbad = tid == 0 ? a.vbad[a.vstride ? cell : 0] : 0;
  unsigned mx = 0;
  const int nown = (zend - zbeg) * nxy;
  double2* raw = reinterpret_cast<double2*>(buf);
  unsigned* grp = reinterpret_cast<unsigned*>(buf + slab);   // largest magnitude of four consecutive points (copy 1)
  for (int b0 = tid; b0 < ((nown + 31) & ~31); b0 += 4 * blockDim.x) {
    double2 u[4];
#pragma unroll
    for (int j = 0; j < 4; ++j) {
      const int i = b0 + j * (int)blockDim.x;
      u[j] = i < nown ? psi[zbeg * nxy + i] : double2{0.0, 0.0};
    }
#pragma unroll
    for (int j = 0; j < 4; ++j) {
      const int i = b0 + j * (int)blockDim.x;
      unsigned m = max((unsigned)__double2hiint(u[j].x) & 0x7fffffffu, (unsigned)__double2hiint(u[j].y) & 0x7fffffffu);
      if (i < nown) {
        raw[PER ? i : (i / nxy) * ps + i % nxy] = u[j];
        if (a.backup) a.backup[(size_t)orb * a.npts + zbeg * nxy + i] = u[j];
      }
      m = max(m, __shfl_xor_sync(0xffffffffu, m, 1));
      m = max(m, __shfl_xor_sync(0xffffffffu, m, 2));
      if ((tid & 3) == 0 && i < nown) grp[i >> 2] = m;
      mx = max(mx, m);
    }
  }
  mx = __reduce_max_sync(0xffffffffu, mx);
  if (lane == 0) s_wmax[warp] = mx;
  // wave vector of the step: coefficient digits of q.D1 and of the diagonal
  if (tid == 0) {
    double q2 = 0.0, bound = a.lap_bound;
    const double* Ac = a.Ap_cell ? a.Ap_cell + 3 * cell : a.Ap;
    for (int d = 0; d < 3; ++d) {
      const double q = a.kpts[3 * k + d] + Ac[d];
      const double c = PER ? q * a.der_fac[d] : 0.0;
      q2 += q * q;
      bound += fabs(c);
      s_cd[d] = digits28(fabs(c) < 2.0 ? __double2ll_rn(c * 144115188075855872.0) : 0);
    }
    const double dg = (a.diag + 0.5 * q2) * a.dt;
    bound += fabs(dg);
    s_cbad = !(bound < 4.1) || fabs(dg) >= 3.0 || vbad;   // (with |dt V| < 1 a digit holds the sum)
    s_diag = digits28(s_cbad ? 0 : __double2ll_rn(dg * 144115188075855872.0));
    if (OBS) {
      const double* Ao = a.Ap_obs_cell ? a.Ap_obs_cell + 3 * cell : a.Ap_obs;
      for (int d = 0; d < 3; ++d) s_qo[d] = a.kpts[3 * k + d] + Ao[d];
    }
  }
  for (int i = tid; i < a.nz + 8; i += blockDim.x) {
    int z = i - 4;
    if (PER) z += z < 0 ? a.nz : (z >= a.nz ? -a.nz : 0);
    unsigned ad = 0;
    if (z >= 0 && z < a.nz) {
      const int owner = z / a.zl;
      const unsigned loc = smem_addr(buf + (z - owner * a.zl) * ps);
      ad = ncta > 1 ? map_cta(loc, owner) : loc;
    }
    paddr[i] = ad;
  }
  __syncthreads();
  if (ncta > 1) asm volatile("barrier.cluster.wait.acquire.aligned;" ::: "memory");
  if (warp == 0) {
    // the smallest largest value of a block: four rows of four planes (of the slab; the last rows and planes where they
    // do not divide by four) and a group of each row, the group of its x-th point
    unsigned mn = 0x7fffffffu;
    const int nbx = a.nx % 4 == 0 ? a.nx / 4 : (a.nx + 2) / 4 + 1, nby = (a.ny + 3) / 4, nzl = zend - zbeg;
#pragma unroll 2
    for (int b = lane; b < nbx * nby * ((nzl + 3) / 4); b += 32) {
      const int r = b / nbx, bz = r / nby, x = min(4 * (b - r * nbx), a.nx - 1);
      const int y0 = min(4 * (r - bz * nby), a.ny - 4), z0 = max(min(4 * bz, nzl - 4), 0);
      unsigned m = 0;
#pragma unroll
      for (int j = 0; j < 16; ++j) m = max(m, grp[(min(z0 + (j >> 2), nzl - 1) * nxy + (y0 + (j & 3)) * a.nx + x) >> 2]);
      mn = min(mn, m);
    }
    unsigned w = lane < (int)(blockDim.x >> 5) ? s_wmax[lane] : 0u;
    w = __reduce_max_sync(0xffffffffu, w);
    mn = __reduce_min_sync(0xffffffffu, mn);
    if (lane < ncta) {
      if (ncta > 1) {
        st_cluster32(map_cta(smem_addr(&s_max[rank]), lane), w);
        st_cluster32(map_cta(smem_addr(&s_min[rank]), lane), mn);
      } else {
        s_max[0] = w;
        s_min[0] = mn;
      }
    }
  }
  if (ncta > 1) cluster_sync(); else __syncthreads();
  unsigned mn = 0x7fffffffu;
  mx = 0;
  for (int r = 0; r < ncta; ++r) {
    mx = max(mx, s_max[r]);
    mn = min(mn, s_min[r]);
  }
  int e = (int)(mx >> 20);
  unsigned bad = s_cbad;
  if (mx == 0) e = 1023;
  else if (e < 600 || e > 1450 || e - (int)(mn >> 20) > kFxRange) bad = 1;
  if (bad) {                                       // (the same in every CTA of the cluster)
    if (rank == 0 && tid == 0) a.need[orb] = 1;
    return;
  }
  const int s = 58 - (e - 1023);
  for (int i = tid; i < nown; i += blockDim.x) {
    const int li = PER ? i : (i / nxy) * ps + i % nxy;
    const double2 u = raw[li];
    const int2 x = digits31(to_fixed(u.x, e)), y = digits31(to_fixed(u.y, e));
    buf[li] = make_int4(x.x, x.y, y.x, y.y);
  }
  if (!PER)
    for (int i = tid; i < 3 * a.zl; i += blockDim.x) buf[i * ps + nxy] = make_int4(0, 0, 0, 0);
  if (ncta > 1) cluster_sync(); else __syncthreads();

  const unsigned bufbytes = (unsigned)slab * sizeof(int4);
  ObsAcc oa;
  if (OBS == 2 && a.natom > 0) fx_project<4>(a, buf, pbase, pho, parto, rank, ncta, false);
  // copy 0 keeps psi; the stages alternate between copies 1 and 2
#pragma unroll 1
  for (int st = 0; st < 4; ++st) {
    const int m = 4 - st;
    const int4* v = buf + (st == 0 ? 0 : (st == 2 ? 2 : 1)) * slab;
    int4* nxt = buf + (st & 1 ? 2 : 1) * slab;
    const unsigned zoff = (unsigned)(st == 0 ? 0 : (st == 2 ? 2 : 1)) * bufbytes;
    if (a.natom > 0) fx_project<1>(a, v, pbase, ph, part, rank, ncta, true);
    auto local_pass = [&](auto acc_tag) {
      constexpr bool ACC = decltype(acc_tag)::value;
#pragma unroll 1
      for (int item = tid; item < nxy * a.nseg; item += blockDim.x) {
        const int seg = item / nxy, col = item - seg * nxy;
        const int z0 = zbeg + seg * ZL, z1 = min(zend, z0 + ZL);
        if (z0 >= z1) continue;
        const int y = col / a.nx, x = col - y * a.nx;
        int ix[8], iy[8];                          // in-plane neighbours: +1, -1, +2, -2, ...
#pragma unroll
        for (int j = 1; j <= 4; ++j) {
          int xp = x + j, xm = x - j, yp = y + j, ym = y - j;
          if (PER) {
            xp -= xp >= a.nx ? a.nx : 0; xm += xm < 0 ? a.nx : 0;
            yp -= yp >= a.ny ? a.ny : 0; ym += ym < 0 ? a.ny : 0;
            ix[2 * j - 2] = y * a.nx + xp; ix[2 * j - 1] = y * a.nx + xm;
            iy[2 * j - 2] = yp * a.nx + x; iy[2 * j - 1] = ym * a.nx + x;
          } else {
            ix[2 * j - 2] = xp < a.nx ? y * a.nx + xp : nxy; ix[2 * j - 1] = xm >= 0 ? y * a.nx + xm : nxy;
            iy[2 * j - 2] = yp < a.ny ? yp * a.nx + x : nxy; iy[2 * j - 1] = ym >= 0 ? ym * a.nx + x : nxy;
          }
        }
        auto zload = [&](int z) -> int4 {          // plane z of this column, in this CTA or a neighbour
          if (z >= zbeg && z < zend) return v[(z - zbeg) * ps + col];
          const unsigned ad = paddr[z + 4];
          if (!PER && ad == 0) return make_int4(0, 0, 0, 0);
          return ld_cluster(ad + zoff + (unsigned)col * sizeof(int4));
        };
        int4 w[ZL + 8];                            // planes z0 - 4 .. z0 + ZL + 3
#pragma unroll
        for (int j = 0; j < 8; ++j) w[j] = zload(z0 - 4 + j);
#pragma unroll
        for (int zz = 0; zz < ZL; ++zz) {
          if (zz > 0 && z0 + zz >= z1) break;
          const int z = z0 + zz, loc = (z - zbeg) * ps;
          w[zz + 8] = zload(z + 4);
          const int4* p = v + loc;
          const int2 vd = Vc[z * nxy + col];
          Acc3 tx, ty;
          const int4 u = w[zz + 4];
          int2 ux, uy;
          if (ACC) {
            ux = digits28s(join31(u.x, u.y));
            uy = digits28s(join31(u.z, u.w));
            oa.norm(ux, uy);
          }
          LapSum lap;
#pragma unroll
          for (int ax = 0; ax < 3; ++ax) {
            DerSum der;
            if (!ISO && ax > 0) lap = LapSum{};
#pragma unroll
            for (int j = 0; j < 4; ++j) {
              const int4 up = ax == 0 ? p[ix[2 * j]] : (ax == 1 ? p[iy[2 * j]] : w[zz + 5 + j]);
              const int4 um = ax == 0 ? p[ix[2 * j + 1]] : (ax == 1 ? p[iy[2 * j + 1]] : w[zz + 3 - j]);
              lap.add(up, um, a.w2[j]);
              if (PER) der.add(up, um, a.w1[j]);
            }
            ll d[2];
            if (!ISO || ax == 2) {
              lap.get(d);
              tx.add64(d[0], a.lap[ax]);
              ty.add64(d[1], a.lap[ax]);
            }
            if (PER) {
              der.get(d);
              tx.add64(d[0], s_cd[ax]);
              ty.add64(d[1], s_cd[ax]);
              if (ACC) oa.cur(ax, ux, uy, d);
            }
          }
          const int2 dg = make_int2(vd.x + s_diag.x, vd.y + s_diag.y);
          tx.add(u.x, u.y, dg);
          ty.add(u.z, u.w, dg);
          // psi + (-i dt / m) H v
          const int4 p0 = buf[loc + col];
          const int2 dx = digits31(join31(p0.x, p0.y) + div_stage(ty.value57(), m, third));
          const int2 dy = digits31(join31(p0.z, p0.w) - div_stage(tx.value57(), m, third));
          bad |= ((unsigned)(dx.x + (1 << 29)) | (unsigned)(dy.x + (1 << 29))) >> 30;
          nxt[loc + col] = make_int4(dx.x, dx.y, dy.x, dy.y);
        }
      }
    };
    if (OBS == 2 && st == 0) local_pass(std::integral_constant<bool, true>{});
    else local_pass(std::integral_constant<bool, false>{});
    if (ncta > 1) cluster_sync(); else __syncthreads();
    if (OBS == 2 && st == 0 && rank == 0 && a.natom > 0) fx_nonlocal_current(a, parto, ncta, s, s_jnl);
    if (a.natom > 0) {
      for (int i = tid; i < a.natom * 8; i += blockDim.x) {
        ll t = 0;
        for (int r = 0; r < ncta; ++r) t += part[(size_t)r * a.natom * 8 + i];
        const double c = (double)t * (a.ecfac[i >> 1] * a.dt);
        if (!(fabs(c) < 1.0e18)) bad = 1;
        const int2 d = digits31(fabs(c) < 1.0e18 ? __double2ll_rn(c) : 0);
        reinterpret_cast<int2*>(ec)[i] = d;
      }
      __syncthreads();
      const int2 sr = a.sp_rng[rank];
      for (int q = sr.x + tid; q < sr.y; q += blockDim.x) {
        ll rx = 0, ry = 0;
        const int e1 = a.sp_off[q + 1];
        for (int ee = a.sp_off[q]; ee < e1; ++ee) {
          const int i = a.pt_ent[ee];
          const int4* ca = ec + a.ent_atom[i] * 4;
          const int4 b01 = a.beta[2 * i], b23 = a.beta[2 * i + 1];
          Acc4 gr, gi;
          gr.add(ca[0].x, ca[0].y, b01.x, b01.y); gi.add(ca[0].z, ca[0].w, b01.x, b01.y);
          gr.add(ca[1].x, ca[1].y, b01.z, b01.w); gi.add(ca[1].z, ca[1].w, b01.z, b01.w);
          gr.add(ca[2].x, ca[2].y, b23.x, b23.y); gi.add(ca[2].z, ca[2].w, b23.x, b23.y);
          gr.add(ca[3].x, ca[3].y, b23.z, b23.w); gi.add(ca[3].z, ca[3].w, b23.z, b23.w);
          const int2 dr = digits31(gr.value(a.Kb)), di = digits31(gi.value(a.Kb));
          const int4 f = ph[i];
          const int2 fc = make_int2(f.x, f.y), fs = make_int2(f.z, f.w);
          Acc3 tr, ti;                             // times conj(ph)
          tr.add(dr.x, dr.y, fc);
          tr.add(di.x, di.y, fs);
          ti.add(di.x, di.y, fc);
          ti.add(-dr.x, -dr.y, fs);
          rx += tr.value57();
          ry += ti.value57();
        }
        const int pg = a.sp_pt[q], zz = pg / nxy;
        int4* dst = nxt + (pg + zz * (ps - nxy) - pbase);
        const int4 o = *dst;
        const int2 dx = digits31(join31(o.x, o.y) + div_stage(ry, m, third));
        const int2 dy = digits31(join31(o.z, o.w) - div_stage(rx, m, third));
        bad |= ((unsigned)(dx.x + (1 << 29)) | (unsigned)(dy.x + (1 << 29))) >> 30;
        *dst = make_int4(dx.x, dx.y, dy.x, dy.y);
      }
      if (ncta > 1) cluster_sync(); else __syncthreads();
    }
  }

  // an orbital out of range anywhere in the cluster: flag only
  bad = __syncthreads_or(bad);
  if (ncta > 1) {
    if (tid < ncta) st_cluster32(map_cta(smem_addr(&s_flag[rank]), tid), bad);
    cluster_sync();
    bad = 0;
    for (int r = 0; r < ncta; ++r) bad |= s_flag[r];
  }
  if (rank == 0 && tid == 0) a.need[orb] = bad ? 1 : 0;
  if (bad) return;

  // final pass: the orbital, the density and (OBS 1) the observables of the propagated orbital
  const int4* v = buf + 2 * slab;
  const unsigned zoff = 2 * bufbytes;
  const double f1 = pow2d(-s);
  const double rfac = 2.0 * a.kw[k] * f1 * f1 * 576460752303423488.0;       // 2^59
  double2* out = a.write_out ? a.psi_out + (size_t)orb * a.npts : nullptr;
  double* rho = a.rho ? a.rho + (size_t)cell * a.npts : nullptr;
  for (int i = tid; i < nown; i += blockDim.x) {
    const int zz = i / nxy, col = i - zz * nxy, pg = zbeg * nxy + i;
    const int4 u = v[zz * ps + col];
    const ll X = join31(u.x, u.y), Y = join31(u.z, u.w);
    if (out) out[pg] = make_double2(to_double(X, s), to_double(Y, s));
    if (rho) {
      // |u|^2 2^2k from the values shifted up by their leading zeros, so that small values keep their digits
      // (LDA takes the cube root of the density)
      const int k2 = __clzll((X ^ (X >> 63)) | (Y ^ (Y >> 63))) - 4;
      const int2 ux = digits27<6>(X << k2), uy = digits27<6>(Y << k2);
      const ll P = mw(ux.x, ux.x, mw(uy.x, uy.x, 0)), Q = mw(ux.x, ux.y, mw(uy.x, uy.y, 1LL << 18));
      const ll R = mw(ux.y, ux.y, mw(uy.y, uy.y, 1LL << 46));
      const double d = __ll2double_rn((P << 7) + (Q >> 19) + (R >> 47));
      if (d != 0.0) atomicAdd(rho + pg, __hiloint2double(__double2hiint(d) - 2 * k2 * (1 << 20), __double2loint(d)) * rfac);
    }
    if (OBS == 1) {
      const int2 ux = digits28s(X), uy = digits28s(Y);
      oa.norm(ux, uy);
      const int y = col / a.nx, x = col - y * a.nx, z = zbeg + zz;
      const int4* p = v + zz * ps;
#pragma unroll
      for (int ax = 0; ax < 3; ++ax) {
        DerSum der;
#pragma unroll
        for (int j = 0; j < 4; ++j) {
          int4 n[2];
#pragma unroll
          for (int g = 0; g < 2; ++g) {
            const int c = (ax == 0 ? x : (ax == 1 ? y : z)) + (g ? -1 - j : 1 + j);
            const int len = ax == 0 ? a.nx : a.ny;
            if (ax == 2) {
              if (c >= zbeg && c < zend) n[g] = v[(c - zbeg) * ps + col];
              else n[g] = ld_cluster(paddr[c + 4] + zoff + (unsigned)col * sizeof(int4));
            } else {
              const int cw = c + (c < 0 ? len : (c >= len ? -len : 0));
              n[g] = p[ax == 0 ? y * a.nx + cw : cw * a.nx + x];
            }
          }
          der.add(n[0], n[1], a.w1[j]);
        }
        ll d[2];
        der.get(d);
        oa.cur(ax, ux, uy, d);
      }
    }
  }
  if (OBS == 0) return;
  if (OBS == 1 && a.natom > 0) fx_project<4>(a, v, pbase, pho, parto, rank, ncta, false);
  // sums of the CTA, then of the cluster (CTA 0): integers within a warp (below 2^53, so exact in FP64), FP64 from there
  ll t16[16];
  ObsAcc::parts(oa.n[0], 2 * oa.n[1], oa.n[2], t16);
#pragma unroll
  for (int d = 0; d < 3; ++d) ObsAcc::parts(oa.j[d][0], oa.j[d][1], oa.j[d][2], t16 + 4 * (d + 1));
  const ll tw = warp_split_sum<16>(t16);           // lane L: total of value L >> 1
  if ((lane & 1) == 0) s_red[warp][lane >> 1] = tw;
  __syncthreads();
  if (tid < 16) {                                  // value tid >> 2, part tid & 3
    const int q = tid & 3;
    double x = 0.0;
    for (int w = 0; w < (int)(blockDim.x >> 5); ++w) x += (double)s_red[w][tid];
    x *= pow2d(28 * (3 - q));
    x += __shfl_xor_sync(0xffffu, x, 1);
    x += __shfl_xor_sync(0xffffu, x, 2);
    if (q == 0) {
      if (ncta > 1) st_cluster64(map_cta(smem_addr(&s_obs[rank][tid >> 2]), 0), __double_as_longlong(x));
      else s_obs[0][tid >> 2] = x;
    }
  }
  if (ncta > 1) cluster_sync(); else __syncthreads();
  if (rank != 0) return;
  if (OBS == 1 && a.natom > 0) {
    fx_nonlocal_current(a, parto, ncta, s, s_jnl);
    __syncthreads();
  }
  if (tid < 8) {
    double x = 0.0, n = 0.0;
    for (int r = 0; r < ncta; ++r) {
      n += s_obs[r][0];
      if (tid >= 1 && tid < 4) x += s_obs[r][tid];
    }
    const double sc = f1 * f1 * pow2d(8);          // u >> 4, D1 >> 4
    n *= sc;
    double res = 0.0;
    if (tid == 0) res = n * a.dV;
    else if (tid < 4) res = (x * sc * a.obs_fac[tid - 1] + s_qo[tid - 1] * n) * a.dV;
    else if (tid < 7) res = a.natom > 0 ? s_jnl[tid - 4] : 0.0;
    a.obs[(size_t)orb * 8 + tid] = res;
  }
}

size_t fx_smem_bytes(int zl, int pstride, int nz, int natom, int ncta) {
  return sizeof(int4) * (3 * (size_t)zl * pstride + 4 * (size_t)natom) + sizeof(ll) * (size_t)ncta * natom * 40 +
         sizeof(unsigned) * (size_t)(nz + 8);
}

bool fx_split(int nx, int ny, int nz, int pstride, int natom, int norb_tot, int* ncta, int* zl, int* zlen, int* nseg) {
  // Cluster size and column segments by the issue cycles of a stage: a warp of 32 columns takes about
  // 500 cycles per plane and 150 more per segment (its z window and neighbour offsets), four schedulers
  // share the warps, and a stage adds about 3000 cycles of projections, scatter and barriers.  Times the
  // waves of orbitals.
  double best = 0.0;
  bool ok = false;
  for (int c = 1; c <= 8; c *= 2) {
    const int planes = (nz + c - 1) / c;
    if (c > nz || (c - 1) * planes >= nz) continue;            // a CTA without planes
    if (fx_smem_bytes(planes, pstride, nz, natom, c) + kFxStaticReserve > 224 * 1024) continue;
    const int waves = (norb_tot + (152 / c) - 1) / (152 / c);
    for (int L : {1, 2, 3, 5}) {
      const int segs = (planes + L - 1) / L;
      const int wi = (nx * ny * segs + 31) / 32;                // warp items
      const double cyc = ((wi + 3) / 4) * (500.0 * L + 150.0) + 3000.0;
      if (!ok || waves * cyc < best) {
        best = waves * cyc;
        *ncta = c; *zl = planes; *zlen = L; *nseg = segs;
        ok = true;
      }
    }
  }
  return ok;
}

template <bool PER, int OBS, bool ISO, int ZL>
static cudaError_t launch_fx_one(const FxArgs& a, size_t smem, cudaStream_t s) {
  auto kern = k_cell_fx<PER, OBS, ISO, ZL>;
  cudaError_t e = cudaFuncSetAttribute(kern, cudaFuncAttributeMaxDynamicSharedMemorySize, (int)smem);
  if (e != cudaSuccess) return e;
  cudaLaunchConfig_t cfg = {};
  cfg.gridDim = dim3((unsigned)(a.ncell * a.nk * a.norb * a.ncta));
  cfg.blockDim = dim3(kFxThreads);
  cfg.dynamicSmemBytes = smem;
  cfg.stream = s;
  cudaLaunchAttribute at[1];
  at[0].id = cudaLaunchAttributeClusterDimension;
  at[0].val.clusterDim.x = (unsigned)a.ncta;
  at[0].val.clusterDim.y = at[0].val.clusterDim.z = 1;
  cfg.attrs = at;
  cfg.numAttrs = 1;
  return cudaLaunchKernelEx(&cfg, kern, a);
}

template <bool PER, int OBS>
static cudaError_t launch_fx_obs(const FxArgs& a, size_t smem, cudaStream_t s) {
  const bool iso = a.lap[0].x == a.lap[1].x && a.lap[0].y == a.lap[1].y && a.lap[0].x == a.lap[2].x && a.lap[0].y == a.lap[2].y;
  switch (a.zlen) {
    case 1: return iso ? launch_fx_one<PER, OBS, true, 1>(a, smem, s) : launch_fx_one<PER, OBS, false, 1>(a, smem, s);
    case 2: return iso ? launch_fx_one<PER, OBS, true, 2>(a, smem, s) : launch_fx_one<PER, OBS, false, 2>(a, smem, s);
    case 3: return iso ? launch_fx_one<PER, OBS, true, 3>(a, smem, s) : launch_fx_one<PER, OBS, false, 3>(a, smem, s);
    default: return iso ? launch_fx_one<PER, OBS, true, 5>(a, smem, s) : launch_fx_one<PER, OBS, false, 5>(a, smem, s);
  }
}

cudaError_t launch_cell_fx(const FxArgs& a, bool periodic, bool obs_at_start, cudaStream_t s) {
  const ll work = (ll)a.npts * (a.vstride ? a.ncell : 1) + (ll)a.nk * a.nsph * (a.phstride ? a.ncell : 1) * (a.obs ? 2 : 1);
  const ll blocks = (work + 127) / 128;
  k_fx_prep<<<(unsigned)(blocks < 152 * 16 ? blocks : 152 * 16), 128, 0, s>>>(a);
  cudaError_t e = cudaGetLastError();
  if (e != cudaSuccess) return e;
  const size_t smem = fx_smem_bytes(a.zl, a.pstride, a.nz, a.natom, a.ncta);
  if (!periodic) return launch_fx_obs<false, 0>(a, smem, s);
  if (!a.obs) return launch_fx_obs<true, 0>(a, smem, s);
  return obs_at_start ? launch_fx_obs<true, 2>(a, smem, s) : launch_fx_obs<true, 1>(a, smem, s);
}

}  // namespace tdks
