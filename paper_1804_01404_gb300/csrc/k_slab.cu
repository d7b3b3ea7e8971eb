// Taylor launches of FP32 orbitals of any grid size in slabs over a thread-block cluster.
//
// The cell kernels (k_orbital.cu) hold an orbital in one SM: grids without a built-in size run one point per
// thread with run-time neighbour addresses (257 instructions per point and stage), at most one or two CTAs
// per SM, orbitals over half of shared memory pass every stage through a global scratch, and few orbitals
// leave most SMs idle.  The tile kernels (k_tile.cu) take three launches per Horner stage.  Here an
// orbital is spread over a cluster of 1 to 8 CTAs, each owning a slab of planes in two shared-memory
// copies, so that two CTAs of different orbitals share an SM where they fit and one's barriers and
// loads overlap the other's arithmetic; the four planes above and below a slab are read from the
// neighbours' shared memory.  A thread owns two x-adjacent points of a column segment (16-byte loads of row
// pairs, the z window in registers, segments unrolled).  Rows are padded to an even length: for an odd nx
// the pad of a periodic row repeats its first point (as a thread's second point it is computed from the same
// values, so it stays equal), the pad of an isolated row is zero.
// All four Horner stages run in one launch; a stage takes two cluster barriers: after the local pass
// (with the partial projections, which every CTA sends to every other) and after the nonlocal scatter.
//
// Taylor steps (with the projections, no density) in a chain, microseconds, without -> here: 32^3 isolated, 16 orbitals,
// 8 atoms 90 -> 55 (12 tile launches with a third of the SMs; now bound by the barriers and the latency of a
// stage); 24^3 periodic, 1024 orbitals, 3 atoms 709 -> 621 (its second copy no longer passes through scratch; bound by
// shared-memory loads and issue slots); 12^3, 1024 orbitals, 1 atom 103 -> 90; 32 x 28 x 28, 128 orbitals, 3 atoms
// 204 -> 156 (with the projectors' values in shared memory one CTA fits an SM instead of two: 204).  Not
// faster: 15 x 18 x 21, 324 orbitals, 4 atoms (125 -> 156: odd rows are read point by point), 20^3 with its size built in
// (217 -> 353).  No rule on sizes tells these apart, so a context times one launch of each and keeps the faster
// (tune_cell, tune_tile).
#include <cuda_runtime.h>

#include <algorithm>
#include <cstdint>
#include <type_traits>

#include "cell_dev.cuh"
#include "slab.h"
#include "warp_sum.cuh"

namespace tdks {

namespace {

constexpr int kSlabThreads = 256;
constexpr size_t kSlabHalfSm = 112 * 1024;       // dynamic shared memory with which two CTAs share an SM

__device__ __forceinline__ unsigned smem_addr(const void* p) { return (unsigned)__cvta_generic_to_shared(p); }
__device__ __forceinline__ unsigned map_cta(unsigned addr, unsigned rank) {
  unsigned r;
  asm volatile("mapa.shared::cluster.u32 %0, %1, %2;" : "=r"(r) : "r"(addr), "r"(rank));
  return r;
}
__device__ __forceinline__ void cluster_sync() {
  asm volatile("barrier.cluster.arrive.release.aligned;\nbarrier.cluster.wait.acquire.aligned;" ::: "memory");
}
__device__ __forceinline__ float4 ld_cluster(unsigned addr) {
  float4 v;
  asm volatile("ld.shared::cluster.v4.f32 {%0, %1, %2, %3}, [%4];" : "=f"(v.x), "=f"(v.y), "=f"(v.z), "=f"(v.w) : "r"(addr) : "memory");
  return v;
}
__device__ __forceinline__ void st_cluster(unsigned addr, float v) {
  asm volatile("st.shared::cluster.f32 [%0], %1;" ::"r"(addr), "f"(v) : "memory");
}
__device__ __forceinline__ void st_cluster(unsigned addr, double v) {
  asm volatile("st.shared::cluster.f64 [%0], %1;" ::"r"(addr), "d"(v) : "memory");
}

struct SlabSmem {
  float2* buf;        // [2][zl * ps]
  float4* beta;       // tables of the slab's sphere entries (beta only where it fits, SlabArgs::beta_smem)
  float2* ph;
  int* ix;            // point index in the slab; sign bit: not the first of the point's entries
  unsigned* lk;       // atom << 16 | 1 + next entry of the same point (0: none)
  float *part, *parto;  // [ncta][natom * 8], [ncta][natom * 32]
  float2* ec;         // [natom * 4]
  int* off;           // [natom + 1] the atoms' entries in the tables
  int* gof;           // [natom] entry in the grid's tables less the entry here
  unsigned* paddr;    // [nz + 8] planes -4 .. nz + 3 of the first copy
};

// phase factors exp(i q.d) of the slab's entries
__device__ __forceinline__ void slab_phases(const SlabArgs& A, const SlabSmem& L, int rank, const float q[3]) {
  const OrbArgs<float>& a = A.o;
  const int lane = threadIdx.x & 31, warp = threadIdx.x >> 5;
  for (int at = warp; at < a.natom; at += kSlabThreads / 32) {
    const int2 r = A.ent_rng[rank * a.natom + at];
    for (int i = r.x + lane; i < r.y; i += 32) {
      float s, c;
      sincosf(q[0] * a.sph_d[3 * i] + q[1] * a.sph_d[3 * i + 1] + q[2] * a.sph_d[3 * i + 2], &s, &c);
      L.ph[L.off[at] + i - r.x] = make_float2(c, s);
    }
  }
}

// Partial projections of this CTA's planes, one warp per (atom, moment, chunk of the atom's entries): sum_i
// beta_ip d_i^(j) ph_i v_i, sent to every CTA (all) or to CTA 0.  NJ = 4: moments 1, d_x, d_y, d_z, one chunk.
template <int NJ>
__device__ __forceinline__ void slab_project(const SlabArgs& A, const SlabSmem& L, const float2* v, float* part, int rank,
                                             bool all) {
  const OrbArgs<float>& a = A.o;
  const int nch = NJ == 1 ? A.nch : 1, per = NJ * nch;
  const int lane = threadIdx.x & 31, warp = threadIdx.x >> 5, jobs = a.natom * per;
  for (int job = warp; job < jobs; job += kSlabThreads / 32) {
    const int at = job / per, j = NJ == 1 ? 0 : job - at * per, ch = NJ == 1 ? job - at * per : 0;
    const int e0 = L.off[at], e1 = L.off[at + 1];
    const float4* bg = reinterpret_cast<const float4*>(a.sph_beta) + L.gof[at];
    const float* dj = NJ > 1 && j > 0 ? a.sph_d + 3 * (size_t)A.ent_rng[rank * a.natom + at].x + j - 1 : nullptr;
    float acc[8] = {0, 0, 0, 0, 0, 0, 0, 0};
#pragma unroll 2
    for (int i = e0 + 32 * ch + lane; i < e1; i += 32 * nch) {
      const float2 u = v[L.ix[i] & 0x7fffffff], f = L.ph[i];
      float re = u.x * f.x - u.y * f.y, im = u.x * f.y + u.y * f.x;
      if (NJ > 1 && j > 0) {
        const float d = dj[3 * (size_t)(i - e0)];
        re *= d;
        im *= d;
      }
      const float4 b = A.beta_smem ? L.beta[i] : bg[i];
      acc[0] += b.x * re; acc[1] += b.x * im;
      acc[2] += b.y * re; acc[3] += b.y * im;
      acc[4] += b.z * re; acc[5] += b.z * im;
      acc[6] += b.w * re; acc[7] += b.w * im;
    }
    const float t = warp_split_sum<8>(acc);        // lane L: total of acc[L >> 2]
    if ((lane & 3) == 0) {
      const unsigned loc = smem_addr(part + ((size_t)rank * jobs + job) * 8 + (lane >> 2));
      for (int c = 0; c < (all ? A.ncta : 1); ++c) st_cluster(map_cta(loc, c), t);
    }
  }
}

}  // namespace

// EVEN: nx is even (pairs of a row never straddle its ends) and the orbitals are 16-byte aligned.  OBS: 0 none,
// 1 norm and current of the propagated orbital, 2 of the input orbital (periodic cells).  ZL: planes of a
// column segment.
template <bool PER, bool EVEN, int OBS, int ZL>
__global__ void __launch_bounds__(kSlabThreads, 2) k_slab(SlabArgs A) {
  using M = CM<float>;
  extern __shared__ __align__(16) unsigned char slab_smem_raw[];
  __shared__ double s_jnl[3], s_obs[8][4];
  __shared__ FF s_red[4][kSlabThreads / 32];
  const OrbArgs<float>& a = A.o;
  const int tid = threadIdx.x, lane = tid & 31, warp = tid >> 5, ncta = A.ncta;
  int rank = 0;
  if (ncta > 1) {
    unsigned r;
    asm volatile("mov.u32 %0, %%cluster_ctarank;" : "=r"(r));
    rank = (int)r;
    // every CTA of the cluster has started before the first access to its shared memory (waited for below)
    asm volatile("barrier.cluster.arrive.release.aligned;" ::: "memory");
  }
  const int orb = blockIdx.x / ncta;
  const int nx = a.nx, ny = a.ny, nz = a.nz, nxy = nx * ny, nxp = A.nxp, hp = nxp >> 1, ps = A.ps;
  const int zbeg = min(nz, rank * A.zl), zend = min(nz, zbeg + A.zl), slab = A.zl * ps, pbase = rank * slab;
  SlabSmem L;
  L.buf = reinterpret_cast<float2*>(slab_smem_raw);
  L.beta = reinterpret_cast<float4*>(L.buf + 2 * slab);
  L.ph = reinterpret_cast<float2*>(L.beta + (A.beta_smem ? A.max_ent : 0));
  L.ec = L.ph + A.max_ent;
  L.part = reinterpret_cast<float*>(L.ec + 4 * a.natom);
  L.parto = L.part + ncta * a.natom * A.nch * 8;
  L.ix = reinterpret_cast<int*>(L.parto + (OBS ? ncta * a.natom * 32 : 0));
  L.lk = reinterpret_cast<unsigned*>(L.ix + A.max_ent);
  L.off = L.ix + 2 * A.max_ent;
  L.gof = L.off + a.natom + 1;
  L.paddr = reinterpret_cast<unsigned*>(L.gof + a.natom);
  const int cell = orb / (a.nk * a.norb), k = (orb - cell * a.nk * a.norb) / a.norb;
  const float2* psi = a.psi_in + (size_t)orb * a.npts;
  const float* Vc = a.V + (size_t)cell * a.vstride;
  const double* ap = a.Ap_cell ? a.Ap_cell + 3 * cell : a.Ap;
  float q[3];
#pragma unroll
  for (int d = 0; d < 3; ++d) q[d] = (float)(a.kpts[3 * k + d] + ap[d]);
  const float diag0 = a.c2x[0] + a.c2y[0] + a.c2z[0] + 0.5f * (q[0] * q[0] + q[1] * q[1] + q[2] * q[2]);
  float qo[3] = {q[0], q[1], q[2]};
  if (OBS) {
    const double* apo = a.Ap_obs_cell ? a.Ap_obs_cell + 3 * cell : a.Ap_obs;
#pragma unroll
    for (int d = 0; d < 3; ++d) qo[d] = (float)(a.kpts[3 * k + d] + apo[d]);
  }

  // set-up: the atoms' table ranges, plane addresses, zero pads
  if (tid == 0) {
    int o = 0;
    for (int at = 0; at < a.natom; ++at) {
      L.off[at] = o;
      const int2 r = A.ent_rng[rank * a.natom + at];
      L.gof[at] = r.x - o;
      o += r.y - r.x;
    }
    L.off[a.natom] = o;
  }
  for (int i = tid; i < nz + 8; i += kSlabThreads) {
    int z = i - 4;
    if (PER) z += z < 0 ? nz : (z >= nz ? -nz : 0);
    unsigned ad = 0;
    if (z >= 0 && z < nz) {
      const int owner = z / A.zl;
      const unsigned loc = smem_addr(L.buf + (z - owner * A.zl) * ps);
      ad = ncta > 1 ? map_cta(loc, owner) : loc;
    }
    L.paddr[i] = ad;
  }
  if (!PER)
    for (int i = tid; i < 2 * A.zl; i += kSlabThreads)
      *reinterpret_cast<float4*>(L.buf + i * ps + nxp * ny) = make_float4(0.f, 0.f, 0.f, 0.f);
  // the slab, pair by pair, four loads in flight (a predicted step also keeps a copy of its input)
  const int npair = (zend - zbeg) * ny * hp;
  float2* bk = a.backup ? a.backup + (size_t)orb * a.npts : nullptr;
  for (int b0 = tid; b0 < npair; b0 += 4 * kSlabThreads) {
    float2 u[4][2];
    int li[4], gi[4], two[4];
#pragma unroll
    for (int j = 0; j < 4; ++j) {
      const int i = b0 + j * kSlabThreads;
      const int row = i / hp, x = 2 * (i - row * hp), z = row / ny, y = row - z * ny;
      li[j] = z * ps + y * nxp + x;
      gi[j] = (zbeg + z) * nxy + y * nx + x;
      two[j] = i < npair ? (x + 1 < nx ? 2 : 1) : 0;
      u[j][0] = u[j][1] = make_float2(0.f, 0.f);
      if (two[j]) {
        if (EVEN) {
          const float4 v = *reinterpret_cast<const float4*>(psi + gi[j]);
          u[j][0] = lo2(v);
          u[j][1] = hi2(v);
        } else {
          u[j][0] = psi[gi[j]];
          if (two[j] == 2) u[j][1] = psi[gi[j] + 1];
          else if (PER) u[j][1] = psi[gi[j] - (nx - 1)];       // the pad repeats the row's first point
        }
      }
    }
#pragma unroll
    for (int j = 0; j < 4; ++j)
      if (two[j]) {
        *reinterpret_cast<float4*>(L.buf + li[j]) = make_float4(u[j][0].x, u[j][0].y, u[j][1].x, u[j][1].y);
        if (bk) {
          bk[gi[j]] = u[j][0];
          if (two[j] == 2) bk[gi[j] + 1] = u[j][1];
        }
      }
  }
  __syncthreads();
  for (int at = warp; at < a.natom; at += kSlabThreads / 32) {
    const int2 r = A.ent_rng[rank * a.natom + at];
    for (int i = r.x + lane; i < r.y; i += 32) {
      const int e = L.off[at] + i - r.x;
      const int2 ln = A.link[i];                   // next entry of the point (-1: none), whether this is the first
      L.ix[e] = (A.sidx[i] - pbase) | (ln.y ? 0 : (int)0x80000000u);
      unsigned nx1 = 0;
      if (ln.x >= 0) {
        const int an = a.ent_atom[ln.x];
        nx1 = 1u + (unsigned)(L.off[an] + ln.x - A.ent_rng[rank * a.natom + an].x);
      }
      L.lk[e] = ((unsigned)at << 16) | nx1;
      if (A.beta_smem) L.beta[e] = *reinterpret_cast<const float4*>(a.sph_beta + 4 * (size_t)i);
    }
  }
  slab_phases(A, L, rank, OBS == 2 ? qo : q);
  if (ncta > 1) {
    asm volatile("barrier.cluster.wait.acquire.aligned;" ::: "memory");
    cluster_sync();
  } else {
    __syncthreads();
  }
  if (OBS == 2 && a.natom > 0) {                   // nonlocal current of the input orbital
    slab_project<4>(A, L, L.buf, L.parto, rank, false);
    __syncthreads();
    slab_phases(A, L, rank, q);
    __syncthreads();
  }

  const unsigned bufbytes = (unsigned)slab * sizeof(float2);
  float os[4] = {0.f, 0.f, 0.f, 0.f};
#pragma unroll 1
  for (int st = 0; st < 4; ++st) {
    const float2* v = L.buf + (st & 1) * slab;
    float2* nxt = L.buf + (1 - (st & 1)) * slab;
    const unsigned zoff = (st & 1) ? bufbytes : 0u;
    const float coef = a.dt / (float)(4 - st);
    if (a.natom > 0) slab_project<1>(A, L, v, L.part, rank, true);
    auto local_pass = [&](auto acc_tag) {
      constexpr bool ACC = decltype(acc_tag)::value;
#pragma unroll 1
      for (int item = tid; item < hp * ny * A.nseg; item += kSlabThreads) {
        const int seg = item / (hp * ny), pc = item - seg * (hp * ny);
        const int z0 = zbeg + seg * ZL, z1 = min(zend, z0 + ZL);
        if (z0 >= z1) continue;
        const int y = pc / hp, x = 2 * (pc - y * hp), col = y * nxp + x, zero = nxp * ny;
        const bool pad = !EVEN && x + 1 >= nx;       // the second point is the row's pad
        const int gA = y * nx + x, gB = pad ? (PER ? y * nx : gA) : gA + 1;
        // in-plane offsets: x - 4 .. x - 1, x + 2 .. x + 5 (EVEN: the four pairs), rows y +- m
        int xo[EVEN ? 4 : 8], yo[8];
        auto wx = [&](int c) {
          if (PER) return y * nxp + c + (c < 0 ? nx : (c >= nx ? -nx : 0));
          return c < 0 || c >= nx ? zero : y * nxp + c;
        };
#pragma unroll
        for (int j = 0; j < (EVEN ? 4 : 8); ++j) xo[j] = wx(EVEN ? x + (j < 2 ? 2 * j - 4 : 2 * j - 2) : x + (j < 4 ? j - 4 : j - 2));
#pragma unroll
        for (int m = 1; m <= 4; ++m) {
          int yp = y + m, ym = y - m;
          if (PER) {
            yp -= yp >= ny ? ny : 0;
            ym += ym < 0 ? ny : 0;
          }
          yo[2 * m - 2] = PER || yp < ny ? yp * nxp + x : zero;
          yo[2 * m - 1] = PER || ym >= 0 ? ym * nxp + x : zero;
        }
        auto zload = [&](int z) -> float4 {          // plane z of this column, in this CTA or a neighbour
          if (z >= zbeg && z < zend) return *reinterpret_cast<const float4*>(v + (z - zbeg) * ps + col);
          const unsigned ad = L.paddr[z + 4];
          if (!PER && ad == 0) return make_float4(0.f, 0.f, 0.f, 0.f);
          return ld_cluster(ad + zoff + (unsigned)col * sizeof(float2));
        };
        float4 w[ZL + 8];                            // planes z0 - 4 .. z0 + ZL + 3
#pragma unroll
        for (int j = 0; j < 8; ++j) w[j] = zload(z0 - 4 + j);
#pragma unroll
        for (int zz = 0; zz < ZL; ++zz) {
          if (zz > 0 && z0 + zz >= z1) break;
          const int z = z0 + zz, loc = (z - zbeg) * ps;
          w[zz + 8] = zload(z + 4);
          const float2* p = v + loc;
          float2 X[8];                               // x - 4 .. x - 1, x + 2 .. x + 5
          if (EVEN) {
#pragma unroll
            for (int j = 0; j < 4; ++j) {
              const float4 t = *reinterpret_cast<const float4*>(p + xo[j]);
              X[2 * j] = lo2(t);
              X[2 * j + 1] = hi2(t);
            }
          } else {
#pragma unroll
            for (int j = 0; j < 8; ++j) X[j] = p[xo[EVEN ? 0 : j]];
          }
          float4 Y[8];
#pragma unroll
          for (int j = 0; j < 8; ++j) Y[j] = *reinterpret_cast<const float4*>(p + yo[j]);
          const float4 W = w[zz + 4];
          float VA, VB;
          float2 PA, PB;
          if (EVEN) {
            const float2 t = *reinterpret_cast<const float2*>(Vc + z * nxy + gA);
            const float4 f = *reinterpret_cast<const float4*>(psi + z * nxy + gA);
            VA = t.x; VB = t.y; PA = lo2(f); PB = hi2(f);
          } else {
            VA = Vc[z * nxy + gA]; VB = Vc[z * nxy + gB];
            PA = psi[z * nxy + gA]; PB = psi[z * nxy + gB];
          }
          // neighbours in local_h_at's order: +1, -1, +2, -2, ... in x, then in y
          auto nbA = [&](int j) -> float2 {
            switch (j) {
              case 0: return hi2(W); case 1: return X[3]; case 2: return X[4]; case 3: return X[2];
              case 4: return X[5];   case 5: return X[1]; case 6: return X[6]; case 7: return X[0];
              default: return lo2(Y[j - 8]);
            }
          };
          auto nbB = [&](int j) -> float2 {
            switch (j) {
              case 0: return X[4]; case 1: return lo2(W); case 2: return X[5]; case 3: return X[3];
              case 4: return X[6]; case 5: return X[2];   case 6: return X[7]; case 7: return X[1];
              default: return hi2(Y[j - 8]);
            }
          };
          float2 DA[3], DB[3];
          const float2 hA = local_h_at<float, PER, ACC && PER>(a, nbA, [&](int j) { return lo2(w[zz + j]); }, diag0 + VA, q, DA);
          const float2 hB = local_h_at<float, PER, ACC && PER>(a, nbB, [&](int j) { return hi2(w[zz + j]); }, diag0 + VB, q, DB);
          if (ACC) {                                 // |u|^2 and Im(conj(u) D1_a u)
            const float2 uA = lo2(W), uB = hi2(W);
            os[0] += uA.x * uA.x + uA.y * uA.y;
#pragma unroll
            for (int d = 0; d < 3; ++d) os[1 + d] += uA.x * DA[d].y - uA.y * DA[d].x;
            if (EVEN || !pad) {
              os[0] += uB.x * uB.x + uB.y * uB.y;
#pragma unroll
              for (int d = 0; d < 3; ++d) os[1 + d] += uB.x * DB[d].y - uB.y * DB[d].x;
            }
          }
          const float2 rA = M::fma(coef, make_float2(hA.y, -hA.x), PA);   // psi + (-i coef) H v
          float2 rB = M::fma(coef, make_float2(hB.y, -hB.x), PB);
          if (!PER && pad) rB = make_float2(0.f, 0.f);
          *reinterpret_cast<float4*>(nxt + loc + col) = make_float4(rA.x, rA.y, rB.x, rB.y);
        }
      }
    };
    if (OBS == 2 && st == 0) local_pass(std::integral_constant<bool, true>{});
    else local_pass(std::integral_constant<bool, false>{});
    if (ncta > 1) cluster_sync(); else __syncthreads();
    if (a.natom > 0) {
      for (int i = tid; i < a.natom * 8; i += kSlabThreads) {
        const int at = i >> 3;
        float t = 0.f;
        for (int r = 0; r < ncta; ++r)
          for (int c = 0; c < A.nch; ++c) t += L.part[((r * a.natom + at) * A.nch + c) * 8 + (i & 7)];
        reinterpret_cast<float*>(L.ec)[i] = t * (a.atomE[i >> 1] * a.dV);
      }
      __syncthreads();
      // nonlocal scatter from the tables: the thread of a point's first entry adds all of them
      for (int e0 = tid; e0 < L.off[a.natom]; e0 += kSlabThreads) {
        const int li = L.ix[e0];
        if (li < 0) continue;
        float re = 0.f, im = 0.f;
        unsigned lk;
        int e = e0;
        do {
          lk = L.lk[e];
          const int at = lk >> 16;
          const float4 b = A.beta_smem ? L.beta[e] : reinterpret_cast<const float4*>(a.sph_beta)[e + L.gof[at]];
          const float2 *c = L.ec + at * 4, f = L.ph[e];
          const float sr2 = b.x * c[0].x + b.y * c[1].x + b.z * c[2].x + b.w * c[3].x;
          const float si2 = b.x * c[0].y + b.y * c[1].y + b.z * c[2].y + b.w * c[3].y;
          re += sr2 * f.x + si2 * f.y;
          im += si2 * f.x - sr2 * f.y;
          e = (int)(lk & 0xffffu) - 1;
        } while (e >= 0);
        const float2 r = M::fma(coef, make_float2(im, -re), nxt[li]);
        nxt[li] = r;
        if (PER && !EVEN && nxp > nx && (li % ps) % nxp == 0) nxt[li + nx] = r;   // the row's pad (odd nx)
      }
      if (ncta > 1) cluster_sync(); else __syncthreads();
    }
  }

  // final pass: the orbital, the density and (OBS 1) the observables of the propagated orbital (copy 0)
  const float2* v = L.buf;
  float2* out = a.write_out ? a.psi_out + (size_t)orb * a.npts : nullptr;
  float* rho = a.rho32 ? a.rho32 + ((size_t)cell * a.nk + k) * a.npts : nullptr;
  for (int i = tid; i < npair; i += kSlabThreads) {
    const int row = i / hp, x = 2 * (i - row * hp), zl = row / ny, y = row - zl * ny;
    const int col = y * nxp + x, z = zbeg + zl, pg = z * nxy + y * nx + x;
    const bool pad = !EVEN && x + 1 >= nx;
    const float2* p = v + zl * ps;
    const float4 W = *reinterpret_cast<const float4*>(p + col);
    if (out) {
      if (EVEN) *reinterpret_cast<float4*>(out + pg) = W;
      else {
        out[pg] = lo2(W);
        if (!pad) out[pg + 1] = hi2(W);
      }
    }
    const float nA = W.x * W.x + W.y * W.y, nB = W.z * W.z + W.w * W.w;
    if (rho) {
      if (EVEN) {
        atomicAdd(reinterpret_cast<float2*>(rho + pg), make_float2(2.0f * nA, 2.0f * nB));
      } else {
        atomicAdd(rho + pg, 2.0f * nA);
        if (!pad) atomicAdd(rho + pg + 1, 2.0f * nB);
      }
    }
    if (OBS == 1) {
      os[0] += nA + (pad ? 0.f : nB);
      float2 d[3][2];
#pragma unroll
      for (int ax = 0; ax < 3; ++ax) d[ax][0] = d[ax][1] = make_float2(0.f, 0.f);
      // half of Im(conj(u) D1_a u) from the forward neighbours (fixed_final_pair of k_orbital.cu)
      auto wrap = [](int c, int n) { return c >= n ? c - n : c; };
      const float2 uA = lo2(W), uB = hi2(W);
#pragma unroll
      for (int m = 1; m <= 4; ++m) {
        const float2* pr = p + y * nxp;
        d[0][0] = M::fma(a.d1x[m - 1], M::sub(pr[wrap(x + m, nx)], uA), d[0][0]);
        d[0][1] = M::fma(a.d1x[m - 1], M::sub(pr[wrap(x + 1 + m, nx)], uB), d[0][1]);
        const float4 yp = *reinterpret_cast<const float4*>(p + wrap(y + m, ny) * nxp + x);
        d[1][0] = M::fma(a.d1y[m - 1], M::sub(lo2(yp), uA), d[1][0]);
        d[1][1] = M::fma(a.d1y[m - 1], M::sub(hi2(yp), uB), d[1][1]);
        const float4 zp = z + m < zend ? *reinterpret_cast<const float4*>(v + (z + m - zbeg) * ps + col)
                                       : ld_cluster(L.paddr[z + m + 4] + (unsigned)col * sizeof(float2));
        d[2][0] = M::fma(a.d1z[m - 1], M::sub(lo2(zp), uA), d[2][0]);
        d[2][1] = M::fma(a.d1z[m - 1], M::sub(hi2(zp), uB), d[2][1]);
      }
#pragma unroll
      for (int ax = 0; ax < 3; ++ax) {
        os[1 + ax] += 2.0f * (W.x * d[ax][0].y - W.y * d[ax][0].x);
        if (!pad) os[1 + ax] += 2.0f * (W.z * d[ax][1].y - W.w * d[ax][1].x);
      }
    }
  }
  if (OBS == 0) {
    if (ncta > 1) cluster_sync();                  // no CTA leaves while a neighbour may still read it
    return;
  }
  if (OBS == 1 && a.natom > 0) {
    __syncthreads();
    slab_phases(A, L, rank, qo);
    __syncthreads();
    slab_project<4>(A, L, v, L.parto, rank, false);
  }
  // sums of the CTA in float-float, then of the cluster (CTA 0) in FP64
#pragma unroll
  for (int j = 0; j < 4; ++j) {
    const FF x = Acc<float>::warp_sum(Acc<float>::add(Acc<float>::zero(), os[j]));
    if (lane == 0) s_red[j][warp] = x;
  }
  __syncthreads();
  if (tid < 4) {
    FF x = Acc<float>::zero();
    for (int w = 0; w < kSlabThreads / 32; ++w) x = Acc<float>::addv(x, s_red[tid][w]);
    const double t = Acc<float>::to_double(x);
    if (ncta > 1) st_cluster(map_cta(smem_addr(&s_obs[rank][tid]), 0), t);
    else s_obs[0][tid] = t;
  }
  if (ncta > 1) cluster_sync(); else __syncthreads();
  if (rank != 0) return;
  // J_nl: sum over atoms and projectors of 2 E_p Im(conj(b^(d)) c) dV^2, warp d takes component d
  if (warp < 3) {
    double sum = 0.0;
    for (int ap4 = lane; ap4 < a.natom * 4; ap4 += 32) {
      const int at = ap4 >> 2, p = ap4 & 3;
      float c[2] = {0.f, 0.f}, b[2] = {0.f, 0.f};
      for (int r = 0; r < ncta; ++r) {
        const float* pc = L.parto + ((size_t)r * a.natom + at) * 32 + 2 * p;
        c[0] += pc[0]; c[1] += pc[1];
        b[0] += pc[8 * (warp + 1)]; b[1] += pc[8 * (warp + 1) + 1];
      }
      sum += (double)(2.0f * a.atomE[ap4] * (b[0] * c[1] - b[1] * c[0]));
    }
#pragma unroll
    for (int o = 16; o > 0; o >>= 1) sum += __shfl_xor_sync(0xffffffffu, sum, o);
    if (lane == 0) s_jnl[warp] = sum * (double)a.dV * (double)a.dV;
  }
  __syncthreads();
  if (tid < 8) {
    double n = 0.0, x = 0.0;
    for (int r = 0; r < ncta; ++r) {
      n += s_obs[r][0];
      if (tid >= 1 && tid < 4) x += s_obs[r][tid];
    }
    double res = 0.0;
    if (tid == 0) res = n * (double)a.dV;
    else if (tid < 4) res = (x + (double)qo[tid - 1] * n) * (double)a.dV;
    else if (tid < 7) res = s_jnl[tid - 4];
    a.obs[(size_t)orb * 8 + tid] = res;
  }
}

size_t slab_smem(const SlabArgs& A, int nz, int natom, bool obs) {
  return sizeof(float2) * (2 * (size_t)A.zl * A.ps + 4 * (size_t)natom) + (size_t)A.max_ent * (8 + 8 + (A.beta_smem ? 16 : 0)) +
         sizeof(float) * (size_t)A.ncta * natom * (8 * A.nch + (obs ? 32 : 0)) + sizeof(int) * (size_t)(2 * natom + 1 + nz + 8);
}

bool slab_split(int nx, int ny, int nz, bool periodic, int natom, const int max_ent[9], int norb_tot, SlabArgs* A) {
  // Cluster size and segments by the cycles of a stage: about 330 issue cycles per plane of a warp of 32 pairs
  // and 120 per segment (window and offsets); two CTAs share an SM where their memory allows it (half the
  // issue slots each, but the 4000 cycles of projection, scatter and barriers of a stage overlap).  Times the
  // waves of clusters, as many at once as the driver says.
  A->nxp = (nx + 1) & ~1;
  A->ps = A->nxp * ny + (periodic ? 0 : 2);
  A->nch = natom > 0 && natom < kSlabThreads / 32 ? kSlabThreads / 32 / natom : 1;
  double best = 0.0;
  bool ok = false;
  const void* kern = periodic ? (const void*)k_slab<true, true, 1, 2> : (const void*)k_slab<false, true, 0, 2>;
  for (int c = 1; c <= 8; ++c) {
    const int planes = (nz + c - 1) / c;
    if (c > nz || (c - 1) * planes >= nz) continue;            // a CTA without planes
    SlabArgs T = *A;
    T.ncta = c; T.zl = planes; T.max_ent = max_ent[c];
    // the projectors' values stay in global memory where the SM then holds two CTAs instead of one
    T.beta_smem = 1;
    size_t smem = slab_smem(T, nz, natom, periodic);
    if (smem > kSlabHalfSm) {
      T.beta_smem = 0;
      const size_t less = slab_smem(T, nz, natom, periodic);
      if (less > kSlabHalfSm && smem <= 222 * 1024) T.beta_smem = 1;
      else smem = less;
    }
    if (smem > 222 * 1024) continue;
    cudaLaunchConfig_t cfg = {};
    cfg.gridDim = dim3((unsigned)c * 512u);
    cfg.blockDim = dim3(kSlabThreads);
    cfg.dynamicSmemBytes = smem;
    cudaLaunchAttribute at[1];
    at[0].id = cudaLaunchAttributeClusterDimension;
    at[0].val.clusterDim.x = (unsigned)c;
    at[0].val.clusterDim.y = at[0].val.clusterDim.z = 1;
    cfg.attrs = at;
    cfg.numAttrs = 1;
    int slots = 0;
    if (cudaFuncSetAttribute(kern, cudaFuncAttributeMaxDynamicSharedMemorySize, (int)smem) != cudaSuccess ||
        cudaOccupancyMaxActiveClusters(&slots, kern, &cfg) != cudaSuccess || slots < 1) {
      cudaGetLastError();
      continue;
    }
    const bool shared = smem <= kSlabHalfSm && norb_tot * c > 152;
    const double waves = (double)((norb_tot + slots - 1) / slots);
    for (int L : {1, 2, 4}) {
      const int segs = (planes + L - 1) / L;
      const int wi = (A->nxp / 2 * ny * segs + 31) / 32;
      const int rounds = (wi + kSlabThreads / 32 - 1) / (kSlabThreads / 32);
      const double busy = rounds * 2 * (330.0 * L + 120.0);    // two warps of the CTA per scheduler
      const double cyc = shared ? std::max(2 * busy, busy + 4000.0) : busy + 4000.0;
      if (!ok || waves * cyc < best) {
        best = waves * cyc;
        A->ncta = c; A->zl = planes; A->zlen = L; A->nseg = segs; A->max_ent = max_ent[c]; A->beta_smem = T.beta_smem;
        ok = true;
      }
    }
  }
  return ok;
}

template <bool PER, bool EVEN, int OBS, int ZL>
static cudaError_t launch_slab_one(const SlabArgs& A, cudaStream_t s) {
  auto kern = k_slab<PER, EVEN, OBS, ZL>;
  const size_t smem = slab_smem(A, A.o.nz, A.o.natom, OBS != 0);
  cudaError_t e = cudaFuncSetAttribute(kern, cudaFuncAttributeMaxDynamicSharedMemorySize, (int)smem);
  if (e != cudaSuccess) return e;
  cudaLaunchConfig_t cfg = {};
  cfg.gridDim = dim3((unsigned)(A.o.ncell * A.o.nk * A.o.norb * A.ncta));
  cfg.blockDim = dim3(kSlabThreads);
  cfg.dynamicSmemBytes = smem;
  cfg.stream = s;
  cudaLaunchAttribute at[1];
  at[0].id = cudaLaunchAttributeClusterDimension;
  at[0].val.clusterDim.x = (unsigned)A.ncta;
  at[0].val.clusterDim.y = at[0].val.clusterDim.z = 1;
  cfg.attrs = at;
  cfg.numAttrs = 1;
  return cudaLaunchKernelEx(&cfg, kern, A);
}

template <bool PER, bool EVEN, int OBS>
static cudaError_t launch_slab_zl(const SlabArgs& A, cudaStream_t s) {
  if (A.zlen == 1) return launch_slab_one<PER, EVEN, OBS, 1>(A, s);
  if (A.zlen == 2) return launch_slab_one<PER, EVEN, OBS, 2>(A, s);
  return launch_slab_one<PER, EVEN, OBS, 4>(A, s);
}

template <bool PER, bool EVEN>
static cudaError_t launch_slab_obs(const SlabArgs& A, cudaStream_t s) {
  if constexpr (PER) {
    if (A.o.obs) return A.o.obs_at_start ? launch_slab_zl<true, EVEN, 2>(A, s) : launch_slab_zl<true, EVEN, 1>(A, s);
  }
  return launch_slab_zl<PER, EVEN, 0>(A, s);
}

cudaError_t launch_slab(const SlabArgs& A, cudaStream_t s) {
  // 16-byte accesses of the caller's orbitals need an even nx and aligned arrays
  const bool even = A.o.nx % 2 == 0 && ((reinterpret_cast<uintptr_t>(A.o.psi_in) | reinterpret_cast<uintptr_t>(A.o.psi_out)) & 15) == 0;
  if (A.o.periodic) return even ? launch_slab_obs<true, true>(A, s) : launch_slab_obs<true, false>(A, s);
  return even ? launch_slab_obs<false, true>(A, s) : launch_slab_obs<false, false>(A, s);
}

}  // namespace tdks
