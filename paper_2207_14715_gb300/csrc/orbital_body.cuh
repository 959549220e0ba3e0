// Body of the orbital kernel for a group of (walker, electron) points (arXiv:2207.14715, Sec. 2.1,
// orbital expansion): basis functions and orbital values, gradients and Laplacians; one block per
// group, shared by the single-system, batched and fused batch kernels.
#pragma once

#include "batch.h"
#include "walker_common.cuh"

namespace vbq {

namespace {

constexpr int kOrbWarps = 8;

// Chunks c = lane, lane + 32, ... of the contraction with groups of WD orbitals (coefficients
// interleaved, stride WD): partial sums of phi, grad phi and lap phi over the chunk's basis
// functions into part[(5 t + k) nch + c].  Basis layout as written by orbital_block.
template <class Tb, int WD>
__device__ __forceinline__ void contract_groups(const SysDev& s, int lane, int nch, const Tb* __restrict__ cq,
                                                const Tb* bv, Tb* part) {
  const int M = s.M;
  for (int c = lane; c < nch; c += 32) {
    const int4 ch = __ldg(reinterpret_cast<const int4*>(s.evq_chunk) + c);
    Tb a[WD][5];
#pragma unroll
    for (int t = 0; t < WD; ++t)
#pragma unroll
      for (int k = 0; k < 5; ++k) a[t][k] = (Tb)0;
    for (int mu = ch.y; mu < ch.z; ++mu) {
      Tb cm[WD], b[5];
      if constexpr (WD == 4 && kSameType<Tb, double>) {
        const double2 c01 = __ldg(reinterpret_cast<const double2*>(cq + ch.w + 4 * mu));
        const double2 c23 = __ldg(reinterpret_cast<const double2*>(cq + ch.w + 4 * mu) + 1);
        cm[0] = c01.x; cm[1] = c01.y; cm[2] = c23.x; cm[3] = c23.y;
      } else if constexpr (WD == 4) {
        const float4 c4 = __ldg(reinterpret_cast<const float4*>(cq + ch.w + 4 * mu));
        cm[0] = c4.x; cm[1] = c4.y; cm[2] = c4.z; cm[3] = c4.w;
      } else {
        cm[0] = __ldg(cq + ch.w + mu);
      }
      if constexpr (kSameType<Tb, double>) {
        b[0] = bv[mu]; b[1] = bv[M + mu]; b[2] = bv[2 * M + mu]; b[3] = bv[3 * M + mu]; b[4] = bv[4 * M + mu];
      } else {
        const float4 b4 = reinterpret_cast<const float4*>(bv)[mu];
        b[0] = b4.x; b[1] = b4.y; b[2] = b4.z; b[3] = b4.w;
        b[4] = reinterpret_cast<const float*>(bv)[4 * M + mu];
      }
#pragma unroll
      for (int t = 0; t < WD; ++t)
#pragma unroll
        for (int k = 0; k < 5; ++k) a[t][k] += cm[t] * b[k];
    }
#pragma unroll
    for (int t = 0; t < WD; ++t)
#pragma unroll
      for (int k = 0; k < 5; ++k) part[(5 * t + k) * nch + c] = a[t][k];
  }
}

// One block: the cnt <= L.wpb points gw0 .. gw0 + cnt - 1 ((walker, electron) pairs in walker-major
// order), each with its own region of shared memory.  The basis evaluation goes by items (shell,
// point), 32 items of one angular momentum to a warp, the d shells first: a warp runs one kind of
// shell, with every lane busy, where a warp per point ran the three kinds one after the other in
// its second round of 32 shells (36 s, 18 p and 6 d shells on the ethylene-shaped system:
// 1.81 -> 1.59 ms for 3001 walkers in double, 0.367 -> 0.332 ms for 6001 in float with the float-float
// values).  Then warp e contracts point e.
template <class Tb>
__device__ __forceinline__ void orbital_block(const SysDev& s, const OrbLayout& L, long long gw0, int cnt,
                                              unsigned char* smem, const double* Rg, Tb* __restrict__ OB,
                                              double* __restrict__ OD) {
  const int tid = threadIdx.x, nt = blockDim.x, lane = tid & 31, wl = tid >> 5, nw = nt >> 5;
  const int nev = s.n_ev, nevd = s.n_ev_det, M = s.M, Nn = s.Nn;
  // q / cnt and q % cnt for q < 2^16 by a multiplication (cnt <= 16)
  const unsigned rcp = (1u << 20) / (unsigned)cnt + 1u;
  auto split = [&](int q, int& hi, int& lo) {
    hi = (int)(((unsigned)q * rcp) >> 20);
    lo = q - hi * cnt;
  };
  const double* Rp = Rg + (size_t)gw0 * 3;
  if constexpr (!kSameType<Tb, double>) {
    for (int q = tid; q < 3 * cnt; q += nt) {
      int d, e;
      split(q, d, e);
      reinterpret_cast<dsf*>(smem + e * L.warp_bytes + L.r3)[d] = ds_from_double(Rp[3 * e + d]);
    }
    __syncthreads();
  }
  // displacement of every point from every nucleus
  for (int q = tid; q < cnt * Nn; q += nt) {
    int a, e;
    split(q, a, e);
    unsigned char* base = smem + e * L.warp_bytes;
    Tb* dis = reinterpret_cast<Tb*>(base + L.dis) + 3 * a;
    if constexpr (kSameType<Tb, double>) {
      const double* nu = s.nuc4 + 4 * a;
#pragma unroll
      for (int d = 0; d < 3; ++d) dis[d] = Rp[3 * e + d] - __ldg(nu + d);
    } else {
      const dsf* r3 = reinterpret_cast<const dsf*>(base + L.r3);
#pragma unroll
      for (int d = 0; d < 3; ++d) dis[d] = ds_diff_f(r3[d], nuc_coord_ds(s, a, d));
      if (OD) center_ds(s, a, r3, reinterpret_cast<dsf*>(base + L.ctab));
    }
  }
  __syncthreads();
  const int i2 = s.S - s.sh_l_off[2], i1 = s.sh_l_off[2] - s.sh_l_off[1], i0 = s.sh_l_off[1];  // shells per l
  const int w2 = (i2 * cnt + 31) >> 5, w1 = (i1 * cnt + 31) >> 5, w0 = (i0 * cnt + 31) >> 5;
  for (int task = wl; task < w2 + w1 + w0; task += nw) {
    const int l = task < w2 ? 2 : (task < w2 + w1 ? 1 : 0);
    const int first = l == 2 ? 0 : (l == 1 ? w2 : w2 + w1), num = l == 2 ? i2 : (l == 1 ? i1 : i0);
    const int q = 32 * (task - first) + lane;
    if (q >= num * cnt) continue;
    int t, e;
    split(q, t, e);
    unsigned char* base = smem + e * L.warp_bytes;
    // one 16-byte record per shell, in the order of l
    const int4 p = __ldg(reinterpret_cast<const int4*>(s.sh_pack_f) + s.sh_l_off[l] + t);
    const int c = p.x & 0xffff, f = p.y, sh = p.z;
    const Tb* dis = reinterpret_cast<const Tb*>(base + L.dis) + 3 * c;
    Tb* bv = reinterpret_cast<Tb*>(base + L.bas);
    if constexpr (kSameType<Tb, double>) {
      gto_shell<double, true>(l, __ldg(s.sh_zeta + sh), s.sh_norm + 6 * sh, dis[0], dis[1], dis[2], bv + f, bv + M + f,
                              bv + 2 * M + f, bv + 3 * M + f, bv + 4 * M + f);
    } else {
      // value and gradient of a function as one 16-byte store (one shared-memory load per function
      // and coefficient in the contraction), Laplacians after them
      gto_shell_emit<float, true>(l, __int_as_float(p.w), s.sh_norm_f + 6 * sh, dis[0], dis[1], dis[2],
                                  [&](int k, float v, float x, float y, float z, float lp) {
                                    reinterpret_cast<float4*>(bv)[f + k] = make_float4(v, x, y, z);
                                    bv[4 * M + f + k] = lp;
                                  });
      if (OD)
        shell_values_ds(s, sh, c, l, f, reinterpret_cast<const dsf*>(base + L.ctab),
                        reinterpret_cast<dsf*>(base + L.bds));
    }
  }
  __syncthreads();
  if (wl >= cnt) return;
  const long long gw = gw0 + wl;
  unsigned char* base = smem + wl * L.warp_bytes;
  const Tb* bv = reinterpret_cast<const Tb*>(base + L.bas);
  const dsf* bds = reinterpret_cast<const dsf*>(base + L.bds);
  Tb* part = reinterpret_cast<Tb*>(base + L.part);
  dsf* partds = reinterpret_cast<dsf*>(base + L.partd);
  // contraction by groups of orbitals sharing a coefficient range (quads: one basis-function
  // load feeds four orbitals); partials component-major, part[(5 t + k) nch + chunk]
  const int nch = s.n_evq_chunk;
  const Tb* cq = kSameType<Tb, double> ? reinterpret_cast<const Tb*>(s.evq_coef)
                                       : reinterpret_cast<const Tb*>(s.evq_coef_f);
  if (s.evq_width == 4)
    contract_groups<Tb, 4>(s, lane, nch, cq, bv, part);
  else
    contract_groups<Tb, 1>(s, lane, nch, cq, bv, part);
  if (!kSameType<Tb, double> && OD)
    for (int c = lane; c < s.n_det_chunk; c += 32) {
      const int4 ch = __ldg(reinterpret_cast<const int4*>(s.det_chunk) + c);
      const float2* cb = reinterpret_cast<const float2*>(s.orb_coef_ds) + ch.w;
      dsf acc = {0.0f, 0.0f};
      for (int mu = ch.y; mu < ch.z; ++mu) {
        const float2 lm = __ldg(cb + mu);
        acc = ds_add(acc, ds_mul(dsf{lm.x, lm.y}, bds[mu]));
      }
      partds[c] = acc;
    }
  __syncwarp();
  Tb* out = OB + (size_t)gw * 5 * nev;
  for (int q = lane; q < nev; q += 32) {
    const int qs = __ldg(s.evq_slot + q), qd = qs >> 2;
    const int c0 = __ldg(s.evq_chunk_off + qd), c1 = __ldg(s.evq_chunk_off + qd + 1);
    const Tb* pp = part + 5 * (qs & 3) * nch;
    Tb v = 0, gx = 0, gy = 0, gz = 0, lp = 0;
    for (int c = c0; c < c1; ++c) {
      v += pp[c]; gx += pp[nch + c]; gy += pp[2 * nch + c]; gz += pp[3 * nch + c]; lp += pp[4 * nch + c];
    }
    if (q < nevd && OD) {  // OD null: the determinant-orbital values in double are not needed
      double vd = 0.0;
      if (kSameType<Tb, double>) {
        vd = (double)v;
      } else {
        const int d0 = __ldg(s.det_chunk_off + q), d1 = __ldg(s.det_chunk_off + q + 1);
        dsf acc = {0.0f, 0.0f};
        for (int c = d0; c < d1; ++c) acc = ds_add(acc, partds[c]);
        vd = ds_to_double(acc);
      }
      OD[(size_t)gw * nevd + q] = vd;
      v = (Tb)vd;
    }
    out[q] = v;
    out[nev + q] = gx;
    out[2 * nev + q] = gy;
    out[3 * nev + q] = gz;
    out[4 * nev + q] = lp;
  }
}

}  // namespace

}  // namespace vbq
