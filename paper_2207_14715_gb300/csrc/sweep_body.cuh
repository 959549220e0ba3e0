// Per-walker body of the VMC sweep (arXiv:2207.14715, Sec. 2.3.1): single-electron Metropolis
// moves with the determinants carried by per-determinant inverses or reference tables;
// shared by the single-system, batched and fused batch kernels.
#pragma once

#include "batch.h"
#include "tab_minors.cuh"
#include "walker_common.cuh"

namespace vbq {

// =====================================================================================
// VMC sweep kernel
// =====================================================================================
// Two ways of carrying the determinants through the moves (template parameter TAB):
//  - per-determinant inverses (TAB = false): every unique determinant's inverse is updated by
//    Sherman-Morrison on an accepted move (Sec. 2.3.1); the ratio of determinant u is
//    rho_u = sum_o v_o Binv_u[o][i].
//  - reference-determinant tables (TAB = true; systems whose per-determinant inverses do not
//    fit in shared memory): each spin carries the inverse B of its reference determinant
//    (u = 0), T = B Phi_X over the orbitals X outside the reference, and the minors q_u =
//    det T[S_u, Q_u] = sgn_u D_u / D_0 (tab_minors.cuh).  Moving electron i to a point with orbital
//    row v gives
//      rho_0 = sum_o v_o B[o][i],  c_x = v_x - sum_o v_o T[o][x],  b = B[:, i] / rho_0,
//      T' = T + b c^T,  q'_u = det T'[S_u, Q_u],
//    and Phi'/Phi = rho_0 Sigma' / Sigma with Sigma = sum_k C_k q_up(k) q_dn(k) (C_k with the signs) =
//    sum_u q_u g_u, where g_u = sum over the terms of u of C_k times the other spin's minor stays
//    as it is while the electrons of one spin move; an accepted move updates B by Sherman-Morrison,
//    T to T' and q to q'.
//    Bound: latency at 9 walkers per SM (the walker's region), over the FP64 pipe, whose
//    instructions are therefore counted: on 48 electrons (70 determinants per spin) about 60 per
//    move and 55 more when it is accepted, where eliminating every determinant's matrix, summing
//    the 256 terms and serial column sums took about 250 and 70.  With the proposals below 9.4 ms per
//    sweep of 8192 walkers, 16.4 with those.
// Each sweep moves every electron once (Sec. 2.3.1).  The determinant inverses come from
// the walker state written by the evaluation at the same positions, or from a fresh LU of
// double-precision orbital values (first sweep without state, and every 'refresh' sweeps).
// The proposed orbital row uses the bulk type; ratios and Sherman-Morrison updates are double.
//
// What a move needs of its own electron alone is prepared for all electrons of a spin before their
// moves (an electron's proposal depends on its own position only, and it moves once per sweep):
// the proposals' orbital rows, for L.ke electrons at a time so that a coefficient and its index serve
// them all and every round of 32 (shell, electron) items is full, and the nuclei's Rbar and e-n
// changes over all (electron, nucleus) pairs.  A move is then left with the other electrons: the
// distances from the proposal, against Rbar and the e-e value of the current pairs, which are kept
// per pair (L.tri) and replaced when a move is accepted.  The float values and sums are those of a
// move that forms everything by itself, bit for bit.  Bound by instruction issue (float) and the
// FP64 pipe (double); a sweep of the ethylene-shaped system went from 1298 to 1080 us (16384 walkers,
// mixed; 1030 in small blocks), 2303 to 2095 us (3001, double; 1512), one of the 48-electron system from 11.5
// to 10.0 ms (8192; 9.4 with at most 16 electrons prepared at once and small blocks).
// One warp, walker w, shared-memory region 'base' of L.warp_bytes bytes.

// f of the Pade + polynomial form at R = r den, den = 1 / (1 + kappa r) (as pade_poly)
template <class Tb> __device__ __forceinline__ Tb pade_value(const PadeT<Tb>& c, Tb r, Tb den) {
  const Tb R = r * den;
  const Tb pd = (Tb)1 / ((Tb)1 + c.a2 * R);
  const Tb R2 = R * R, R3 = R2 * R, R4 = R3 * R, R5 = R4 * R;
  return c.a1 * R * pd + c.q[0] * R2 + c.q[1] * R3 + c.q[2] * R4 + c.q[3] * R5;
}

// (x, y) pairs: the old and new side of a move's e-e-n sums.  In float each operation is one packed
// instruction on both (independent, correctly rounded: the same values as two scalar ones).
template <class Tb> struct Pair2 { Tb o, n; };
__device__ __forceinline__ Pair2<double> pair_fma(Pair2<double> a, Pair2<double> b, Pair2<double> c) {
  return {fma(a.o, b.o, c.o), fma(a.n, b.n, c.n)};
}
__device__ __forceinline__ Pair2<double> pair_mul(Pair2<double> a, Pair2<double> b) { return {a.o * b.o, a.n * b.n}; }
__device__ __forceinline__ Pair2<double> pair_add(Pair2<double> a, Pair2<double> b) { return {a.o + b.o, a.n + b.n}; }
__device__ __forceinline__ Pair2<float> pair_fma(Pair2<float> a, Pair2<float> b, Pair2<float> c) {
  Pair2<float> d;
  asm("{\n\t.reg .b64 a, b, c;\n\tmov.b64 a, {%2, %3};\n\tmov.b64 b, {%4, %5};\n\tmov.b64 c, {%6, %7};\n\t"
      "fma.rn.f32x2 a, a, b, c;\n\tmov.b64 {%0, %1}, a;\n\t}"
      : "=f"(d.o), "=f"(d.n)
      : "f"(a.o), "f"(a.n), "f"(b.o), "f"(b.n), "f"(c.o), "f"(c.n));
  return d;
}
__device__ __forceinline__ Pair2<float> pair_mul(Pair2<float> a, Pair2<float> b) {
  Pair2<float> d;
  asm("{\n\t.reg .b64 a, b;\n\tmov.b64 a, {%2, %3};\n\tmov.b64 b, {%4, %5};\n\t"
      "mul.rn.f32x2 a, a, b;\n\tmov.b64 {%0, %1}, a;\n\t}"
      : "=f"(d.o), "=f"(d.n)
      : "f"(a.o), "f"(a.n), "f"(b.o), "f"(b.n));
  return d;
}
__device__ __forceinline__ Pair2<float> pair_add(Pair2<float> a, Pair2<float> b) {
  Pair2<float> d;
  asm("{\n\t.reg .b64 a, b;\n\tmov.b64 a, {%2, %3};\n\tmov.b64 b, {%4, %5};\n\t"
      "add.rn.f32x2 a, a, b;\n\tmov.b64 {%0, %1}, a;\n\t}"
      : "=f"(d.o), "=f"(d.n)
      : "f"(a.o), "f"(a.n), "f"(b.o), "f"(b.n));
  return d;
}

// r^2 of a proposal's basis functions: the products rounded one by one, or (FUSED) fused.  The
// single-system and the batch kernels each keep to one form whatever the compiler would contract,
// so that their trajectories stay the ones of earlier builds.
template <bool FUSED> __device__ __forceinline__ float norm2(float x, float y, float z) {
  if constexpr (FUSED) return fmaf(z, z, fmaf(x, x, __fmul_rn(y, y)));
  return __fadd_rn(__fadd_rn(__fmul_rn(x, x), __fmul_rn(y, y)), __fmul_rn(z, z));
}

// Values of a shell (as gto_shell_emit with r^2 given): emit(c, chi_c)
template <class Emit>
__device__ __forceinline__ void shell_values(int l, float z, const float* nrm, float r2, float dx, float dy, float dz,
                                             Emit&& emit) {
  const float e = z < 0.0f ? vexp(z * vsqrt(r2)) : (z == 0.0f ? 1.0f : vexp(-z * r2));
  if (l == 0) {
    emit(0, __ldg(nrm) * e);
  } else if (l == 1) {
    const float d[3] = {dx, dy, dz};
#pragma unroll
    for (int c = 0; c < 3; ++c) emit(c, __ldg(nrm + c) * e * d[c]);
  } else {
    constexpr int ia[6] = {0, 1, 2, 0, 0, 1}, ib[6] = {0, 1, 2, 1, 2, 2};  // xx yy zz xy xz yz
    const float d[3] = {dx, dy, dz};
#pragma unroll
    for (int c = 0; c < 6; ++c) emit(c, __ldg(nrm + c) * e * (d[ia[c]] * d[ib[c]]));
  }
}

// Rows of the proposals of cnt <= KE electrons (float form): rnd [cnt][3] their positions, out [cnt][ldo].
template <int KE, bool FUSED>
__device__ __forceinline__ void proposal_rows(const SysDev& s, int lane, int sp, int cnt, const dsf* rnd, float* bas,
                                              float* part, bool alias, float* out, int ldo) {
  constexpr int kLog = KE == 4 ? 2 : (KE == 2 ? 1 : 0);
  const int Nn = s.Nn;
  // the displacements, lane el Nn + a, shared by shuffles with the lanes of that nucleus's shells
  // (too many nuclei: each item forms its own)
  const bool shuf = KE * Nn <= 32;
  float cx = 0.0f, cy = 0.0f, cz = 0.0f;
  if (shuf && lane < cnt * Nn) {
    const DivStep ea(lane, Nn);
    cx = ds_diff_f(rnd[3 * ea.hi], nuc_coord_ds(s, ea.lo, 0));
    cy = ds_diff_f(rnd[3 * ea.hi + 1], nuc_coord_ds(s, ea.lo, 1));
    cz = ds_diff_f(rnd[3 * ea.hi + 2], nuc_coord_ds(s, ea.lo, 2));
  }
  for (int i0 = 0; i0 < KE * s.S; i0 += 32) {  // every lane takes part in each round (the shuffles)
    const int i = i0 + lane, t = i >> kLog, el = i & (KE - 1);
    const bool act = t < s.S && el < cnt;
    // one 16-byte record per shell, in the order of l
    const int4 p = act ? __ldg(reinterpret_cast<const int4*>(s.sh_pack_f) + t) : make_int4(0, 0, 0, 0);
    const int c = p.x & 0xffff, l = p.x >> 16, f = p.y, sh = p.z;
    float dx, dy, dz;
    if (shuf) {
      const int src = el * Nn + c;
      dx = __shfl_sync(kFull, cx, src);
      dy = __shfl_sync(kFull, cy, src);
      dz = __shfl_sync(kFull, cz, src);
    } else if (act) {
      dx = ds_diff_f(rnd[3 * el], nuc_coord_ds(s, c, 0));
      dy = ds_diff_f(rnd[3 * el + 1], nuc_coord_ds(s, c, 1));
      dz = ds_diff_f(rnd[3 * el + 2], nuc_coord_ds(s, c, 2));
    }
    if (act)
      shell_values(l, __int_as_float(p.w), s.sh_norm_f + 6 * sh, norm2<FUSED>(dx, dy, dz), dx, dy, dz,
                   [&](int k, float v) { bas[KE * (f + k) + el] = v; });
  }
  __syncwarp();
  // contraction in balanced chunks: one coefficient serves the KE electrons
  for (int c0 = 0; c0 < s.n_occ_chunk[sp]; c0 += 32) {
    const int c = c0 + lane;
    float v[KE];
#pragma unroll
    for (int k = 0; k < KE; ++k) v[k] = 0.0f;
    if (c < s.n_occ_chunk[sp]) {
      const int4 ch = __ldg(reinterpret_cast<const int4*>(s.occ_chunk[sp]) + c);
      const float* cb = s.orb_coef_f + ch.w;
#pragma unroll 4
      for (int mu = ch.y; mu < ch.z; ++mu) {
        const float cm = __ldg(cb + mu);
        float b[KE];
        if constexpr (KE == 4) {
          const float4 q = reinterpret_cast<const float4*>(bas)[mu];
          b[0] = q.x; b[1] = q.y; b[2] = q.z; b[3] = q.w;
        } else if constexpr (KE == 2) {
          const float2 q = reinterpret_cast<const float2*>(bas)[mu];
          b[0] = q.x; b[1] = q.y;
        } else {
          b[0] = bas[mu];
        }
#pragma unroll
        for (int k = 0; k < KE; ++k) v[k] += cm * b[k];
      }
    }
    if (alias) __syncwarp();  // one round: the partial sums take the place of the basis values
    if (c < s.n_occ_chunk[sp])
#pragma unroll
      for (int k = 0; k < KE; ++k) part[KE * c + k] = v[k];
  }
  __syncwarp();
  const int nocc = s.nocc[sp];
  for (int i = lane; i < KE * nocc; i += 32) {
    const int q = i >> kLog, el = i & (KE - 1);
    const int c0 = __ldg(s.occ_chunk_off[sp] + q), c1 = __ldg(s.occ_chunk_off[sp] + q + 1);
    float v = 0.0f;
    for (int c = c0; c < c1; ++c) v += part[KE * c + el];
    if (el < cnt) out[el * ldo + q] = v;
  }
  __syncwarp();
}

template <class Tb, bool TAB, bool BATCH>
__device__ __forceinline__ void sweep_body(const SysDev& s, const SweepLayout& L, int w, unsigned char* base,
                                           double* __restrict__ Rg, int nsweeps, int refresh,
                                           double* __restrict__ state, int state_valid, double step, uint64_t seed,
                                           uint32_t step0, uint32_t tag, uint32_t woff, int* __restrict__ nacc) {
  const int lane = threadIdx.x & 31;
  double* Binv[2] = {reinterpret_cast<double*>(base + L.Binv0), reinterpret_cast<double*>(base + L.Binv1)};
  double* ldet = reinterpret_cast<double*>(base + L.ldet);
  double* dsg = reinterpret_cast<double*>(base + L.dsg);
  double* wk = reinterpret_cast<double*>(base + L.wk);
  double* PhiO = reinterpret_cast<double*>(base + L.PhiO);
  double* basd = reinterpret_cast<double*>(base + L.bas);
  Tb* bas = reinterpret_cast<Tb*>(base + L.bas);
  double* vrowd = reinterpret_cast<double*>(base + L.vrow);
  Tb* part = reinterpret_cast<Tb*>(base + L.part);
  double* partd = reinterpret_cast<double*>(base + L.part);
  double* rho = reinterpret_cast<double*>(base + L.rho);
  double* rinv = reinterpret_cast<double*>(base + L.rinv);
  double* cvec = reinterpret_cast<double*>(base + L.cvec);
  double* scr = reinterpret_cast<double*>(base + L.scratch);
  // of the prepared electrons (L.all: every electron; else up to L.grp of the moving spin): proposed positions
  // (and their float-float copies), Rbar and e-n change per nucleus; orbital rows of the moving spin's (L.rows: all)
  double* rtab = reinterpret_cast<double*>(base + L.rtab);  // [][3]
  dsf* rtds = reinterpret_cast<dsf*>(base + L.rtds);        // [][3]
  Tb* svn = reinterpret_cast<Tb*>(base + L.svn);            // [][Nn]
  Tb* den = reinterpret_cast<Tb*>(base + L.den);            // [][Nn]
  Tb* vrows = reinterpret_cast<Tb*>(base + L.vrows);        // [][nocc]
  // current positions: [Nn][SA] Rbar(r_ja) (its powers formed where used; the row stride padded so that
  // lanes on different nuclei read different banks), and per pair Rbar(r_ij) and the e-e value
  const int SA = s.N + 1, UP = s.N + 1;
  Tb* Sv = reinterpret_cast<Tb*>(base + L.Sv);
  Tb* ut = reinterpret_cast<Tb*>(base + L.ut);
  Tb* ft = reinterpret_cast<Tb*>(base + L.ft);
  // the move: (current, proposed) powers 1..4 of Rbar(r_ej), and the proposed pairs' Rbar and e-e value
  Pair2<Tb>* Up = reinterpret_cast<Pair2<Tb>*>(base + L.up);  // [4][UP]
  Tb* ue = reinterpret_cast<Tb*>(base + L.ue);
  Tb* fe = reinterpret_cast<Tb*>(base + L.fe);

  const int N = s.N, Nn = s.Nn, Nup = s.Nup, U0 = s.U[0], ldo = L.nocc_max;
  const Tb kap = (Tb)s.kappa;
  const Tb* cE = een_coefs<Tb>(s);
  double* Rw = Rg + (size_t)w * 3 * N;  // current positions in double; accepted moves are written through
  // positions as the bulk-type arithmetic reads them (float-float copies in the mixed form)
  double* Rs = reinterpret_cast<double*>(base + L.R);
  dsf* Rds = reinterpret_cast<dsf*>(base + L.R);
  Coords<Tb> C;
  for (int i = lane; i < 3 * N; i += 32) {
    if constexpr (kSameType<Tb, double>) Rs[i] = Rw[i];
    else Rds[i] = ds_from_double(Rw[i]);
  }
  if constexpr (kSameType<Tb, double>) C.R = Rs;
  else C.R = Rds;
  __syncwarp();
  // Rbar and e-e value of a pair from its difference vector
  auto pair_values = [&](Tb dx, Tb dy, Tb dz, bool same, Tb& u, Tb& f) {
    const Tb r = vsqrt(dx * dx + dy * dy + dz * dz);
    u = (Tb)1 / ((Tb)1 + kap * r);
    f = pade_value<Tb>(ee_coef_t<Tb>(s, same), r, u);
  };
  auto tri = [](int i, int j) { return i > j ? i * (i - 1) / 2 + j : j * (j - 1) / 2 + i; };
  // e-e-n lanes: (nucleus a, part of the partners); with more than 32 nuclei lanes loop over them
  const int np = max(1, 32 / Nn);
  int ea0 = lane, ej0 = 0, ej1 = N;
  if (np > 1) {
    const DivStep ap(lane, np);
    ea0 = ap.hi;
    ej0 = ap.lo * N / np;
    ej1 = (ap.lo + 1) * N / np;
  }
  // walker state: [Binv spin 0][Binv spin 1][ln|det| (Ut)][sign (Ut)][r_k = D_k/Phi (nterm)]
  // [ln|Phi|][sign Phi]; the sweep starts from the inverses and the term ratios and carries
  // both (and ln|Phi|) through its moves
  const int nb0 = s.U[0] * s.n[0] * s.n[0], nb1 = s.U[1] * s.n[1] * s.n[1], Ut = U0 + s.U[1];
  double lnPhi = 0.0, sgnPhi = 1.0;
  // product of the accepted moves' |Phi'/Phi| since ln|Phi| was last set, as a mantissa in
  // [1, 2) and a binary exponent (bit operations; one logarithm per sweep instead of one per move)
  double pm = 1.0;
  int pe = 0;
  // reference-determinant tables (TAB): T per spin, the minors of both spins in wk, proposed minors,
  // the move's c_x, the rows of T that the minors read, the weights g_u and w of the moving spin,
  // and Sigma with its reciprocal
  double* Tt[2] = {reinterpret_cast<double*>(base + L.T0), reinterpret_cast<double*>(base + L.T1)};
  double* qn = reinterpret_cast<double*>(base + L.qn);
  double* cxv = reinterpret_cast<double*>(base + L.cx);
  double* Tn = reinterpret_cast<double*>(base + L.Tn);
  double* gw = reinterpret_cast<double*>(base + L.gw);
  double* wrow = reinterpret_cast<double*>(base + L.wrow);
  double Sig = 1.0, iSig = 1.0;
  const bool from_state = !TAB && state && state_valid;
  if (from_state) {
    const double* st = state + (size_t)w * s.state_doubles;
    warp_copy(Binv[0], st, nb0, lane);
    warp_copy(Binv[1], st + nb0, nb1, lane);
    warp_copy(wk, st + nb0 + nb1 + 2 * Ut, s.nterm, lane);
    lnPhi = st[nb0 + nb1 + 2 * Ut + s.nterm];
    sgnPhi = st[nb0 + nb1 + 2 * Ut + s.nterm + 1];
  }
  __syncwarp();
  int accepted = 0;
  const uint32_t wid = woff + (uint32_t)w;

  for (int sw = 0; sw < nsweeps; ++sw) {
    const bool do_refresh = (sw == 0) ? !from_state : (refresh > 0 && sw % refresh == 0);
    if (do_refresh) {
      // double-precision orbital values of every electron, then the inverse of every unique determinant
      auto orbital_values = [&](int e, int sp) {  // of electron e, in vrowd
        basis_at<double, false>(s, lane, Rw[3 * e], Rw[3 * e + 1], Rw[3 * e + 2], basd, nullptr, nullptr, nullptr,
                                nullptr);
        __syncwarp();
        for (int c0 = 0; c0 < s.n_occ_chunk[sp]; c0 += 32) {
          const int c = c0 + lane;
          double v = 0.0;
          if (c < s.n_occ_chunk[sp]) {
            const int4 ch = __ldg(reinterpret_cast<const int4*>(s.occ_chunk[sp]) + c);
            const double* cb = s.orb_coef + ch.w;
            for (int mu = ch.y; mu < ch.z; ++mu) v = fma(__ldg(cb + mu), basd[mu], v);
          }
          if (L.alias) __syncwarp();
          if (c < s.n_occ_chunk[sp]) partd[c] = v;
        }
        __syncwarp();
        for (int q = lane; q < s.nocc[sp]; q += 32) {
          const int c0 = __ldg(s.occ_chunk_off[sp] + q), c1 = __ldg(s.occ_chunk_off[sp] + q + 1);
          double v = 0.0;
          for (int c = c0; c < c1; ++c) v += partd[c];
          vrowd[q] = v;
        }
        __syncwarp();
      };
      if constexpr (TAB) {
        // per spin: the reference's matrix in place of its inverse and the X values in PhiO, then
        // the inverse, T = B Phi_X and every minor
        for (int sp = 0; sp < 2; ++sp) {
          const int n = s.n[sp], e0 = sp ? Nup : 0, nx = s.n_x[sp];
          double* B = Binv[sp];
          double* T = Tt[sp];
          for (int i = 0; i < n; ++i) {
            orbital_values(e0 + i, sp);
            for (int o = lane; o < n; o += 32) B[i * n + o] = vrowd[__ldg(s.det_loc[sp] + o)];
            for (int x = lane; x < nx; x += 32) PhiO[i * nx + x] = vrowd[__ldg(s.tab_xl[sp] + x)];
            __syncwarp();
          }
          if (n > 0) {
            warp_inverse(B, n, nullptr, n, reinterpret_cast<int*>(scr), B);
          }
          for (DivStep ox(lane, max(nx, 1)); ox.hi < n && nx > 0; ox.next(nx)) {
            double v = 0.0;
            for (int e = 0; e < n; ++e) v = fma(B[ox.hi * n + e], PhiO[e * nx + ox.lo], v);
            T[ox.hi * nx + ox.lo] = v;
          }
          __syncwarp();
          for (DivStep ox(lane, max(nx, 1)); ox.hi < s.tab[sp].ns && nx > 0; ox.next(nx))
            Tn[ox.hi * nx + ox.lo] = T[__ldg(s.tab[sp].sl + ox.hi) * nx + ox.lo];
          __syncwarp();
          tab_values<true, true>(s.tab[sp], lane, Tn, wk + (sp ? s.tab[0].nv : 0));
        }
      } else {
        for (int e = 0; e < N; ++e) {
          const int sp = e >= Nup ? 1 : 0;
          orbital_values(e, sp);
          for (int q = lane; q < s.nocc[sp]; q += 32) PhiO[e * ldo + q] = vrowd[q];
          __syncwarp();
        }
        for (int sp = 0; sp < 2; ++sp)
          invert_all<double>(s, sp, lane, PhiO, ldo, s.det_loc[sp], sp ? L.G1 : L.G0, Binv[sp], nullptr, nullptr,
                             scr, ldet + (sp ? U0 : 0), dsg + (sp ? U0 : 0), nullptr, 0, nullptr);
      }
    }
    if (!TAB && do_refresh) {
      term_ratios(s, lane, ldet, dsg, wk, lnPhi, sgnPhi);  // wk: r_k = D_k / Phi
      pm = 1.0;
      pe = 0;
      __syncwarp();
    }
    if (sw == 0 || do_refresh) {
      // tables of the current positions (a refactorisation uses their place; moves keep them current)
      for (DivStep ia(lane, Nn); ia.hi < N; ia.next(Nn)) {
        const int i = ia.hi, a = ia.lo;
        const Tb dx = C.en(s, i, a, 0), dy = C.en(s, i, a, 1), dz = C.en(s, i, a, 2);
        const Tb r = vsqrt(dx * dx + dy * dy + dz * dz);
        Sv[a * SA + i] = (Tb)1 / ((Tb)1 + kap * r);
      }
      if (L.tri)
        for (int p = lane; p < N * (N - 1) / 2; p += 32) {
          int i = (int)((1.0f + sqrtf(1.0f + 8.0f * (float)p)) * 0.5f);  // row of the triangle, to one
          if (i * (i - 1) / 2 > p) --i;
          if (i * (i + 1) / 2 <= p) ++i;
          const int j = p - i * (i - 1) / 2;
          pair_values(C.ee(i, j, 0), C.ee(i, j, 1), C.ee(i, j, 2), (i < Nup) == (j < Nup), ut[p], ft[p]);
        }
    }
    const uint32_t st = step0 + (uint32_t)sw;
    double uac = 0.0;  // acceptance uniform of the prepared electron 'lane' (at most 32 of them)
    auto accept_position = [&](int e, int ip) {
      if (lane < 3) {
        const double x = rtab[3 * ip + lane];
        Rw[3 * e + lane] = x;
        if constexpr (kSameType<Tb, double>) Rs[3 * e + lane] = x;
        else Rds[3 * e + lane] = rtds[3 * ip + lane];
      }
      for (int a = lane; a < Nn; a += 32) Sv[a * SA + e] = svn[ip * Nn + a];
      if (L.tri)
        for (int j = lane; j < N; j += 32)
          if (j != e) {
            ut[tri(e, j)] = ue[j];
            ft[tri(e, j)] = fe[j];
          }
    };
    int e0 = 0;  // first of the electrons prepared together
    for (int e = 0; e < N; ++e) {
      const int sp = e >= Nup ? 1 : 0, ie = e - (sp ? Nup : 0), n = s.n[sp], G = sp ? L.G1 : L.G0;
      if (e == 0 || e == Nup || (!L.all && e - e0 == L.grp)) {
        e0 = e;
        // one electron per lane: the proposed position R_e + step (2u - 1) per coordinate (electron e
        // has not moved yet in this sweep when its turn comes) and the acceptance uniform; in the
        // mixed form also the float-float copy of the proposal
        const int cnt = L.all ? N - e : min(L.grp, n - ie);
        if (e == 0 || !L.all) {
          if (lane < cnt) {
            double u[4], Rc[3];  // the position's latency runs under the random numbers
#pragma unroll
            for (int d = 0; d < 3; ++d) Rc[d] = Rw[3 * (e + lane) + d];
            uniforms2(seed, wid, st, (uint32_t)(e + lane), tag, 0, u[0], u[1]);
            uniforms2(seed, wid, st, (uint32_t)(e + lane), tag, 1, u[2], u[3]);
#pragma unroll
            for (int d = 0; d < 3; ++d) {
              const double x = __dadd_rn(Rc[d], __dmul_rn(step, __dsub_rn(__dmul_rn(2.0, u[d]), 1.0)));
              rtab[3 * lane + d] = x;
              if constexpr (!kSameType<Tb, double>) rtds[3 * lane + d] = ds_from_double(x);
            }
            uac = u[3];
          }
          __syncwarp();
          // nuclei: Rbar at the proposals and the change of the e-n terms
          for (DivStep ia(lane, Nn); ia.hi < cnt; ia.next(Nn)) {
            const int i = ia.hi, a = ia.lo;
            Tb dn[3], dc[3];
#pragma unroll
            for (int d = 0; d < 3; ++d) {
              if constexpr (kSameType<Tb, double>) dn[d] = (Tb)(rtab[3 * i + d] - __ldg(s.nuc4 + 4 * a + d));
              else dn[d] = ds_diff_f(rtds[3 * i + d], nuc_coord_ds(s, a, d));
              dc[d] = C.en(s, e + i, a, d);
            }
            const PadeT<Tb> c = en_coef_t<Tb>(s, a);
            const Tb rn_ = vsqrt(dn[0] * dn[0] + dn[1] * dn[1] + dn[2] * dn[2]);
            const Tb rc_ = vsqrt(dc[0] * dc[0] + dc[1] * dc[1] + dc[2] * dc[2]);
            const Tb sn = (Tb)1 / ((Tb)1 + kap * rn_), sc = (Tb)1 / ((Tb)1 + kap * rc_);
            svn[i * Nn + a] = sn;
            den[i * Nn + a] = pade_value<Tb>(c, rn_, sn) - pade_value<Tb>(c, rc_, sc);
          }
        }
        const int p0 = L.all ? e : 0;  // the spin's first electron among the prepared ones
        const int nr = L.rows ? (e == 0 ? N : 0) : (L.all ? n : cnt);
        // orbital rows at the proposals (bulk type)
        if constexpr (kSameType<Tb, double>) {
          for (int i = 0; i < nr; ++i) {
            const double* r = rtab + 3 * (p0 + i);
            basis_at<double, false>(s, lane, r[0], r[1], r[2], bas, nullptr, nullptr, nullptr, nullptr);
            __syncwarp();
            for (int c0 = 0; c0 < s.n_occ_chunk[sp]; c0 += 32) {
              const int c = c0 + lane;
              double v = 0.0;
              if (c < s.n_occ_chunk[sp]) {
                const int4 ch = __ldg(reinterpret_cast<const int4*>(s.occ_chunk[sp]) + c);
                const double* cb = s.orb_coef + ch.w;
                for (int mu = ch.y; mu < ch.z; ++mu) v += __ldg(cb + mu) * bas[mu];
              }
              if (L.alias) __syncwarp();
              if (c < s.n_occ_chunk[sp]) part[c] = v;
            }
            __syncwarp();
            for (int q = lane; q < s.nocc[sp]; q += 32) {
              const int c0 = __ldg(s.occ_chunk_off[sp] + q), c1 = __ldg(s.occ_chunk_off[sp] + q + 1);
              double v = 0.0;
              for (int c = c0; c < c1; ++c) v += part[c];
              vrows[i * ldo + q] = v;
            }
            __syncwarp();
          }
        } else {
          for (int i = 0; i < nr;) {
            const int left = nr - i;
            const dsf* r = rtds + 3 * (p0 + i);
            float* out = vrows + i * ldo;
            if (L.ke == 4 && left > 2) {
              proposal_rows<4, BATCH>(s, lane, sp, min(left, 4), r, bas, part, L.alias, out, ldo);
              i += 4;
            } else if (L.ke >= 2 && left > 1) {
              proposal_rows<2, BATCH>(s, lane, sp, 2, r, bas, part, L.alias, out, ldo);
              i += 2;
            } else {
              proposal_rows<1, BATCH>(s, lane, sp, 1, r, bas, part, L.alias, out, ldo);
              ++i;
            }
          }
        }
        __syncwarp();
      }
      if (TAB && (e == 0 || e == Nup)) {
        // the moving spin's weights g_u and Sigma: the other spin's minors stay until the next spin
        const double* wo = wk + (sp ? 0 : s.tab[0].nv);
        const double* wm = wk + (sp ? s.tab[0].nv : 0);
        double sg = 0.0;
        for (int u = lane; u < s.U[sp]; u += 32) {
          const int ud = u + (sp ? U0 : 0);
          double g = 0.0;
          for (int t = __ldg(s.det_term_off + ud); t < __ldg(s.det_term_off + ud + 1); ++t) {
            const int k = __ldg(s.det_term + t);
            g = fma(__ldg(s.tab_coef + k), wo[__ldg(s.term_det + 2 * k + 1 - sp)], g);
          }
          gw[u] = g;
          sg = fma(wm[u], g, sg);
        }
        Sig = warp_sum(sg);
        iSig = nonzero(Sig) ? recip(Sig) : 0.0;
        __syncwarp();
      }
      const int ip = L.all ? e : e - e0;  // its place among the prepared electrons
      const double uacc = __shfl_sync(kFull, uac, ip);
      auto dnew_e = [&](int j, int d) -> Tb {  // proposed position minus electron j
        if constexpr (kSameType<Tb, double>) return (Tb)(rtab[3 * ip + d] - Rs[3 * j + d]);
        else return ds_diff_f(rtds[3 * ip + d], Rds[3 * j + d]);
      };
      for (int q = lane; q < s.nocc[sp]; q += 32) vrowd[q] = widen(vrows[(L.rows ? e : e - e0) * ldo + q]);
      __syncwarp();
      const LaneGroup lgp(lane, G);
      const int U = s.U[sp], ng = lgp.ng, g = lgp.g, gl = lgp.gl;
      const int* dl = s.det_loc[sp];
      double rphi = 0.0, r0 = 0.0, Sig_new = 0.0;
      if constexpr (TAB) {
        // rho_0, c_x, b = B[:, i] / rho_0 (in cvec), the proposed minors and Sigma'.  The n_x + 1
        // column sums (the last is rho_0) share the warp: PX columns of 32 / PX partial sums.
        const int nx = s.n_x[sp];
        const TabMinors& tm = s.tab[sp];
        const double* B = Binv[sp];
        const double* T = Tt[sp];
        int PX = 1;
        while (PX <= nx && PX < 32) PX <<= 1;
        for (int cb = 0; cb <= nx; cb += PX) {
          const int lg = __ffs(PX) - 1, c = cb + (lane & (PX - 1)), st = 32 >> lg;
          const double* col = c < nx ? T + c : B + ie;
          const int ld = c < nx ? nx : n;
          double a = 0.0;
          if (c <= nx)
            for (int o = lane >> lg; o < n; o += st) a = fma(vrowd[__ldg(dl + o)], col[o * ld], a);
          for (int off = PX; off < 32; off <<= 1) a += __shfl_xor_sync(kFull, a, off);
          if (c < nx && lane < PX) cxv[c] = vrowd[__ldg(s.tab_xl[sp] + c)] - a;
          if (nx >= cb && nx < cb + PX) r0 = __shfl_sync(kFull, a, nx - cb);
        }
        const double ir0 = nonzero(r0) ? recip(r0) : 0.0;
        if (lane < n) cvec[lane] = B[lane * n + ie] * ir0;
        __syncwarp();
        for (DivStep ox(lane, max(nx, 1)); ox.hi < tm.ns && nx > 0; ox.next(nx)) {
          const int o = __ldg(tm.sl + ox.hi);
          Tn[ox.hi * nx + ox.lo] = fma(cvec[o], cxv[ox.lo], T[o * nx + ox.lo]);
        }
        __syncwarp();
        tab_values<true, true>(tm, lane, Tn, qn);
        double sg = 0.0;
        for (int u = lane; u < U; u += 32) sg = fma(qn[u], gw[u], sg);
        Sig_new = warp_sum(sg);
        rphi = (nonzero(r0) && nonzero(Sig)) ? r0 * Sig_new * iSig : 0.0;
        if (!finite_bits(rphi)) rphi = 0.0;  // an overflowing ratio is rejected (the tables are refreshed)
      }
      // determinant ratios rho_u = sum_o v_occ(o) Binv_u[o][ie], RG lanes per determinant.  With
      // one pass over the determinants (the usual case) the lanes' products are formed here and
      // reduced after the Jastrow distances below, whose float work then covers their latency.
      const int RG = sp ? L.RG1 : L.RG0;
      const LaneGroup lgr(lane, RG);
      const bool one_pass = U <= lgr.ng;
      const int ur = lgr.g;
      double rpart = 0.0;
      if constexpr (!TAB) {
        if (one_pass) {
          if (ur < U) {
            const double* Bu = Binv[sp] + ur * n * n + ie;
            const int* du = dl + ur * n;
            for (int o = lgr.gl; o < n; o += RG) rpart = fma(vrowd[__ldg(du + o)], Bu[o * n], rpart);
          }
        } else {
          for (int ub = 0; ub < U; ub += lgr.ng) {
            const int u = ub + lgr.g;
            double r = 0.0;
            if (u < U) {
              const double* Bu = Binv[sp] + u * n * n + ie;
              const int* du = dl + u * n;
              for (int o = lgr.gl; o < n; o += RG) r = fma(vrowd[__ldg(du + o)], Bu[o * n], r);
            }
            r = group_sum(r, RG);
            if (u < U && lgr.gl == 0) rho[u] = r;
          }
        }
      }
      // Jastrow change of the terms that involve electron e (Sec. 2.1): items e-n (a) and e-e (j),
      // then e-e-n (a, part of the partners) through the pair sums Y^{k,q} = sum_{j != e} u_ej^k s_j^q
      // (the terms of e are s_e^A Y^{k,B} + s_e^B Y^{k,A}).
      Tb dj = 0;
      for (int t = lane; t < Nn + N; t += 32) {
        if (t < Nn) {
          dj += den[ip * Nn + t];
          continue;
        }
        const int j = t - Nn;
        if (j == e) continue;
        const bool same = (e < Nup) == (j < Nup);
        Tb un, f1, uo, f0;
        pair_values(dnew_e(j, 0), dnew_e(j, 1), dnew_e(j, 2), same, un, f1);
        if (L.tri) {
          const int p = tri(e, j);
          uo = ut[p];
          f0 = ft[p];
          ue[j] = un;
          fe[j] = f1;
        } else {
          pair_values(C.ee(e, j, 0), C.ee(e, j, 1), C.ee(e, j, 2), same, uo, f0);
        }
        dj += f1 - f0;
        const Pair2<Tb> u1{uo, un};
        Pair2<Tb> pw = u1;
#pragma unroll
        for (int k = 0; k < 4; ++k) {
          Up[k * UP + j] = pw;
          pw = pair_mul(pw, u1);
        }
      }
      if constexpr (!TAB) {
        if (one_pass) {
          rpart = group_sum(rpart, RG);
          if (ur < U && lgr.gl == 0) rho[ur] = rpart;
        }
      }
      __syncwarp();
      if constexpr (!TAB) {
        // the structure sum's per-lane parts; they are reduced after the Jastrow change,
        // together with its sum: the double reduction's latency then overlaps the float work
        for (int k = lane; k < s.nterm; k += 32)
          rphi += __ldg(s.term_coef + k) * wk[k] * rho[__ldg(s.term_det + 2 * k + sp)];
      }
      if (s.een_on) {
        // e-e-n items (nucleus a, part of the partners j), every k in each: the pair sums
        // are linear in the partners, so each part adds its own share of the change, and all
        // lanes run the same code (no divergence over k)
        for (int a = ea0; a < Nn; a += (np > 1 ? Nn : 32)) {
          Tb Y0[6];
          Pair2<Tb> Y[4][5];  // k - 1, q <= 5 - k
#pragma unroll
          for (int q = 0; q < 6; ++q) Y0[q] = (Tb)0;
#pragma unroll
          for (int k = 0; k < 4; ++k)
#pragma unroll
            for (int q = 0; q < 5; ++q) Y[k][q] = {(Tb)0, (Tb)0};
          for (int j = ej0; j < ej1; ++j) {
            if (j == e) continue;
            const Tb svj = Sv[a * SA + j];
            const Pair2<Tb> s1{svj, svj};
            Pair2<Tb> sj[6];
            sj[1] = s1;
#pragma unroll
            for (int q = 2; q < 6; ++q) sj[q] = pair_mul(sj[q - 1], s1);
#pragma unroll
            for (int q = 1; q < 6; ++q) Y0[q] += sj[q].o;
#pragma unroll
            for (int k = 0; k < 4; ++k) {
              const Pair2<Tb> u = Up[k * UP + j];
              Y[k][0] = pair_add(Y[k][0], u);
#pragma unroll
              for (int q = 1; q <= 4 - k; ++q) Y[k][q] = pair_fma(u, sj[q], Y[k][q]);
            }
          }
          Pair2<Tb> S[6];
          S[0] = {(Tb)1, (Tb)1};
          S[1] = {Sv[a * SA + e], svn[ip * Nn + a]};
#pragma unroll
          for (int q = 2; q < 6; ++q) S[q] = pair_mul(S[q - 1], S[1]);
          const Tb* c = cE + kNeen * __ldg(s.nuc_elem + a);
          een_for_each([&](auto tc) {
            constexpr int q = decltype(tc)::value;
            constexpr int tk = een_klm(q).k, A = een_klm(q).l + een_klm(q).m, B = een_klm(q).m;
            Pair2<Tb> YA, YB;
            if constexpr (tk == 0) {
              YA = {Y0[A], Y0[A]};
              YB = {Y0[B], Y0[B]};
            } else {
              YA = Y[tk - 1][A];
              YB = Y[tk - 1][B];
            }
            const Pair2<Tb> x = pair_fma(S[A], YB, pair_mul(S[B], YA));
            dj += c[q] * (x.n - x.o);
          });
        }
      }
      Tb dJ;
      if constexpr (TAB) {
        dJ = warp_sum(dj);
      } else {
#pragma unroll
        for (int o = 16; o > 0; o >>= 1) {
          rphi += __shfl_xor_sync(kFull, rphi, o);
          dj += __shfl_xor_sync(kFull, dj, o);
        }
        dJ = dj;
      }
      double ej;
      if constexpr (kSameType<Tb, double>) ej = vexp(2.0 * dJ);
      else ej = f2d_bits(vexp(2.0f * dJ));
      const double prob = rphi * rphi * ej;
      const bool acc = less_nonneg(uacc, prob);  // uacc in [0, 1), prob >= 0 or NaN
      if (TAB && acc) {
        // T <- T + b c^T; B <- B - b w^T with w = v^T B - e_i (lane j owns w_j); q <- q'
        const int nx = s.n_x[sp], vo = sp ? s.tab[0].nv : 0;
        double* T = Tt[sp];
        double* B = Binv[sp];
        for (DivStep ox(lane, max(nx, 1)); ox.hi < n && nx > 0; ox.next(nx)) {
          double& t = T[ox.hi * nx + ox.lo];
          t = fma(cvec[ox.hi], cxv[ox.lo], t);
        }
        if (lane < n) {
          const int j = lane;
          double w0 = (j == ie) ? -1.0 : 0.0, w1 = 0.0;
          int o = 0;
          for (; o + 1 < n; o += 2) {
            w0 = fma(vrowd[__ldg(dl + o)], B[o * n + j], w0);
            w1 = fma(vrowd[__ldg(dl + o + 1)], B[(o + 1) * n + j], w1);
          }
          if (o < n) w0 = fma(vrowd[__ldg(dl + o)], B[o * n + j], w0);
          wrow[j] = w0 + w1;
        }
        __syncwarp();
        for (DivStep oj(lane, n); oj.hi < n; oj.next(n)) {
          double& x = B[oj.hi * n + oj.lo];
          x = fma(-cvec[oj.hi], wrow[oj.lo], x);
        }
        for (int u = lane; u < s.tab[sp].nv; u += 32) wk[vo + u] = qn[u];
        Sig = Sig_new;
        iSig = recip(Sig);  // an accepted ratio is nonzero, so Sigma is
        accept_position(e, ip);
        ++accepted;
      } else if (!TAB && acc) {
        // the reciprocals 1/rho_u and 1/(Phi'/Phi), one per lane
        for (int q = lane; q <= U; q += 32) rinv[q] = recip(q < U ? rho[q] : rphi);
        __syncwarp();
        // Sherman-Morrison: Binv <- Binv - Binv[:, ie] (v^T Binv - e_ie^T) / rho, two lane-group
        // passes at a time (determinants u and u + ng): their row products are independent
        // chains, so each hides the other's latency without extra double instructions
        for (int ub = 0; ub < U; ub += 2 * ng) {
          const int ua = ub + g, uc = ub + ng + g;
          const bool aa = ua < U, ac = uc < U, two = ub + ng < U;  // ac implies aa; two: warp-uniform
          double* Ba = Binv[sp] + (aa ? ua : 0) * n * n;
          double* Bc = Binv[sp] + (ac ? uc : 0) * n * n;
          double* cva = cvec + g * n;
          double* cvc = cvec + (ng + g) * n;
          if (aa && gl < n) cva[gl] = Ba[gl * n + ie];
          if (ac && gl < n) cvc[gl] = Bc[gl * n + ie];
          const double ira = aa ? rinv[ua] : 0.0, irc = ac ? rinv[uc] : 0.0;
          __syncwarp();
          if (aa && gl < n) {
            const int j = gl;
            const int* da = dl + ua * n;
            const int* dc = dl + (ac ? uc : ua) * n;
            double wa = (j == ie) ? -1.0 : 0.0, wc = wa;
            if (two) {
              for (int o = 0; o < n; ++o) {
                wa = fma(vrowd[__ldg(da + o)], Ba[o * n + j], wa);
                if (ac) wc = fma(vrowd[__ldg(dc + o)], Bc[o * n + j], wc);
              }
            } else {
              for (int o = 0; o < n; ++o) wa = fma(vrowd[__ldg(da + o)], Ba[o * n + j], wa);
            }
            const double fa = wa * ira, fc = wc * irc;
            for (int o = 0; o < n; ++o) {
              Ba[o * n + j] = fma(-cva[o], fa, Ba[o * n + j]);
              if (ac) Bc[o * n + j] = fma(-cvc[o], fc, Bc[o * n + j]);
            }
          }
          __syncwarp();
        }
        const double irphi = rinv[U];
        {
          const long long b = __double_as_longlong(fabs(rphi) * pm);
          pe += (int)((b >> 52) & 0x7ff) - 1023;
          pm = __longlong_as_double((b & 0x800fffffffffffffLL) | (1023LL << 52));
        }
        // an accepted rphi is nonzero: its sign bit is its sign; flip sgnPhi's sign bit
        if (__double_as_longlong(rphi) < 0)
          sgnPhi = __longlong_as_double(__double_as_longlong(sgnPhi) ^ (long long)0x8000000000000000ull);
        for (int k = lane; k < s.nterm; k += 32) wk[k] *= rho[__ldg(s.term_det + 2 * k + sp)] * irphi;
        accept_position(e, ip);
        ++accepted;
      }
      __syncwarp();
    }
  }
  if (nacc && lane == 0) nacc[w] += accepted;
  lnPhi += log(pm) + (double)pe * 0.69314718055994530942;  // ln 2
  if (!TAB && state) {  // the carried inverses, term ratios and ln|Phi| at the final positions
    double* st = state + (size_t)w * s.state_doubles;
    for (int q = lane; q < nb0; q += 32) st[q] = Binv[0][q];
    for (int q = lane; q < nb1; q += 32) st[nb0 + q] = Binv[1][q];
    for (int k = lane; k < s.nterm; k += 32) st[nb0 + nb1 + 2 * Ut + k] = wk[k];
    if (lane == 0) {
      st[nb0 + nb1 + 2 * Ut + s.nterm] = lnPhi;
      st[nb0 + nb1 + 2 * Ut + s.nterm + 1] = sgnPhi;
    }
  }
}

}  // namespace vbq
