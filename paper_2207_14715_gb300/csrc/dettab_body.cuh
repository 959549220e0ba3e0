// Per-walker body of the determinant kernel on reference-determinant tables (arXiv:2207.14715,
// Sec. 2.1 determinant expansion): shared by the single-system and the fused batch kernels.
#pragma once

#include "tab_minors.cuh"
#include "walker_common.cuh"

namespace vbq {

namespace {

// ALONE: whether the system may hold determinants formed by themselves.
template <class Tb, bool ALONE>
__device__ __forceinline__ void dettab_body(const SysDev& s, const DetTabLayout& L, int w, unsigned char* base,
                                            const Tb* JG, const Tb* JL, const double* JS, const Tb* OB,
                                            const double* OD, double* __restrict__ logpsi,
                                            double* __restrict__ sgn_out, double* __restrict__ eloc,
                                            double* __restrict__ vg_ws, double* __restrict__ grad,
                                            Tb* __restrict__ Og, Tb* __restrict__ dELg) {
  const int lane = threadIdx.x & 31;
  const int N = s.N, Nup = s.Nup, U0 = s.U[0];
  const int nev = s.n_ev, nevd = s.n_ev_det;
  double* vg = reinterpret_cast<double*>(base + L.vg);
  double* Bd[2] = {reinterpret_cast<double*>(base + L.B0), reinterpret_cast<double*>(base + L.B1)};
  double* TX[2] = {reinterpret_cast<double*>(base + L.T0), reinterpret_cast<double*>(base + L.T1)};
  double* V[2] = {reinterpret_cast<double*>(base + L.v0), reinterpret_cast<double*>(base + L.v1)};
  int* perm = reinterpret_cast<int*>(base + L.perm);
  double* Tn = reinterpret_cast<double*>(base + L.Tn);    // [ns][nx] the rows of T that the minors read
  double* PX = reinterpret_cast<double*>(base + L.PX);    // [n][nx] Phi_X, then staged cofactors, then (with derivatives) L_X - L_0 T
  double* Ls = reinterpret_cast<double*>(base + L.Ls);    // [n][nevd] dressed Laplacian of the spin's electrons
  double* adj = reinterpret_cast<double*>(base + L.adj);
  double* gT = reinterpret_cast<double*>(base + L.gT);    // [ns][nx] Gamma
  double* Gam = reinterpret_cast<double*>(base + L.Gam);  // [nx][n] h = Gamma B
  double* tdet = reinterpret_cast<double*>(base + L.tdet);  // t_u of both spins, with derivatives only
  Tb* G = reinterpret_cast<Tb*>(base + L.G);

  for (int q = lane; q < 3 * N; q += 32) G[q] = JG[(size_t)w * 3 * N + q];
  const double lnJ = JS[2 * (size_t)w], V_pot = JS[2 * (size_t)w + 1];
  __syncwarp();

  // ---- per spin: inverse of the reference, T and every minor ----
  double lg0 = 0.0;
  int sg0 = 1;
  for (int sp = 0; sp < 2; ++sp) {
    const int n = s.n[sp], e0 = sp ? Nup : 0, nx = s.n_x[sp];
    const TabMinors& tm = s.tab[sp];
    if (n > 0) {
      const double* od = OD + ((size_t)w * N + e0) * nevd;
      for (DivStep ex(lane, max(nx, 1)); ex.hi < n && nx > 0; ex.next(nx))
        PX[ex.hi * nx + ex.lo] = od[ex.hi * nevd + __ldg(s.tab_x[sp] + ex.lo)];
      double* B = Bd[sp];
      const GroupDet d = warp_inverse(od, nevd, s.det_ev[sp], n, perm, B);
      const int sg = d.sgn;
      sg0 *= sg;
      lg0 += sg != 0 ? log(d.mant) + (double)d.ex * 0.6931471805599453
                     : 0.0;
      double* T = TX[sp];  // T = B Phi_X
      for (DivStep ox(lane, max(nx, 1)); ox.hi < n && nx > 0; ox.next(nx)) {
        double a = 0.0;
        for (int e = 0; e < n; ++e) a = fma(B[ox.hi * n + e], PX[e * nx + ox.lo], a);
        T[ox.hi * nx + ox.lo] = a;
      }
      __syncwarp();
      for (DivStep rx(lane, max(nx, 1)); rx.hi < tm.ns && nx > 0; rx.next(nx))
        Tn[rx.hi * nx + rx.lo] = T[__ldg(tm.sl + rx.hi) * nx + rx.lo];
      __syncwarp();
    }
    tab_values<ALONE, false>(tm, lane, Tn, V[sp]);
  }

  // ---- structure sum: Sigma = sum_k C_k q_up(k) q_dn(k), each spin's minors scaled by a power of
  // two so that the largest lies in [1, 2) (ln|Phi| takes the exponents) ----
  double scale[2];
  int esum = 0;
  for (int sp = 0; sp < 2; ++sp) {
    unsigned top = 0;
    for (int u = lane; u < s.U[sp]; u += 32) top = max(top, (unsigned)__double2hiint(V[sp][u]) & 0x7ff00000u);
    for (int o = 16; o > 0; o >>= 1) top = max(top, __shfl_xor_sync(kFull, top, o));
    const int e = min(max((int)(top >> 20) - 1023, -1000), 1000);
    scale[sp] = __longlong_as_double((long long)(1023 - e) << 52);
    esum += e;
  }
  // g_u of a determinant: sum over its terms of C_k times the other spin's minor (scaled)
  auto weight = [&](int sp, int u) {
    const int ud = u + (sp ? U0 : 0);
    double g = 0.0;
    for (int t = __ldg(s.det_term_off + ud); t < __ldg(s.det_term_off + ud + 1); ++t) {
      const int k = __ldg(s.det_term + t);
      g = fma(__ldg(s.tab_coef + k), V[1 - sp][__ldg(s.term_det + 2 * k + 1 - sp)], g);
    }
    return g * scale[1 - sp];
  };
  double Sig = 0.0;
  for (int u = lane; u < U0; u += 32) {
    const double g = weight(0, u);
    adj[u] = g;
    Sig = fma(V[0][u] * scale[0], g, Sig);
  }
  Sig = warp_sum(Sig);
  const bool ok = sg0 != 0 && nonzero(Sig);
  const double iS = ok ? 1.0 / Sig : 0.0;
  const double lnPhi = ok ? lg0 + log(fabs(Sig)) + (double)esum * 0.6931471805599453 : -INFINITY;
  const double sgnPhi = ok ? (Sig > 0.0 ? (double)sg0 : -(double)sg0) : 0.0;
  __syncwarp();

  // ---- per spin: Gamma = d ln Sigma / d T from adj_u = d ln Sigma / d q_u, then C and h, the
  // derivatives of ln|Phi| with respect to the orbital values; K[Phi]/Phi and grad_i ln|Phi| ----
  double kin_loc = 0.0, kphi_loc = 0.0;
  for (int sp = 0; sp < 2; ++sp) {
    const int n = s.n[sp], e0 = sp ? Nup : 0, nx = s.n_x[sp], U = s.U[sp];
    const TabMinors& tm = s.tab[sp];
    if (n == 0) {
      for (int u = lane; u < U; u += 32) tdet[u + (sp ? U0 : 0)] = 0.0;
      continue;
    }
    const int* ref = s.det_ev[sp];
    const int* xl = s.tab_x[sp];
    double* B = Bd[sp];
    const double* T = TX[sp];
    const double f = iS * scale[sp];
    for (int u = lane; u < U; u += 32) adj[u] = (sp == 0 ? adj[u] : weight(1, u)) * f;
    for (DivStep rx(lane, max(nx, 1)); rx.hi < tm.ns && nx > 0; rx.next(nx))
      Tn[rx.hi * nx + rx.lo] = T[__ldg(tm.sl + rx.hi) * nx + rx.lo];
    for (DivStep eq(lane, nevd); eq.hi < n; eq.next(nevd)) {
      const Tb* ob = OB + ((size_t)w * N + e0 + eq.hi) * 5 * nev + eq.lo;
      const Tb* g = G + 3 * (e0 + eq.hi);
      const double d = widen(g[0]) * widen(ob[nev]) + widen(g[1]) * widen(ob[2 * nev]) + widen(g[2]) * widen(ob[3 * nev]);
      Ls[eq.hi * nevd + eq.lo] = fma(2.0, d, widen(ob[4 * nev]));
    }
    __syncwarp();
    tab_adjoint<ALONE>(tm, lane, Tn, V[sp], adj, gT, PX, L.sd);
    // h[x][i] = sum_o Gamma[o][x] B[o][i]
    for (DivStep xe(lane, n); xe.hi < nx; xe.next(n)) {
      double h = 0.0;
      for (int r = 0; r < tm.ns; ++r) h = fma(gT[r * nx + xe.hi], B[__ldg(tm.sl + r) * n + xe.lo], h);
      Gam[xe.hi * n + xe.lo] = h;
      kphi_loc = fma(h, Ls[xe.lo * nevd + __ldg(xl + xe.hi)], kphi_loc);
    }
    __syncwarp();
    if (Og) {  // per determinant t_u = tr(B L_0) + (d q_u along Yhat) / q_u, Yhat = B (L_X - L_0 T)
      double t0 = 0.0;
      for (DivStep oe(lane, n); oe.hi < n; oe.next(n))
        t0 = fma(B[oe.hi * n + oe.lo], Ls[oe.lo * nevd + __ldg(ref + oe.hi)], t0);
      t0 = warp_sum(t0);
      for (DivStep ex(lane, max(nx, 1)); ex.hi < n && nx > 0; ex.next(nx)) {
        double a = Ls[ex.hi * nevd + __ldg(xl + ex.lo)];
        for (int o = 0; o < n; ++o) a = fma(-Ls[ex.hi * nevd + __ldg(ref + o)], T[o * nx + ex.lo], a);
        PX[ex.hi * nx + ex.lo] = a;
      }
      __syncwarp();
      for (DivStep rx(lane, max(nx, 1)); rx.hi < tm.ns && nx > 0; rx.next(nx)) {
        const int o = __ldg(tm.sl + rx.hi);
        double a = 0.0;
        for (int e = 0; e < n; ++e) a = fma(B[o * n + e], PX[e * nx + rx.lo], a);
        gT[rx.hi * nx + rx.lo] = a;
      }
      __syncwarp();
      double* td = tdet + (sp ? U0 : 0);
      tab_derivatives<ALONE>(tm, U, lane, Tn, V[sp], gT, td);
      for (int u = lane; u < U; u += 32) td[u] = nonzero(V[sp][u]) ? t0 + td[u] / V[sp][u] : 0.0;
      __syncwarp();
    }
    // grad_i ln|Phi| = sum_o B[o][i] grad phi_o + sum_x h[x][i] (grad phi_x - sum_o T[o][x] grad phi_o)
    //               = sum_o C[o][i] grad phi_o + sum_x h[x][i] grad phi_x,  C = B - T h
    // (C in double, in place of B, which is not read again; the sums in the bulk type: the
    // gradient feeds the drift and the Jastrow-parameter derivatives, not E_L); the same C and h
    // give K[Phi]/Phi = sum C L_0 + sum h L_X in double: C is of the size of the wave function's own
    // derivatives where the reference is small, and B and the traces t_u are not
    for (DivStep oe(lane, n); oe.hi < n; oe.next(n)) {
      double c = B[oe.hi * n + oe.lo];
      for (int x = 0; x < nx; ++x) c = fma(-T[oe.hi * nx + x], Gam[x * n + oe.lo], c);
      B[oe.hi * n + oe.lo] = c;
      kphi_loc = fma(c, Ls[oe.lo * nevd + __ldg(ref + oe.hi)], kphi_loc);
    }
    __syncwarp();
    for (int e = lane; e < n; e += 32) {
      const Tb* ob = OB + ((size_t)w * N + e0 + e) * 5 * nev;
      Tb g[3] = {0, 0, 0};
#pragma unroll 4
      for (int o = 0; o < n; ++o) {
        const int col = __ldg(ref + o);
        const Tb c = narrow<Tb>(B[o * n + e]);
#pragma unroll
        for (int d = 0; d < 3; ++d) g[d] += c * ob[(1 + d) * nev + col];
      }
      for (int x = 0; x < nx; ++x) {
        const Tb h = narrow<Tb>(Gam[x * n + e]);
        const int colx = __ldg(xl + x);
#pragma unroll
        for (int d = 0; d < 3; ++d) g[d] += h * ob[(1 + d) * nev + colx];
      }
      const int i = e0 + e;
      const double G0 = widen(G[3 * i]), G1 = widen(G[3 * i + 1]), G2 = widen(G[3 * i + 2]);
      vg[3 * i] = G0 + widen(g[0]);
      vg[3 * i + 1] = G1 + widen(g[1]);
      vg[3 * i + 2] = G2 + widen(g[2]);
      kin_loc += widen(JL[(size_t)w * N + i]) + G0 * G0 + G1 * G1 + G2 * G2;
    }
    __syncwarp();
  }
  const double kphi = warp_sum(ok ? kphi_loc : 0.0);
  const double kin = warp_sum(kin_loc) + kphi;
  const double EL = -0.5 * kin + V_pot;
  if (lane == 0) {
    logpsi[w] = lnJ + lnPhi;
    sgn_out[w] = sgnPhi;
    eloc[w] = EL;
  }
  __syncwarp();
  for (int q = lane; q < 3 * N; q += 32) {
    vg_ws[(size_t)w * 3 * N + q] = vg[q];
    if (grad) grad[(size_t)w * 3 * N + q] = vg[q];
  }
  if (!Og) return;
  // structure coefficients: O_I = Phi_I/Phi, E_L,I = -1/2 (K[Phi_I] - O_I K[Phi])
  const int P = s.P;
  Tb* Ow = Og + (size_t)w * P;
  Tb* Ew = dELg ? dELg + (size_t)w * P : nullptr;
  for (int q = lane; q < s.n_cparam; q += 32) {
    double o = 0.0, kk = 0.0;
    for (int ts = __ldg(s.cpar_off + q); ts < __ldg(s.cpar_off + q + 1); ++ts) {
      const int t = __ldg(s.cpar_st + ts), k = __ldg(s.sterm_k + t);
      const int a = __ldg(s.term_det + 2 * k), b = __ldg(s.term_det + 2 * k + 1);
      const double r = __ldg(s.sterm_d + t) * __ldg(s.tab_sgn + k) * (V[0][a] * scale[0]) * (V[1][b] * scale[1]) * iS;
      o += r;
      kk += r * (tdet[a] + tdet[U0 + b]);
    }
    Ow[q] = (Tb)o;
    if (Ew) Ew[q] = (Tb)(-0.5 * (kk - o * kphi));
  }
}

}  // namespace

}  // namespace vbq
