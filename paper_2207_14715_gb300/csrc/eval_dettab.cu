// Determinant part of the evaluation through a reference determinant and tables
// (arXiv:2207.14715, Sec. 2.1: every determinant of a spin shares the inactive orbitals and
// differs from the others by a few active columns), for systems whose per-determinant
// inverses do not fit in shared memory.  One warp per walker.  Per spin:
//   A_0 = reference determinant (u = 0), B = A_0^-1 by the whole-warp Gauss-Jordan (double);
//   T = B Phi_X over the orbitals X outside the reference;
//   determinant u replaces the reference slots S_u by the orbitals Q_u (k_u <= 4):
//     D_u = sgn_u D_0 q_u,  q_u = det T[S_u, Q_u]  (tab_minors.cuh).
// With Sigma = sum_k C_k q_up(k) q_dn(k) the derivatives of ln|Phi| with respect to the orbital
// values phi_o(r_i) and phi_x(r_i) are
//   h[x][i] = sum_o Gamma[o][x] B[o][i],  C[o][i] = B[o][i] - sum_x T[o][x] h[x][i],
//   Gamma[o][x] = d ln Sigma / d T[o][x] = sum_u (d ln Sigma / d q_u) (cofactor of (o, x) in q_u),
// which give grad_i ln|Phi| and, on the Jastrow-dressed Laplacians L = lap phi + 2 grad ln J . grad phi,
// K[Phi]/Phi.  The traces t_u = tr(A_u^-1 L_u) are formed for structure-coefficient derivatives only.
//
// Bound: the FP64 pipe (about 2400 instructions per walker on 48 electrons, a quarter of them the
// two inverses) and latency at 10 walkers per SM (22.5 KB each): 0.85 ms per 4096 walkers,
// 2.36 with traces and inverses of every determinant's own minor (36 KB, 6 walkers per SM).
#include "dettab_body.cuh"

namespace vbq {

namespace {
constexpr int kDetTabWarps = 12;
// ALONE: for systems with determinants formed by themselves (tab_minors.cuh), whose functions would cost the
// others registers (an evaluation of 4096 walkers with 10 active orbitals 0.49 in place of 0.41 ms).
// 512: at most 128 registers, so that small blocks can put 16 warps on an SM (without spills; 137 otherwise).
template <class Tb, bool ALONE>
__global__ void __launch_bounds__(ALONE ? 512 : 32 * kDetTabWarps, 1)
    dettab_kernel(const SysDev s, const DetTabLayout L, int W, const Tb* __restrict__ JG, const Tb* __restrict__ JL,
                  const double* __restrict__ JS, const Tb* __restrict__ OB, const double* __restrict__ OD,
                  double* __restrict__ logpsi, double* __restrict__ sgn_out, double* __restrict__ eloc,
                  double* __restrict__ vg_ws, double* __restrict__ grad, Tb* __restrict__ Og, Tb* __restrict__ dELg) {
  extern __shared__ __align__(16) unsigned char smem[];
  const int wl = threadIdx.x >> 5;
  const int w = blockIdx.x * L.wpb + wl;
  if (w >= W) return;
  dettab_body<Tb, ALONE>(s, L, w, smem + wl * L.warp_bytes, JG, JL, JS, OB, OD, logpsi, sgn_out, eloc, vg_ws, grad, Og,
                         dELg);
}

}  // namespace

int make_dettab_layout(const SysDev& s, int tb, int max_smem, DetTabLayout& L) {
  int off = 0;
  auto take = [&](int bytes) {
    const int o = off;
    off = align16(off + bytes);
    return o;
  };
  const int N = s.N, nevd = std::max(s.n_ev_det, 1);
  const TabMinors* m = s.tab;
  const int nmax = std::max(std::max(s.n[0], s.n[1]), 1);
  const int nx = std::max(std::max(s.n[0] * s.n_x[0], s.n[1] * s.n_x[1]), 1);
  const int nt = std::max(std::max(m[0].ns * s.n_x[0], m[1].ns * s.n_x[1]), 1);
  L.vg = take(8 * 3 * N);
  L.G = take(tb * 3 * N);
  L.B0 = take(8 * std::max(s.n[0] * s.n[0], 1));
  L.B1 = take(8 * std::max(s.n[1] * s.n[1], 1));
  L.T0 = take(8 * std::max(s.n[0] * s.n_x[0], 1));
  L.T1 = take(8 * std::max(s.n[1] * s.n_x[1], 1));
  L.v0 = take(8 * m[0].nv);
  L.v1 = take(8 * m[1].nv);
  L.tdet = take(8 * (s.U[0] + s.U[1]));
  L.perm = take(4 * nmax);
  L.Tn = take(8 * nt);
  L.Ls = take(8 * nmax * nevd);
  L.adj = take(8 * std::max(s.U[0], s.U[1]));
  L.gT = take(8 * nt);
  L.Gam = take(8 * nx);
  // Phi_X, and over it the cofactors of 32 determinants formed by themselves, of fewer where these
  // would not fit (with the shared memory that a batched launch keeps for itself)
  L.sd = m[0].nd + m[1].nd > 0 ? 32 : 1;
  while (16 * L.sd > nx && L.sd > 1 && off + 128 * L.sd > max_smem - 1024) L.sd /= 2;
  L.PX = take(8 * (m[0].nd + m[1].nd > 0 ? std::max(nx, 16 * L.sd) : nx));
  L.warp_bytes = off;
  int wpb = max_smem / off;
  if (wpb > kDetTabWarps) wpb = kDetTabWarps;
  if (wpb < 1) return VBQMC_ERR_CAPACITY;
  L.wpb = wpb;
  return VBQMC_OK;
}

template <class Tb>
cudaError_t launch_dettab(const SysDev& s, const DetTabLayout& L, int W, const Tb* JG, const Tb* JL, const double* JS,
                          const Tb* OB, const double* OD, double* logpsi, double* sign, double* eloc, double* vg_ws,
                          double* grad, Tb* O, Tb* dEL, cudaStream_t st) {
  DetTabLayout D = L;
  D.wpb = walkers_per_block(W, L.wpb, kDetTabWarps, L.warp_bytes);
  const int smem = D.wpb * D.warp_bytes;
  const auto kernel = s.tab[0].nd + s.tab[1].nd > 0 ? dettab_kernel<Tb, true> : dettab_kernel<Tb, false>;
  cudaError_t e = open_shared_memory((const void*)kernel);
  if (e != cudaSuccess) return e;
  kernel<<<(W + D.wpb - 1) / D.wpb, 32 * D.wpb, smem, st>>>(s, D, W, JG, JL, JS, OB, OD, logpsi, sign, eloc, vg_ws, grad,
                                                            O, dEL);
  return cudaGetLastError();
}
template cudaError_t launch_dettab<float>(const SysDev&, const DetTabLayout&, int, const float*, const float*,
                                          const double*, const float*, const double*, double*, double*, double*,
                                          double*, double*, float*, float*, cudaStream_t);
template cudaError_t launch_dettab<double>(const SysDev&, const DetTabLayout&, int, const double*, const double*,
                                           const double*, const double*, const double*, double*, double*, double*,
                                           double*, double*, double*, double*, cudaStream_t);

}  // namespace vbq
