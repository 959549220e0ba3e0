// VMC sweep kernel for sm_103a (arXiv:2207.14715, Sec. 2.3.1): one warp per walker, the
// walker's inverses and tables in shared memory.  (The evaluation kernels are in
// eval_jastrow.cu, eval_orbitals.cu and eval_det.cu.)
//
// Precision: template parameter Tb is the bulk type (proposal rows and Jastrow changes); the
// determinant ratios and Sherman-Morrison updates of the inverses are always double.
#include "sweep_body.cuh"

namespace vbq {

template <class Tb, bool TAB>
__global__ void __launch_bounds__(512, 1) sweep_kernel(const SysDev s, const SweepLayout L, int W, double* __restrict__ Rg,
                                                    int nsweeps, int refresh, double* __restrict__ state, int state_valid,
                                                    double step, uint64_t seed, uint32_t step0, uint32_t tag,
                                                    uint32_t woff, int* __restrict__ nacc) {
  extern __shared__ __align__(16) unsigned char smem[];
  const int wl = threadIdx.x >> 5;
  const int w = blockIdx.x * L.wpb + wl;
  if (w >= W) return;
  sweep_body<Tb, TAB, false>(s, L, w, smem + wl * L.warp_bytes, Rg, nsweeps, refresh, state, state_valid, step, seed, step0,
                      tag, woff, nacc);
}

// All systems of a batch: blocks loop over work items; warp wl takes walker first + wl.
template <class Tb>
__global__ void __launch_bounds__(512, 1) sweep_batch_kernel(const BatchSys* __restrict__ sys,
                                                          const BatchItem* __restrict__ items, int nitems,
                                                          const BatchCall* __restrict__ call) {
  extern __shared__ __align__(16) unsigned char smem[];
  const int wl = threadIdx.x >> 5;
  for (int it = blockIdx.x; it < nitems; it += gridDim.x) {
    // the warps' shared-memory regions depend on the item's system: start together
    __syncthreads();
    const BatchItem item = items[it];
    if (wl >= item.count) continue;
    const BatchSys& b = sys[item.sys];
    sweep_body<Tb, false, true>(b.dev, b.sweep, item.first + wl, smem + wl * b.sweep.warp_bytes, b.R, call->nsweeps,
                                call->refresh, b.state, call->state_valid, call->step, call->seed, call->step0, b.tag,
                                0u, b.nacc);
  }
}

// =====================================================================================
// layouts and launchers
// =====================================================================================
int make_sweep_layout(const SysDev& s, int tb, int max_smem, SweepLayout& L) {
  int off = 0;
  auto take = [&](int bytes) {
    const int o = off;
    off = align16(off + bytes);
    return o;
  };
  const int N = s.N, Ut = s.U[0] + s.U[1];
  L.tab = s.msd ? 1 : 0;
  L.G0 = group_size(s.n[0]);
  L.G1 = group_size(s.n[1]);
  // a double instruction costs the same whatever the number of active lanes: the ratios take
  // the lane-group size with the fewest double instructions per move (passes over the
  // determinants times the products per lane plus the reduction levels)
  auto ratio_group = [](int n, int U, int G) {
    int best = G, bc = 1 << 30;
    for (int g = 1, lg = 0; g <= G; g <<= 1, ++lg) {
      const int per = 32 / g, c = ((U + per - 1) / per) * ((n + g - 1) / g + lg);
      if (c < bc) {
        bc = c;
        best = g;
      }
    }
    return best;
  };
  L.RG0 = ratio_group(s.n[0], s.U[0], L.G0);
  L.RG1 = ratio_group(s.n[1], s.U[1], L.G1);
  L.nocc_max = std::max(std::max(s.nocc[0], s.nocc[1]), 1);
  L.R = take(8 * 3 * N);  // double, or float pairs
  if (L.tab) {  // reference inverse and tables per spin, q_u of both spins, proposed q_u, c_x
    L.Binv0 = take(8 * s.n[0] * s.n[0]);
    L.Binv1 = take(8 * s.n[1] * s.n[1]);
    L.T0 = take(8 * std::max(s.n[0] * s.n_x[0], 1));
    L.T1 = take(8 * std::max(s.n[1] * s.n_x[1], 1));
    const TabMinors *m = s.tab;
    L.wk = take(8 * (m[0].nv + m[1].nv));
    L.qn = take(8 * std::max(m[0].nv, m[1].nv));
    L.cx = take(8 * std::max(std::max(s.n_x[0], s.n_x[1]), 1));
    L.Tn = take(8 * std::max(std::max(m[0].ns * s.n_x[0], m[1].ns * s.n_x[1]), 1));
    L.gw = take(8 * std::max(s.U[0], s.U[1]));
    L.wrow = take(8 * std::max(s.n[0], s.n[1]));
  } else {
    L.Binv0 = take(8 * s.U[0] * s.n[0] * s.n[0]);
    L.Binv1 = take(8 * s.U[1] * s.n[1] * s.n[1]);
    L.wk = take(8 * s.nterm);
  }
  L.vrow = take(8 * L.nocc_max);
  const int nmax = std::max(s.n[0], s.n[1]), nch = std::max(std::max(s.n_occ_chunk[0], s.n_occ_chunk[1]), 1);
  int cv = 0, scr = 0;
  for (int sp = 0; sp < 2; ++sp) {
    const int n = s.n[sp], G = sp ? L.G1 : L.G0, ng = L.tab ? 1 : 32 / G;
    cv = std::max(cv, 8 * (L.tab ? 1 : 2) * ng * n);  // Sherman-Morrison stages two passes' columns
    scr = std::max(scr, L.tab ? 4 * n + 16 : inverse_scratch_bytes(n, s.U[sp], G, true));
  }
  // What the moves keep (tables of the current positions, proposals) shares its place with a
  // refactorisation's ln|det|, signs and orbital matrix, consumed by the term ratios before the tables
  // are formed.  Then come the basis values and partial sums of either, over them the buffers of a
  // move, and over all of these the scratch of the inverses (past the orbital matrix).
  const int over0 = off;
  auto place = [&](int grp, int ke, bool all, bool tri, bool rows) {  // end of the walker's region
    off = over0;
    L.ke = ke;
    L.grp = grp;
    const int np = all ? N : grp;
    L.all = all ? 1 : 0;
    L.rows = rows ? 1 : 0;
    L.tri = tri ? 1 : 0;
    L.rtab = take(8 * 3 * np);
    L.rtds = take(tb == 4 ? 8 * 3 * np : 16);
    L.svn = take(tb * np * s.Nn);
    L.den = take(tb * np * s.Nn);
    L.vrows = take(tb * (rows ? N : (all ? nmax : grp)) * L.nocc_max);
    L.Sv = take(tb * (N + 1) * s.Nn);
    L.ut = take(tri ? tb * (N * (N - 1) / 2 + 1) : 0);
    L.ft = take(tri ? tb * (N * (N - 1) / 2 + 1) : 0);
    const int moves_end = off;
    off = over0;
    if (L.tab) {  // the X values of one spin; the reference's values are formed where its inverse goes
      L.ldet = L.dsg = off;
      L.PhiO = take(8 * std::max(std::max(s.n[0] * s.n_x[0], s.n[1] * s.n_x[1]), 1));
    } else {
      L.ldet = take(8 * Ut);
      L.dsg = take(8 * Ut);
      L.PhiO = take(8 * N * L.nocc_max);
    }
    L.scratch = off;
    const int scr_end = align16(off + std::max(scr, 16));
    const int shared0 = off = std::max(off, moves_end);
    L.bas = take(std::max(8 * s.M, tb * L.ke * s.M));
    L.alias = nch <= 32 ? 1 : 0;
    const int part_bytes = std::max(8 * nch, tb * L.ke * nch);
    L.part = L.alias ? L.bas : take(part_bytes);
    if (L.alias) off = std::max(off, align16(L.bas + part_bytes));
    const int basis_end = off;
    off = shared0;
    L.up = take(2 * tb * 4 * (N + 1));
    L.ue = take(tb * N);
    L.fe = take(tb * N);
    L.rho = take(8 * std::max(s.U[0], s.U[1]));
    L.rinv = take(8 * (std::max(s.U[0], s.U[1]) + 1));
    L.cvec = take(std::max(cv, 8));
    return off = std::max(std::max(off, basis_end), scr_end);
  };
  // the pair tables, and both spins prepared at once (one electron per lane), where as many
  // walkers share a block with them
  auto fit = [&](int bytes) { return std::min(16, max_smem / std::max(bytes, 1)); };
  // electrons prepared at once: 16 of a spin (a second group of a large spin costs little and its
  // place is saved), fewer where nothing fits otherwise
  int grp = std::min(16, nmax);
  while (grp > 1 && place(grp, 1, false, false, false) > max_smem) grp = grp > 4 ? 4 : 1;
  const int most = fit(place(grp, 1, false, false, false));
  int ke = 1;  // electrons a round of proposal rows takes: their displacements lie in one warp's lanes
  for (int k = 4; k > 1 && ke == 1; k >>= 1)
    if (tb == 4 && k * s.Nn <= 32 && fit(place(grp, k, false, false, false)) == most) ke = k;
  const bool tri = fit(place(grp, ke, false, true, false)) == most;
  const bool all = N <= 32 && fit(place(grp, ke, true, tri, false)) == most;
  const bool rows = all && s.same_occ && fit(place(grp, ke, true, tri, true)) == most;
  place(grp, ke, all, tri, rows);
  L.warp_bytes = off;
  int wpb = max_smem / off;
  if (wpb > 16) wpb = 16;
  if (wpb < 1) return VBQMC_ERR_CAPACITY;
  L.wpb = wpb;
  return VBQMC_OK;
}

int walkers_per_block(int W, int most, int sm_warps, int bytes) {
  int dev = 0, sms = 0, sm_smem = 0;
  if (W < 1 || cudaGetDevice(&dev) != cudaSuccess ||
      cudaDeviceGetAttribute(&sms, cudaDevAttrMultiProcessorCount, dev) != cudaSuccess ||
      cudaDeviceGetAttribute(&sm_smem, cudaDevAttrMaxSharedMemoryPerMultiprocessor, dev) != cudaSuccess || sms < 1)
    return most;
  auto resident = [&](int p) { return std::max(1, std::min(sm_warps / p, sm_smem / (p * bytes + 1024))); };
  int warps = 0;  // the most walkers on an SM
  for (int p = 1; p <= most; ++p) warps = std::max(warps, p * resident(p));
  if ((long)W > 2L * warps * sms)
    for (int p = std::min(2, most); p <= most; ++p)
      if (p * resident(p) == warps) {
        if (resident(p) > 1 || p == 1) return p;
        break;  // one block fills the SM: whole rounds
      }
  long best_cost = 0;
  int best = most;
  for (int p = most; p >= 1; --p) {
    const long res = resident(p);
    const long blocks = ((long)W + p - 1) / p, full = blocks / (res * sms), rest = blocks - full * res * sms;
    const long cost = full * (100 + 3 * p * res) + (rest ? 100 + 3 * p * ((rest + sms - 1) / sms) : 0);
    if (full && res > 4) break;
    if (p == most || 100 * cost < 98 * best_cost) {
      best_cost = cost;
      best = p;
    }
  }
  return best;
}

cudaError_t open_shared_memory(const void* fn, int static_bytes) {
  int dev = 0, most = 0;
  cudaError_t e = cudaGetDevice(&dev);
  if (e == cudaSuccess) e = cudaDeviceGetAttribute(&most, cudaDevAttrMaxSharedMemoryPerBlockOptin, dev);
  return e == cudaSuccess
             ? cudaFuncSetAttribute(fn, cudaFuncAttributeMaxDynamicSharedMemorySize, most - static_bytes)
             : e;
}

int per_determinant_region_bytes(const SysDev& s) {
  int off = 0;
  auto take = [&](int bytes) { off = align16(off + bytes); };
  const int N = s.N, Ut = s.U[0] + s.U[1], nocc = std::max(std::max(s.nocc[0], s.nocc[1]), 1);
  for (int b : {8 * 3 * N, 8 * 3 * N, 8 * s.U[0] * s.n[0] * s.n[0], 8 * s.U[1] * s.n[1] * s.n[1], 8 * s.nterm}) take(b);
  const int over0 = off;
  for (int b : {8 * 4 * N, 8 * 3 * N, 4 * (2 * N + 7 * s.Nn + 10 * (N + 1))}) take(b);
  const int moves_end = off;
  off = over0;
  for (int b : {8 * Ut, 8 * Ut, 8 * N * nocc}) take(b);
  off = std::max(off, moves_end);
  int cv = 0, scr = 0;
  for (int sp = 0; sp < 2; ++sp) {
    const int n = s.n[sp], ng = 32 / group_size(n);
    cv = std::max(cv, 16 * ng * n);
    scr = std::max(scr, ng * (8 * n * n + 4 * n) + 16);
  }
  const int shared0 = off;
  for (int b : {8 * s.M, 8 * nocc, 8 * std::max(std::max(s.n_occ_chunk[0], s.n_occ_chunk[1]), 1),
                8 * std::max(s.U[0], s.U[1]), 8 * (std::max(s.U[0], s.U[1]) + 1), std::max(cv, 8)})
    take(b);
  off = std::max(off, align16(shared0 + std::max(scr, 16)));
  take(4 * (N * s.Nn + (N + 1) * s.Nn));
  return off;
}

template <class Tb>
static cudaError_t launch_sweep_t(const SysDev& s, const SweepLayout& L, int W, double* R, int nsweeps, int refresh,
                                  double* state, int state_valid, double step, uint64_t seed, uint32_t step0, uint32_t tag,
                                  uint32_t woff, int* nacc, cudaStream_t st) {
  SweepLayout Lw = L;
  Lw.wpb = walkers_per_block(W, L.wpb, 16, L.warp_bytes);
  const int smem = Lw.wpb * Lw.warp_bytes;
  const void* fn = Lw.tab ? (const void*)sweep_kernel<Tb, true> : (const void*)sweep_kernel<Tb, false>;
  cudaError_t e = open_shared_memory(fn);
  if (e != cudaSuccess) return e;
  const int blocks = (W + Lw.wpb - 1) / Lw.wpb;
  if (Lw.tab)
    sweep_kernel<Tb, true><<<blocks, 32 * Lw.wpb, smem, st>>>(s, Lw, W, R, nsweeps, refresh, nullptr, 0, step, seed,
                                                              step0, tag, woff, nacc);
  else
    sweep_kernel<Tb, false><<<blocks, 32 * Lw.wpb, smem, st>>>(s, Lw, W, R, nsweeps, refresh, state, state_valid, step,
                                                               seed, step0, tag, woff, nacc);
  return cudaGetLastError();
}

template <class Tb>
cudaError_t launch_sweep_batch(const BatchSys* sys, const BatchItem* items, int nitems, const BatchCall* call,
                               int grid, int warps, int smem, cudaStream_t st) {
  sweep_batch_kernel<Tb><<<grid, 32 * warps, smem, st>>>(sys, items, nitems, call);
  return cudaGetLastError();
}
int batch_grid(const void* fn, int nitems, int warps, int smem, int persist) {
  cudaFuncAttributes own;
  if (cudaFuncGetAttributes(&own, fn) != cudaSuccess) return -1;
  if (open_shared_memory(fn, (int)own.sharedSizeBytes) != cudaSuccess) return -1;
  if (persist <= 0) return nitems;
  int bps = 0, dev = 0, sms = 0;
  if (cudaOccupancyMaxActiveBlocksPerMultiprocessor(&bps, fn, 32 * warps, smem) != cudaSuccess) return -1;
  if (cudaGetDevice(&dev) != cudaSuccess || cudaDeviceGetAttribute(&sms, cudaDevAttrMultiProcessorCount, dev) != cudaSuccess)
    return -1;
  const long long g = (long long)persist * std::max(bps, 1) * sms;
  return (int)std::max<long long>(1, std::min<long long>(g, nitems));
}
int sweep_batch_grid(int is_float, int nitems, int warps, int smem, int persist) {
  return batch_grid(is_float ? (const void*)sweep_batch_kernel<float> : (const void*)sweep_batch_kernel<double>, nitems,
                    warps, smem, persist);
}

template cudaError_t launch_sweep_batch<float>(const BatchSys*, const BatchItem*, int, const BatchCall*, int, int, int,
                                               cudaStream_t);
template cudaError_t launch_sweep_batch<double>(const BatchSys*, const BatchItem*, int, const BatchCall*, int, int, int,
                                                cudaStream_t);

cudaError_t launch_sweep(int precision, const SysDev& s, const SweepLayout& L, int W, double* R, int nsweeps,
                         int refresh, double* state, int state_valid, double step, uint64_t seed, uint32_t step0, uint32_t tag,
                         uint32_t woff, int* nacc, cudaStream_t st) {
  if (precision == VBQMC_MIXED)
    return launch_sweep_t<float>(s, L, W, R, nsweeps, refresh, state, state_valid, step, seed, step0, tag, woff, nacc,
                                 st);
  return launch_sweep_t<double>(s, L, W, R, nsweeps, refresh, state, state_valid, step, seed, step0, tag, woff, nacc,
                                st);
}

}  // namespace vbq
