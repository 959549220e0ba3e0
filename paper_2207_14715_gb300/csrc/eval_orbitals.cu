// Orbitals at every electron (arXiv:2207.14715, Sec. 2.1: phi_p = sum_mu lambda_{p mu} chi_mu):
// basis functions with gradients and Laplacians, then the contraction in balanced chunks of
// the nonzero coefficients, four orbitals of equal coefficient range at a time.  One block per eight
// (walker, electron) points; results go to the evaluation workspace:
//   OB [W][N][5][n_ev] bulk type: phi, d/dx, d/dy, d/dz, lap phi of the evaluated orbitals
//   OD [W][N][n_det_ev] double: values of the orbitals that enter determinants; in the mixed
//      form these come from float-float basis values and coefficients, and OB holds them
//      rounded to float.

#include "orbital_body.cuh"

namespace vbq {

namespace {
template <class Tb>
__global__ void __launch_bounds__(32 * kOrbWarps, 4) orbital_kernel(const SysDev s, const OrbLayout L, int W,
                                                                     const double* __restrict__ Rg,
                                                                     Tb* __restrict__ OB, double* __restrict__ OD) {
  extern __shared__ __align__(16) unsigned char smem[];
  const long long gw0 = (long long)blockIdx.x * L.wpb;
  orbital_block<Tb>(s, L, gw0, (int)min((long long)L.wpb, (long long)W * s.N - gw0), smem, Rg, OB, OD);
}

template <class Tb>
__global__ void __launch_bounds__(32 * kOrbWarps, 4)
    orbital_batch_kernel(const BatchSys* __restrict__ sys, const BatchItem* __restrict__ items, int nitems) {
  extern __shared__ __align__(16) unsigned char smem[];
  for (int it = blockIdx.x; it < nitems; it += gridDim.x) {
    // the points' shared-memory regions depend on the item's system: start together
    __syncthreads();
    const BatchItem item = items[it];
    const BatchSys& b = sys[item.sys];
    orbital_block<Tb>(b.dev, b.lay.orb, item.first, item.count, smem, b.R, static_cast<Tb*>(b.OB), b.OD);
  }
}

}  // namespace

int make_orb_layout(const SysDev& s, int tb, int max_smem, OrbLayout& L) {
  int off = 0;
  auto take = [&](int bytes) {
    const int o = off;
    off = align16(off + bytes);
    return o;
  };
  const int M = s.M;
  L.bas = take(5 * M * tb);
  L.bds = take(tb == 4 ? 8 * M : 16);
  L.ctab = take(tb == 4 ? 8 * 4 * s.Nn : 16);
  L.part = take(5 * s.evq_width * tb * std::max(s.n_evq_chunk, 1));
  L.partd = take(tb == 4 ? 8 * std::max(s.n_det_chunk, 1) : 16);
  L.table_bytes = off;
  if (kOrbWarps * off > max_smem) return VBQMC_ERR_CAPACITY;  // the limit on the size of a system
  L.r3 = take(8 * 3);
  L.dis = take(tb * 3 * s.Nn);
  // consecutive points 16 bytes apart in the banks: lanes on different points store side by side
  while (off % 128 != 16) off += 16;
  L.warp_bytes = off;
  L.wpb = std::min(kOrbWarps, max_smem / off);
  return VBQMC_OK;
}

template <class Tb>
cudaError_t launch_orbitals(const SysDev& s, const OrbLayout& L, int W, const double* R, Tb* OB, double* OD,
                            cudaStream_t st) {
  const int smem = L.wpb * L.warp_bytes;
  cudaError_t e = open_shared_memory((const void*)orbital_kernel<Tb>);
  if (e != cudaSuccess) return e;
  const long long points = (long long)W * s.N;
  orbital_kernel<Tb><<<(unsigned)((points + L.wpb - 1) / L.wpb), 32 * kOrbWarps, smem, st>>>(s, L, W, R, OB, OD);
  return cudaGetLastError();
}

template <class Tb>
cudaError_t launch_orbitals_batch(const BatchSys* sys, const BatchItem* items, int nitems, int grid, int warps,
                                  int smem, cudaStream_t st) {
  orbital_batch_kernel<Tb><<<grid, 32 * warps, smem, st>>>(sys, items, nitems);
  return cudaGetLastError();
}
int orbital_batch_grid(int is_float, int nitems, int warps, int smem, int persist) {
  return batch_grid(is_float ? (const void*)orbital_batch_kernel<float> : (const void*)orbital_batch_kernel<double>,
                    nitems, warps, smem, persist);
}
template cudaError_t launch_orbitals_batch<float>(const BatchSys*, const BatchItem*, int, int, int, int, cudaStream_t);
template cudaError_t launch_orbitals_batch<double>(const BatchSys*, const BatchItem*, int, int, int, int, cudaStream_t);

template cudaError_t launch_orbitals<float>(const SysDev&, const OrbLayout&, int, const double*, float*, double*,
                                            cudaStream_t);
template cudaError_t launch_orbitals<double>(const SysDev&, const OrbLayout&, int, const double*, double*, double*,
                                             cudaStream_t);

}  // namespace vbq
