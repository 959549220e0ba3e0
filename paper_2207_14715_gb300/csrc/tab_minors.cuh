// Replacement determinants of the reference tables (arXiv:2207.14715, Sec. 2.1 determinant
// expansion): every determinant of a spin is the reference with the slots S_u replaced by the
// orbitals Q_u (k_u <= 4), D_u / D_0 = sgn_u det T[S_u, Q_u], and the minors share their own
// minors.  Laplace expansion along the first row writes a k x k minor through k minors of size
// k - 1 on the remaining rows, and its derivatives are its k^2 cofactors: both mostly other
// determinants' minors; set-up adds the few that are not (TabMinors, vbqmc_internal.h).  The values
// of one size are formed by all lanes together from those of the size below.
//
// Accuracy: where the reference is small next to the other determinants, T is a large matrix of
// rank one plus a remainder (the reference's own column), and minors cancel: the 2 x 2 minors are
// formed as Kahan's difference of products and the 3 x 3 minors with the error terms of their
// products and sums, so that the expansion loses no more than an elimination with pivoting
// (which removes the rank-one part in its first step); the cofactors of the derivatives are minors
// of this kind as well.
//
// Work: 4, 23 and 4 instructions on the FP64 pipe per 32 minors of size 2, 3 and 4 (64 cycles of a
// sub-partition each), where eliminating every determinant's own matrix took about 60 per 32
// determinants with four divisions in a chain (150 with the inverses for the derivatives).
//
// Arrays of one spin: Tn [ns][nx] the rows of T that take part, v [nv] the minors without the
// determinants' signs (slot u < U: determinant u; then the added ones).
#pragma once

#include "wf_device.cuh"

namespace vbq {

// a b - c d to a few units in the last place of the result
__device__ __forceinline__ double diff_of_products(double a, double b, double c, double d) {
  const double w = c * d;
  const double e = fma(-c, d, w);
  return fma(a, b, -w) + e;
}
// a x - b y + c z with the rounding errors of the products and of the first sums added back
__device__ __forceinline__ double dot3(double a, double x, double b, double y, double c, double z) {
  const double p = a * x, q = -(b * y), r = c * z;
  double e = fma(a, x, -p) + (fma(-b, y, -q) + fma(c, z, -r));
  const double s = p + q, sb = s - p;
  e += (p - (s - sb)) + (q - sb);
  const double t = s + r, tb = t - s;
  e += (s - (t - tb)) + (r - tb);
  return t + e;
}

// det Tn[rows][cols] of the minor e (an entry of the list ld) without its row i and column j (i < 0:
// the whole minor), by Laplace expansion; the sign (-1)^(i + j) is not included.
static __device__ __noinline__ double tab_submatrix(const double* Tn, int nx, const int* __restrict__ e, int i, int j) {
  int r[4], c[4], k = 0;
  for (int q = 0, kk = __ldg(e + 1); q < kk; ++q)
    if (q != i) r[k++] = __ldg(e + 2 + q) * nx;
  k = 0;
  for (int q = 0, kk = __ldg(e + 1); q < kk; ++q)
    if (q != j) c[k++] = __ldg(e + 6 + q);
  auto t = [&](int a, int b) { return Tn[r[a] + c[b]]; };
  auto d2 = [&](int a, int x, int y) {  // rows a, a + 1
    return diff_of_products(t(a, x), t(a + 1, y), t(a, y), t(a + 1, x));
  };
  auto d3 = [&](int a, int x, int y, int z) {
    return dot3(t(a, x), d2(a + 1, y, z), t(a, y), d2(a + 1, x, z), t(a, z), d2(a + 1, x, y));
  };
  if (k == 2) return d2(0, 0, 1);
  if (k == 3) return d3(0, 0, 1, 2);
  return t(0, 0) * d3(1, 1, 2, 3) - t(0, 1) * d3(1, 0, 2, 3) + t(0, 2) * d3(1, 0, 1, 3) - t(0, 3) * d3(1, 0, 1, 2);
}

// v from Tn, all levels.
__device__ __forceinline__ void tab_values(const TabMinors& m, int lane, const double* Tn, double* v) {
  if (lane == 0) v[0] = 1.0;
  for (int i = lane; i < m.n1; i += 32) {
    const int2 e = __ldg(reinterpret_cast<const int2*>(m.l1) + i);
    v[e.x] = Tn[e.y];
  }
  for (int i = lane; i < m.n2; i += 32) {
    const int4 e = __ldg(reinterpret_cast<const int4*>(m.l2) + i);
    v[e.x] = diff_of_products(Tn[e.y & 0xffff], Tn[e.y >> 16], Tn[e.z & 0xffff], Tn[e.z >> 16]);
  }
  __syncwarp();
  for (int i = lane; i < m.n3; i += 32) {
    const int4 e = __ldg(reinterpret_cast<const int4*>(m.l3) + i);
    v[e.x] = dot3(Tn[e.y & 0xffff], v[e.y >> 16], Tn[e.z & 0xffff], v[e.z >> 16], Tn[e.w & 0xffff], v[e.w >> 16]);
  }
  __syncwarp();
  for (int i = lane; i < m.n4; i += 32) {
    const int4 e = __ldg(reinterpret_cast<const int4*>(m.l4) + 2 * i);
    const int last = __ldg(m.l4 + 8 * i + 4);
    double d = Tn[e.y & 0xffff] * v[e.y >> 16];
    d = fma(-Tn[e.z & 0xffff], v[e.z >> 16], d);
    d = fma(Tn[e.w & 0xffff], v[e.w >> 16], d);
    v[e.x] = fma(-Tn[last & 0xffff], v[last >> 16], d);
  }
  for (int i = lane; i < m.nd; i += 32) v[__ldg(m.ld + 10 * i)] = tab_submatrix(Tn, m.nx, m.ld + 10 * i, -1, -1);
  __syncwarp();
}

// the cofactor an entry of rt or du names: 1, an entry of Tn or a minor
__device__ __forceinline__ double tab_cofactor(int code, const double* Tn, const double* v) {
  return code < 0 ? 1.0 : (code >= 0x10000 ? Tn[code - 0x10000] : v[code]);
}

// gT [ns nx] = sum_u adj[u] d q_u / d Tn over the determinants.
__device__ __forceinline__ void tab_adjoint(const TabMinors& m, int lane, const double* Tn, const double* v,
                                            const double* adj, double* gT) {
  for (int i = lane; i < m.ns * m.nx; i += 32) {
    double x = 0.0;
    for (int t = __ldg(m.rt_off + i); t < __ldg(m.rt_off + i + 1); ++t) {
      const int2 e = __ldg(reinterpret_cast<const int2*>(m.rt) + t);  // determinant (sign in bit 31), cofactor
      const double a = adj[e.x & 0x7fffffff], f = tab_cofactor(e.y, Tn, v);
      x = e.x < 0 ? fma(-a, f, x) : fma(a, f, x);
    }
    for (int q = 0; q < m.nd; ++q) {  // the determinants expanded by themselves that hold this entry
      const int* e = m.ld + 10 * q;
      int a = -1, b = -1;
      for (int j = 0, k = __ldg(e + 1); j < k; ++j) {
        if (__ldg(e + 2 + j) * m.nx == i - i % m.nx) a = j;
        if (__ldg(e + 6 + j) == i % m.nx) b = j;
      }
      if (a < 0 || b < 0) continue;
      const double c = adj[__ldg(e)] * tab_submatrix(Tn, m.nx, e, a, b);
      x += ((a + b) & 1) ? -c : c;
    }
    gT[i] = x;
  }
  __syncwarp();
}

// dv[u] = the derivative of q_u along dTn, for the U determinants.
__device__ __forceinline__ void tab_derivatives(const TabMinors& m, int U, int lane, const double* Tn, const double* v,
                                                const double* dTn, double* dv) {
  for (int u = lane; u < U; u += 32) {
    double x = 0.0;
    for (int t = __ldg(m.du_off + u); t < __ldg(m.du_off + u + 1); ++t) {
      const int2 e = __ldg(reinterpret_cast<const int2*>(m.du) + t);  // Tn index (sign in bit 31), cofactor
      const double d = dTn[e.x & 0x7fffffff], f = tab_cofactor(e.y, Tn, v);
      x = e.x < 0 ? fma(-d, f, x) : fma(d, f, x);
    }
    dv[u] = x;
  }
  __syncwarp();
  for (int i = lane; i < m.nd; i += 32) {
    const int* e = m.ld + 10 * i;
    double x = 0.0;
    for (int a = 0, k = __ldg(e + 1); a < k; ++a)
      for (int b = 0; b < k; ++b) {
        const double c = dTn[__ldg(e + 2 + a) * m.nx + __ldg(e + 6 + b)] * tab_submatrix(Tn, m.nx, e, a, b);
        x += ((a + b) & 1) ? -c : c;
      }
    dv[__ldg(e)] = x;
  }
  __syncwarp();
}

}  // namespace vbq
