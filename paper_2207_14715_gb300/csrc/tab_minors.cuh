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
// products and sums, so that a 4 x 4 minor's last sum is the only one that cancels (three times the error of an
// elimination with pivoting, which removes the rank-one part in its first step; ln|Phi|, its gradient and
// E_L are as accurate); the cofactors of the derivatives are minors of this kind as well.
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

// Determinants formed each by itself (list ld, up to 32 at a time, one per lane), k x k block of Tn in
// registers.  Values of a move by elimination with partial pivoting: about 40 FP64 instructions per 32
// determinants (k = 4), and where the reference is small an error a third of the expansion's, whose last
// sum cancels.  Values of an evaluation by the expansion along the first row (120), in the arithmetic of
// the cofactors that its derivatives take.
// Cofactors as expansions over the 2 x 2 minors of the rows (0, 1) and (2, 3), which the 16 share: about
// 420 per 32 determinants.  They are gathered by Tn entry from a round's cofactors in shared memory, in the
// order of the list.  Expanding with row and column lists in local memory, every entry of Tn searching the
// whole list, took 4.84 ms for two sweeps and 6.79 ms for an evaluation with derivatives (4096 walkers,
// 189 determinants of a spin over 18 orbitals, mixed), eliminations and inverses per determinant 3.21 and
// 3.34 ms, this form 1.79 and 2.05 ms.
template <int K>
__device__ __forceinline__ void tab_block(const double* Tn, int nx, int4 e, double (&t)[K][K]) {
#pragma unroll
  for (int a = 0; a < K; ++a) {
    const double* row = Tn + ((e.y >> (8 * a)) & 0xff) * nx;
#pragma unroll
    for (int b = 0; b < K; ++b) {
      const unsigned c = (unsigned)(b < 2 ? e.z : e.w);
      t[a][b] = row[(b & 1) ? c >> 16 : c & 0xffffu];
    }
  }
}
template <int K> __device__ __forceinline__ double tab_eliminate(double (&t)[K][K]) {
  double det = 1.0;
#pragma unroll
  for (int c = 0; c < K; ++c) {
#pragma unroll
    for (int r = c + 1; r < K; ++r) {  // the largest |t_rc| to the diagonal (bit order is value order)
      const bool up = (__double_as_longlong(t[r][c]) & 0x7fffffffffffffffll) >
                      (__double_as_longlong(t[c][c]) & 0x7fffffffffffffffll);
#pragma unroll
      for (int j = c; j < K; ++j) {
        const double x = up ? t[r][j] : t[c][j];
        t[r][j] = up ? t[c][j] : t[r][j];
        t[c][j] = x;
      }
      if (up) det = -det;
    }
    const double p = t[c][c];
    det *= p;
    if (c + 1 == K) break;
    const double ip = nonzero(p) ? recip_dd(p) : 0.0;
#pragma unroll
    for (int r = c + 1; r < K; ++r) {
      const double f = t[r][c] * ip;
#pragma unroll
      for (int j = c + 1; j < K; ++j) t[r][j] = fma(-f, t[c][j], t[r][j]);
    }
  }
  return det;
}
template <int K> __device__ __forceinline__ double tab_expand(const double (&t)[K][K]) {
  auto d2 = [&](int x, int y) { return diff_of_products(t[K - 2][x], t[K - 1][y], t[K - 2][y], t[K - 1][x]); };
  if constexpr (K == 3) return dot3(t[0][0], d2(1, 2), t[0][1], d2(0, 2), t[0][2], d2(0, 1));
  auto d3 = [&](int x, int y, int z) { return dot3(t[1][x], d2(y, z), t[1][y], d2(x, z), t[1][z], d2(x, y)); };
  double d = t[0][0] * d3(1, 2, 3);
  d = fma(-t[0][1], d3(0, 2, 3), d);
  d = fma(t[0][2], d3(0, 1, 3), d);
  return fma(-t[0][K - 1], d3(0, 1, 2), d);
}
template <bool PIVOT> static __device__ __noinline__ double tab_value(const double* Tn, int nx, int4 e) {
  if (((unsigned)e.x >> 28) == 4u) {
    double t[4][4];
    tab_block<4>(Tn, nx, e, t);
    return PIVOT ? tab_eliminate<4>(t) : tab_expand<4>(t);
  }
  double t[3][3];
  tab_block<3>(Tn, nx, e, t);
  return PIVOT ? tab_eliminate<3>(t) : tab_expand<3>(t);
}
// emit(a, b, signed cofactor of row a and column b) for the k x k entries
template <class Emit> __device__ __forceinline__ void tab_cofactors(const double* Tn, int nx, int4 e, Emit&& emit) {
  if (((unsigned)e.x >> 28) == 4u) {
    // a pair of rows at a time, over the minors of the other pair (a loop: all 16 at once would take the
    // registers of four warps per SM)
#pragma unroll 1
    for (int h = 0; h < 4; h += 2) {
      const double* row[2] = {Tn + ((e.y >> (8 * h)) & 0xff) * nx, Tn + ((e.y >> (8 * h + 8)) & 0xff) * nx};
      const double* other[2] = {Tn + ((e.y >> (16 - 8 * h)) & 0xff) * nx, Tn + ((e.y >> (24 - 8 * h)) & 0xff) * nx};
      const int col[4] = {e.z & 0xffff, (int)((unsigned)e.z >> 16), e.w & 0xffff, (int)((unsigned)e.w >> 16)};
      auto at = [](int x, int y) { return x == 0 ? y - 1 : (x == 1 ? y + 1 : 5); };  // x < y
      double m[6];
#pragma unroll
      for (int x = 0; x < 3; ++x)
#pragma unroll
        for (int y = x + 1; y < 4; ++y)
          m[at(x, y)] = diff_of_products(other[0][col[x]], other[1][col[y]], other[0][col[y]], other[1][col[x]]);
#pragma unroll
      for (int a = 0; a < 2; ++a)
#pragma unroll
        for (int b = 0; b < 4; ++b) {  // along the pair's other row
          const int x = b == 0 ? 1 : 0, y = b <= 1 ? 2 : 1, z = b <= 2 ? 3 : 2;
          const double* r = row[1 - a];
          const double c = dot3(r[col[x]], m[at(y, z)], r[col[y]], m[at(x, z)], r[col[z]], m[at(x, y)]);
          emit(h + a, b, ((a + b) & 1) ? -c : c);
        }
    }
    return;
  }
  double t[3][3];
  tab_block<3>(Tn, nx, e, t);
#pragma unroll
  for (int a = 0; a < 3; ++a)
#pragma unroll
    for (int b = 0; b < 3; ++b) {
      const int p = a == 0 ? 1 : 0, q = a <= 1 ? 2 : 1, x = b == 0 ? 1 : 0, y = b <= 1 ? 2 : 1;
      const double c = diff_of_products(t[p][x], t[q][y], t[p][y], t[q][x]);
      emit(a, b, ((a + b) & 1) ? -c : c);
    }
}
// gT += adj times the cofactors of the nd determinants of the list; stage [16][sd], sd <= 32 a power of two:
// determinants of a round.
static __device__ __noinline__ void tab_adjoint_alone(int nd, int nx, const int* ld, const int* lr_off, const int* lh,
                                                      const int* le, int lane, const double* Tn, const double* adj,
                                                      double* gT, double* stage, int sd) {
  for (int d0 = 0; d0 < nd; d0 += sd) {
    const int d = d0 + lane;
    if (lane < sd && d < nd) {
      const int4 e = __ldg(reinterpret_cast<const int4*>(ld) + d);
      const double a = adj[e.x & 0xfffffff];
      tab_cofactors(Tn, nx, e, [&](int i, int j, double f) { stage[(4 * i + j) * sd + lane] = a * f; });
    }
    __syncwarp();
    const int r = d0 >> 5, in = d0 & 31;
    for (int h = __ldg(lr_off + r) + lane; h < __ldg(lr_off + r + 1); h += 32) {
      const int2 e = __ldg(reinterpret_cast<const int2*>(lh) + h);
      double x = gT[e.x];
      for (int q = e.y, end = __ldg(lh + 2 * h + 3); q < end; ++q) {
        const int c = __ldg(le + q), k = (c >> 4) - in;
        if ((unsigned)k < (unsigned)sd) x += stage[(c & 15) * sd + k];
      }
      gT[e.x] = x;
    }
    __syncwarp();
  }
}
static __device__ __noinline__ void tab_derivatives_alone(int nd, int nx, const int* ld, int lane, const double* Tn,
                                                          const double* dTn, double* dv) {
  for (int d = lane; d < nd; d += 32) {
    const int4 e = __ldg(reinterpret_cast<const int4*>(ld) + d);
    double x = 0.0;
    tab_cofactors(Tn, nx, e, [&](int i, int j, double f) {
      const unsigned cols = (unsigned)(j < 2 ? e.z : e.w);
      x = fma(dTn[((e.y >> (8 * i)) & 0xff) * nx + (int)((j & 1) ? cols >> 16 : cols & 0xffffu)], f, x);
    });
    dv[e.x & 0xfffffff] = x;
  }
}

// v from Tn, all levels (ALONE = false: for systems without determinants formed by themselves; PIVOT: how
// these are formed).
template <bool ALONE, bool PIVOT>
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
  for (int i = lane; ALONE && i < m.nd; i += 32) {
    const int4 e = __ldg(reinterpret_cast<const int4*>(m.ld) + i);
    v[e.x & 0xfffffff] = tab_value<PIVOT>(Tn, m.nx, e);
  }
  __syncwarp();
}

// the cofactor an entry of rt or du names: 1, an entry of Tn or a minor
__device__ __forceinline__ double tab_cofactor(int code, const double* Tn, const double* v) {
  return code < 0 ? 1.0 : (code >= 0x10000 ? Tn[code - 0x10000] : v[code]);
}

// gT [ns nx] = sum_u adj[u] d q_u / d Tn over the determinants; stage [16][sd] as tab_adjoint_alone.
template <bool ALONE>
__device__ __forceinline__ void tab_adjoint(const TabMinors& m, int lane, const double* Tn, const double* v,
                                            const double* adj, double* gT, double* stage, int sd) {
  for (int i = lane; i < m.ns * m.nx; i += 32) {
    double x = 0.0;
    for (int t = __ldg(m.rt_off + i); t < __ldg(m.rt_off + i + 1); ++t) {
      const int2 e = __ldg(reinterpret_cast<const int2*>(m.rt) + t);  // determinant (sign in bit 31), cofactor
      const double a = adj[e.x & 0x7fffffff], f = tab_cofactor(e.y, Tn, v);
      x = e.x < 0 ? fma(-a, f, x) : fma(a, f, x);
    }
    gT[i] = x;
  }
  __syncwarp();
  if (ALONE && m.nd) tab_adjoint_alone(m.nd, m.nx, m.ld, m.lr_off, m.lh, m.le, lane, Tn, adj, gT, stage, sd);
}

// dv[u] = the derivative of q_u along dTn, for the U determinants.
template <bool ALONE>
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
  if (ALONE && m.nd) tab_derivatives_alone(m.nd, m.nx, m.ld, lane, Tn, dTn, dv);
  __syncwarp();
}

}  // namespace vbq
