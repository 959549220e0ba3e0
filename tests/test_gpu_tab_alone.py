"""Determinants of the reference tables that are formed each by itself (few replaced slots over many
orbitals, where shared minors would outnumber the determinants): values and cofactors directly, and sweeps
and evaluations of systems that take them, in both forms and with the tables carried over the moves.

Bounds of the direct test, eps = 2^-53: elimination with partial pivoting gives the determinant of M + E
with |E| <= 256 eps max|M| (k <= 4 terms of |L| |U|, growth at most 8, 8 roundings each with the reciprocal's),
that is an error of at most 256 eps max|M| sum |cofactor|; a cofactor's 2 x 2 minors are within 4 eps, its
compensated sum within 4 eps of the result more, together 8 eps sum |entry| |minor|; a value by expansion adds
the first row's products.  Inputs: random matrices, alone and with a rank-one part 10^3, 10^6 and 10^9 times as
large (a small reference).

Systems: FP64 as the other table systems (ln|Psi|, E_L 1e-10, gradient 1e-9, derivatives 1e-8 of
max(1, |x|), trajectories 1e-12); mixed sweeps follow the FP64 form but where a decision falls within float
rounding of its threshold (512 x 2 x 10 moves: 97 % of the walkers, as for the other table systems).
The direct test stages the cofactors of 32 determinants at a time and, as systems do whose region leaves less
room, of 8, 2 and 1."""
import ctypes
import dataclasses
import itertools
import os
import subprocess
import tempfile
from fractions import Fraction

import numpy as np
import pytest

from paper_2207_14715_gb300 import systems as S

pytestmark = pytest.mark.gpu
torch = pytest.importorskip("torch")

CSRC = os.path.join(os.path.dirname(os.path.dirname(os.path.abspath(__file__))), "paper_2207_14715_gb300", "csrc")

PROBE = r"""
#include "tab_minors.cuh"
// determinant d of the list ld [nd][4]: val [nd] by elimination, vex [nd] by expansion, and through the staged gather (adj = the unit vector of
// d's slot) its cofactors in g [nd][ns nx]; dv: the derivative along dT
__global__ void probe(int nd, int ns, int nx, int sd, const int* ld, const int* lr, const int* lh, const int* le,
                      const double* T, const double* dT, double* adj, double* val, double* vex, double* g, double* dv) {
  __shared__ double Tn[1024], stage[512], gT[1024];
  const int lane = threadIdx.x;
  for (int i = lane; i < ns * nx; i += 32) Tn[i] = T[i];
  __syncwarp();
  for (int d = lane; d < nd; d += 32) {
    val[d] = vbq::tab_value<true>(Tn, nx, reinterpret_cast<const int4*>(ld)[d]);
    vex[d] = vbq::tab_value<false>(Tn, nx, reinterpret_cast<const int4*>(ld)[d]);
  }
  for (int d = 0; d < nd; ++d) {
    for (int i = lane; i < nd; i += 32) adj[i] = i == d ? 1.0 : 0.0;
    for (int i = lane; i < ns * nx; i += 32) gT[i] = 0.0;
    __syncwarp();
    vbq::tab_adjoint_alone(nd, nx, ld, lr, lh, le, lane, Tn, adj, gT, stage, sd);
    for (int i = lane; i < ns * nx; i += 32) g[(size_t)d * ns * nx + i] = gT[i];
    __syncwarp();
  }
  vbq::tab_derivatives_alone(nd, nx, ld, lane, Tn, dT, dv);
}
extern "C" int run(int nd, int ns, int nx, int sd, const int* ld, const int* lr, int nlr, const int* lh, int nlh,
                   const int* le, int nle, const double* T, const double* dT, double* val, double* vex, double* g, double* dv) {
  const size_t t = 8 * (size_t)ns * nx, n = 8 * (size_t)nd, size[11] = {2 * n, 4 * (size_t)nlr, 4 * (size_t)nlh,
                                                                         4 * (size_t)nle, t, t, n, n, n, n * ns * nx, n};
  const void* in[6] = {ld, lr, lh, le, T, dT};
  void* p[11] = {};
  cudaError_t e = cudaSuccess;
  for (int i = 0; i < 11 && e == cudaSuccess; ++i) {
    e = cudaMalloc(&p[i], size[i]);
    if (e == cudaSuccess && i < 6) e = cudaMemcpy(p[i], in[i], size[i], cudaMemcpyHostToDevice);
  }
  if (e == cudaSuccess) {
    probe<<<1, 32>>>(nd, ns, nx, sd, (int*)p[0], (int*)p[1], (int*)p[2], (int*)p[3], (double*)p[4], (double*)p[5],
                     (double*)p[6], (double*)p[7], (double*)p[8], (double*)p[9], (double*)p[10]);
    e = cudaGetLastError();
  }
  if (e == cudaSuccess) e = cudaMemcpy(val, p[7], size[7], cudaMemcpyDeviceToHost);
  if (e == cudaSuccess) e = cudaMemcpy(vex, p[8], size[8], cudaMemcpyDeviceToHost);
  if (e == cudaSuccess) e = cudaMemcpy(g, p[9], size[9], cudaMemcpyDeviceToHost);
  if (e == cudaSuccess) e = cudaMemcpy(dv, p[10], size[10], cudaMemcpyDeviceToHost);
  for (void* q : p) cudaFree(q);
  return (int)e;
}
"""


@pytest.fixture(scope="module")
def probe():
    if not torch.cuda.is_available():
        pytest.skip("no CUDA device")
    d = tempfile.mkdtemp(prefix="tab_probe_")
    src, so = os.path.join(d, "probe.cu"), os.path.join(d, "probe.so")
    with open(src, "w") as f:
        f.write(PROBE)
    subprocess.run([os.environ.get("NVCC", "nvcc"), "-gencode", "arch=compute_103a,code=sm_103a", "-O3",
                    "-std=c++17", "-shared", "-Xcompiler", "-fPIC", "-I", CSRC, src, "-o", so], check=True)
    return ctypes.CDLL(so)


def lists(dets, nx):
    """The kernel's lists for determinants (rows, columns), slot = position (vbqmc_internal.h)."""
    ld, lr, lh, le = [], [0], [], []
    for d0 in range(0, len(dets), 32):
        entry = []
        for q, (rows, cols) in enumerate(dets[d0:d0 + 32]):
            k = len(rows)
            c = list(cols) + [0] * (4 - k)
            ld += [d0 + q | k << 28, sum(r << 8 * i for i, r in enumerate(rows)), c[0] | c[1] << 16, c[2] | c[3] << 16]
            entry += [(rows[i] * nx + cols[j], q << 4 | 4 * i + j) for i in range(k) for j in range(k)]
        for t, group in itertools.groupby(sorted(entry), key=lambda e: e[0]):
            lh += [t, len(le)]
            le += [c for _, c in group]
        lr.append(len(lh) // 2)
    lh += [-1, len(le)]
    return [np.array(x, np.int64).astype(np.uint32).view(np.int32) for x in (ld, lr, lh, le)]


def exact_det(M):
    n = len(M)
    if n == 1:
        return M[0][0]
    return sum((-1) ** j * M[0][j] * exact_det([r[:j] + r[j + 1:] for r in M[1:]]) for j in range(n))


@pytest.mark.parametrize("scale", [0.0, 1e3, 1e6, 1e9])
@pytest.mark.parametrize("nd,sd", [(1, 32), (31, 32), (33, 32), (40, 32), (40, 8), (40, 2), (33, 1)])
def test_values_and_cofactors(probe, nd, sd, scale):
    rng = np.random.default_rng(nd + sd)
    ns, nx = 5, 13
    T = scale * np.outer(rng.normal(size=ns), rng.normal(size=nx)) + rng.normal(size=(ns, nx))
    dT = rng.normal(size=(ns, nx))
    if nd > 2:
        T[:, 0] = 0.0  # singular minors
    dets = []
    for q in range(nd):  # k = 4 before k = 3, as the set-up orders them
        k = 4 if q < (2 * nd + 2) // 3 else 3
        dets.append((sorted(rng.choice(ns, k, replace=False).tolist()), sorted(rng.choice(nx, k, replace=False).tolist())))
    ld, lr, lh, le = lists(dets, nx)
    val, vex, g, dv = np.empty(nd), np.empty(nd), np.empty((nd, ns, nx)), np.empty(nd)
    p = lambda a: ctypes.c_void_p(a.ctypes.data)  # noqa: E731
    assert probe.run(nd, ns, nx, sd, p(ld), p(lr), len(lr), p(lh), len(lh), p(le), len(le), p(T), p(dT), p(val), p(vex),
                     p(g), p(dv)) == 0
    eps = 2.0 ** -53
    for q, (rows, cols) in enumerate(dets):
        k = len(rows)
        M = [[Fraction(T[r, c]) for c in cols] for r in rows]
        cof = np.empty((k, k))
        bound, along, tol = np.empty((k, k)), Fraction(0), 0.0
        for i in range(k):
            for j in range(k):
                sub = [r[:j] + r[j + 1:] for a, r in enumerate(M) if a != i]
                c = (-1) ** (i + j) * exact_det(sub)
                cof[i, j] = float(c)
                o = {0: 0, 1: 0, 2: k - 2, 3: k - 2}[i] if k == 4 else 0  # row of 'sub' the expansion runs along
                rest = sub[:o] + sub[o + 1:]
                if k == 4:
                    bound[i, j] = 8 * eps * sum(abs(float(sub[o][m])) * abs(float(exact_det([x[:m] + x[m + 1:] for x in rest])))
                                                for m in range(3)) + 8 * eps * abs(cof[i, j])
                else:
                    bound[i, j] = 8 * eps * abs(cof[i, j])
                d = Fraction(dT[rows[i], cols[j]])
                along += d * c
                tol += abs(float(d)) * (bound[i, j] + 16 * eps * abs(cof[i, j]))
        det = exact_det(M)
        top = max(abs(float(x)) for r in M for x in r)
        assert abs(val[q] - float(det)) <= 256 * eps * top * np.abs(cof).sum()
        row = np.abs(T[rows[0], cols])  # the first row's products, their sum within 4 roundings each
        assert abs(vex[q] - float(det)) <= (row * (bound[0] + 8 * eps * np.abs(cof[0]))).sum()
        got = np.zeros((ns, nx))
        got[np.ix_(rows, cols)] = cof
        lim = np.zeros((ns, nx))
        lim[np.ix_(rows, cols)] = bound
        assert (np.abs(g[q] - got) <= lim).all()
        assert abs(dv[q] - float(along)) <= tol


def system(n_pairs, n_active, n_structures, seed=5):
    """n_pairs singlet pairs drawn from n_active active orbitals per structure, one core, on the nuclei and
    basis of the open-shell test system."""
    base = S.small_open_shell(params=False)
    rng = np.random.default_rng(seed)
    orb = np.concatenate([base.orb_coef[:1], rng.normal(size=(n_active, base.M)) / np.sqrt(base.M)])
    strs, seen = [], set()
    while len(strs) < n_structures:
        q = [int(v) for v in 1 + rng.permutation(n_active)[:2 * n_pairs]]
        prs = tuple(sorted((min(q[2 * j:2 * j + 2]), max(q[2 * j:2 * j + 2])) for j in range(n_pairs)))
        if prs not in seen:
            seen.add(prs)
            strs.append(([0], list(prs), []))
    io, ina, po, prs, uo, un = S._structures(strs)
    n = 1 + n_pairs
    return dataclasses.replace(
        base, orb_coef=orb, orb_class=np.full(len(orb), -1, np.int32), orb_kind=np.ones(len(orb), np.int32), n_up=n,
        n_dn=n, c_vb=1.0 + 0.3 * rng.uniform(-1, 1, n_structures), inact_off=io, inact=ina, pair_off=po, pairs=prs,
        unp_off=uo, unp=un, cparam=np.arange(1, n_structures, dtype=np.int32), jas_param=True, step=0.3)


@pytest.fixture(scope="module")
def vb():
    if not torch.cuda.is_available():
        pytest.skip("no CUDA device")
    from paper_2207_14715_gb300 import build, vbqmc
    build.build()
    return vbqmc


SYSTEMS = [(4, 20, 24), (3, 30, 30)]  # k = 4 and 3, and k = 3 alone


@pytest.mark.parametrize("size", SYSTEMS)
@pytest.mark.parametrize("refresh", [0, 1])
def test_fp64_matches_oracle(vb, orc, size, refresh):
    spec, W = system(*size), 24
    ctx = vb.create(0)
    ctx.set_system(0, spec)
    assert ctx.launch_info(0, vb.FP64)["tables"]
    R0 = S.initial_walkers(spec, W, 3)
    R = torch.tensor(R0, device="cuda")
    z = lambda *s: torch.zeros(s, dtype=torch.float64, device="cuda")  # noqa: E731
    lp, sg, el, g, O, dE = z(W), z(W), z(W), torch.zeros_like(R), z(W, spec.n_params), z(W, spec.n_params)
    ctx.eval_walkers(0, vb.FP64, R, lp, sg, el, g, O, dE)
    ref = orc.evaluate(spec, R0, derivs=True, grad=True)
    rel = lambda a, b: (np.abs(a.cpu().numpy() - b) / np.maximum(1.0, np.abs(b))).max()  # noqa: E731
    assert (sg.cpu().numpy() == ref["sign"]).all()
    assert rel(lp, ref["logpsi"]) < 1e-10 and rel(el, ref["eloc"]) < 1e-10 and rel(g, ref["grad"]) < 1e-9
    assert rel(O, ref["O"]) < 1e-8 and rel(dE, ref["dEL"]) < 1e-8
    ctx.vmc_steps(0, vb.FP64, R, 3, spec.step, 11, step0=2, refresh=refresh)
    Ro = orc.vmc(spec, R0, 3, spec.step, seed=11, step0=2, eloc=False)[0]
    assert np.abs(R.cpu().numpy() - Ro).max() < 1e-12
    ctx.close()


@pytest.mark.parametrize("size", SYSTEMS)
@pytest.mark.parametrize("refresh", [0, 1])
def test_mixed_follows_fp64(vb, size, refresh):
    spec = system(*size)
    R0 = S.initial_walkers(spec, 512, 12)
    ctx = vb.create(0)
    ctx.set_system(0, spec)
    out = []
    for prec in (vb.FP64, vb.MIXED):
        R = torch.tensor(R0, device="cuda")
        ctx.vmc_steps(0, prec, R, 2, spec.step, 77, step0=3, refresh=refresh)
        out.append(R.cpu().numpy())
    same = np.all(np.abs(out[0] - out[1]) < 1e-9, axis=(1, 2))
    assert same.mean() > 0.97, same.mean()
    ctx.close()


def test_batched_step_matches_single(vb):
    """One FP64 step of a batch that holds such a system against the single-system calls: the same moves
    (1e-12) and E_L to 1e-8 of max(1, |E_L|) (separately compiled kernels)."""
    spec, W = system(*SYSTEMS[0]), 70
    ctx = vb.create(0)
    ctx.set_system(0, spec)
    ctx.set_system(1, S.h2_vb())
    R0 = S.initial_walkers(spec, W, 4)
    z = lambda *s: torch.zeros(s, dtype=torch.float64, device="cuda")  # noqa: E731
    R, R1 = torch.tensor(R0, device="cuda"), torch.tensor(R0, device="cuda")
    Rh = torch.tensor(S.initial_walkers(S.h2_vb(), 64, 4), device="cuda")
    lp, sg, el, l1, s1, e1, lh, sh, eh = z(W), z(W), z(W), z(W), z(W), z(W), z(64), z(64), z(64)
    batch = vb.Batch(ctx, [0, 1], [W, 64], vb.FP64)
    batch.vmc_steps([R, Rh], 1, 0.3, 9, step0=1, refresh=0, logpsi=[lp, lh], sign=[sg, sh], eloc=[el, eh])
    torch.cuda.synchronize()
    batch.close()
    ctx.vmc_steps(0, vb.FP64, R1, 1, 0.3, 9, step0=1, refresh=0, logpsi=l1, sign=s1, eloc=e1)
    torch.cuda.synchronize()
    assert (R - R1).abs().max() < 1e-12 and torch.equal(sg, s1)
    assert ((el - e1).abs() / e1.abs().clamp(min=1.0)).max() < 1e-8
    ctx.close()
