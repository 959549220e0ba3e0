"""Set-up of the reference tables' minors (vbqmc_internal.h: TabMinors) on the host: the lists that the kernels
walk, walked here on random tables.  Every determinant's value is its minor, every derivative list gives its
cofactors, by entry and by determinant, shared minors and determinants formed by themselves alike.

Tables of normal entries: minors of order <= 4 by expansion are within a few roundings of sums of at most 24
products of at most 4 entries, cofactors likewise: 1e-12 of the largest of them."""
import ctypes
import dataclasses
import os
import subprocess

import numpy as np
import pytest

from paper_2207_14715_gb300 import systems as S
from paper_2207_14715_gb300 import vbqmc

CSRC = os.path.join(os.path.dirname(os.path.abspath(vbqmc.__file__)), "csrc")
LISTS = ["sl", "l1", "l2", "l3", "l4", "rt_off", "rt", "du_off", "du", "ld", "lr_off", "lh", "le"]

SOURCE = r"""
#include "%(csrc)s/vbqmc_internal.h"
static vbq::SysHost* h;
extern "C" int setup(const vbqmc_system_desc* d) {
  std::string err;
  delete h;
  h = new vbq::SysHost();
  return vbq::build_system(d, *h, err);
}
extern "C" void sizes(int sp, int* out) {
  const vbq::TabMinorsHost& t = h->tab_min[sp];
  int v[6] = {h->tab_ok, h->U[sp], t.ns, t.nx, t.nv, h->n[sp]};
  for (int i = 0; i < 6; ++i) out[i] = v[i];
}
extern "C" int list(int sp, int which, const int** data) {
  const vbq::TabMinorsHost& t = h->tab_min[sp];
  const std::vector<int>* l[] = {%(lists)s, &h->tab_det[sp]};
  *data = l[which]->data();
  return (int)l[which]->size();
}
"""


@pytest.fixture(scope="module")
def host(tmp_path_factory):
    d = tmp_path_factory.mktemp("minors")
    src, so = str(d / "minors.cpp"), str(d / "minors.so")
    with open(src, "w") as f:
        f.write(SOURCE % dict(csrc=CSRC, lists=", ".join("&t." + x for x in LISTS)))
    subprocess.run(["g++", "-O1", "-std=c++17", "-shared", "-fPIC", src, os.path.join(CSRC, "system_host.cpp"), "-o", so],
                   check=True)
    return ctypes.CDLL(so)


def _pairs(n_pairs, n_active, n_structures, seed=5):
    """n_pairs singlet pairs drawn from n_active active orbitals per structure, one core."""
    base = S.small_open_shell(params=False)
    rng = np.random.default_rng(seed)
    orb = np.concatenate([base.orb_coef[:1], rng.normal(size=(n_active, base.M))])
    strs = []
    for _ in range(n_structures):
        q = [int(v) for v in 1 + rng.permutation(n_active)[:2 * n_pairs]]
        strs.append(([0], sorted((min(q[2 * j:2 * j + 2]), max(q[2 * j:2 * j + 2])) for j in range(n_pairs)), []))
    io, ina, po, prs, uo, un = S._structures(strs)
    n = 1 + n_pairs
    return dataclasses.replace(
        base, orb_coef=orb, orb_class=np.full(len(orb), -1, np.int32), orb_kind=np.ones(len(orb), np.int32), n_up=n,
        n_dn=n, c_vb=np.ones(n_structures), inact_off=io, inact=ina, pair_off=po, pairs=prs, unp_off=uo, unp=un)


CASES = {"h2": S.h2_vb, "ethylene": S.ethylene_vb, "open_shell": S.small_open_shell, "dmc48": S.dmc48,
         "molecule": lambda: S.random_molecule(0), "shared": lambda: _pairs(4, 9, 6), "alone4": lambda: _pairs(4, 20, 24),
         "alone3": lambda: _pairs(3, 30, 30), "pairs": lambda: _pairs(2, 24, 40), "single": lambda: _pairs(1, 8, 6)}


@pytest.mark.parametrize("name", sorted(CASES))
def test_lists(host, name):
    desc = vbqmc._desc(CASES[name]())
    assert host.setup(ctypes.byref(desc[0] if isinstance(desc, tuple) else desc)) == 0
    for sp in (0, 1):
        size = (ctypes.c_int * 6)()
        host.sizes(sp, size)
        ok, U, ns, nx, nv, n = size
        assert ok
        L = {}
        for i, x in enumerate(LISTS + ["det"]):
            p = ctypes.POINTER(ctypes.c_int)()
            m = host.list(sp, i, ctypes.byref(p))
            L[x] = np.array(p[:m], np.int64)
        if n == 0:
            continue
        T = np.random.default_rng(7).normal(size=(ns, nx))
        t = T.ravel()
        row = {s: i for i, s in enumerate(L["sl"])}
        dets = [(r[0], [row[s] for s in r[2:2 + r[0]]], list(r[6:6 + r[0]])) for r in L["det"].reshape(U, -1)]
        alone = name.startswith("alone")
        assert (len(L["ld"]) > 0) == alone and len(L["ld"]) % 4 == 0
        # values, size by size
        v = np.full(nv, np.nan)
        v[0] = 1.0
        for c, e in L["l1"].reshape(-1, 2):
            v[c] = t[e]
        for c, a, b, _ in L["l2"].reshape(-1, 4):
            v[c] = t[a & 0xffff] * t[a >> 16] - t[b & 0xffff] * t[b >> 16]
        for l, k in ((L["l3"].reshape(-1, 4), 3), (L["l4"].reshape(-1, 8), 4)):
            for e in l:
                v[e[0]] = sum((-1) ** j * t[e[1 + j] & 0xffff] * v[e[1 + j] >> 16] for j in range(k))
        lone = {}
        for c, rows, c01, c23 in L["ld"].reshape(-1, 4) & 0xffffffff:
            k = c >> 28
            cols = [c01 & 0xffff, c01 >> 16, c23 & 0xffff, c23 >> 16][:k]
            lone[c & 0xfffffff] = (k, [(rows >> 8 * i) & 0xff for i in range(k)], cols)
            v[c & 0xfffffff] = np.linalg.det(T[np.ix_(lone[c & 0xfffffff][1], cols)])
        cof = np.zeros((U, ns * nx))
        for u, (k, rows, cols) in enumerate(dets):
            M = T[np.ix_(rows, cols)]
            assert abs(v[u] - (np.linalg.det(M) if k else 1.0)) <= 1e-12 * max(1.0, np.abs(T).max() ** 4)
            if u in lone:
                assert lone[u] == (k, rows, cols) and k >= 3
            for i in range(k):
                for j in range(k):
                    sub = np.delete(np.delete(M, i, 0), j, 1)
                    cof[u, rows[i] * nx + cols[j]] = (-1) ** (i + j) * (np.linalg.det(sub) if k > 1 else 1.0)
        # derivatives by determinant and by entry, each cofactor 1, a minor or an entry
        code = lambda c: 1.0 if c < 0 else (t[c - 0x10000] if c >= 0x10000 else v[c])  # noqa: E731
        got = np.zeros((2, U, ns * nx))
        du, rt = L["du"].reshape(-1, 2), L["rt"].reshape(-1, 2)
        assert len(L["du_off"]) == U + 1 and len(L["rt_off"]) == ns * nx + 1
        for u in range(U):
            for e, c in du[L["du_off"][u]:L["du_off"][u + 1]]:
                got[0, u, e & 0x7fffffff] += -code(c) if e < 0 else code(c)
        for e in range(ns * nx):
            for u, c in rt[L["rt_off"][e]:L["rt_off"][e + 1]]:
                got[1, u & 0x7fffffff, e] += -code(c) if u < 0 else code(c)
        # the determinants formed by themselves: entries of each round of 32, every cofactor once
        order, heads = list(L["ld"].reshape(-1, 4)[:, 0] & 0xfffffff), L["lh"].reshape(-1, 2)
        assert heads[-1, 1] == len(L["le"]) and L["lr_off"][-1] == len(heads) - 1
        for r in range(len(L["lr_off"]) - 1):
            for h in range(L["lr_off"][r], L["lr_off"][r + 1]):
                for c in L["le"][heads[h, 1]:heads[h + 1, 1]]:
                    u = order[32 * r + (c >> 4)]
                    k, rows, cols = lone[u]
                    i, j = (c & 15) >> 2, c & 3
                    assert rows[i] * nx + cols[j] == heads[h, 0]
                    got[:, u, heads[h, 0]] += cof[u, heads[h, 0]]
        assert np.abs(got - cof).max() <= 1e-12 * max(1.0, np.abs(T).max() ** 3)
