"""Reference tables whose determinants need minors of their own: few replaced slots over many
orbitals, so that the shared expansion of the minors adds more values than determinants (it then
expands each determinant by itself), and a smaller one that stays shared, against the oracle.

Tolerances as for the other table systems: FP64 ln|Psi| and E_L 1e-10, gradient 1e-9, derivatives
1e-8 of max(1, |x|), sweeps move for move (positions to 1e-12)."""
import dataclasses

import numpy as np
import pytest

from paper_2207_14715_gb300 import systems as S

pytestmark = pytest.mark.gpu
torch = pytest.importorskip("torch")


def system(n_pairs, n_active, n_structures, seed=5):
    """n_pairs singlet pairs drawn from n_active well-separated active orbitals per structure, one
    core, on the nuclei and basis of the open-shell test system."""
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


@pytest.mark.parametrize("n_pairs,n_active,n_structures", [(4, 22, 12), (4, 9, 6), (3, 20, 10), (2, 5, 3), (1, 3, 2)])
def test_tables_match_oracle(orc, n_pairs, n_active, n_structures):
    if not torch.cuda.is_available():
        pytest.skip("no CUDA device")
    from paper_2207_14715_gb300 import build, vbqmc
    build.build()
    spec = system(n_pairs, n_active, n_structures)
    ctx = vbqmc.create(0)
    ctx.set_system(0, spec)
    ctx.use_tables(0, True)
    W = 40
    R0 = S.initial_walkers(spec, W, 3)
    R = torch.tensor(R0, device="cuda")
    lp, sg, el = (torch.zeros(W, dtype=torch.float64, device="cuda") for _ in range(3))
    O = torch.zeros((W, spec.n_params), dtype=torch.float64, device="cuda")
    dE = torch.zeros_like(O)
    g = torch.zeros_like(R)
    ctx.eval_walkers(0, vbqmc.FP64, R, lp, sg, el, g, O, dE)
    ref = orc.evaluate(spec, R0, derivs=True, grad=True)
    rel = lambda a, b: (np.abs(a.cpu().numpy() - b) / np.maximum(1.0, np.abs(b))).max()
    assert (sg.cpu().numpy() == ref["sign"]).all()
    assert rel(lp, ref["logpsi"]) < 1e-10 and rel(el, ref["eloc"]) < 1e-10 and rel(g, ref["grad"]) < 1e-9
    assert rel(O, ref["O"]) < 1e-8 and rel(dE, ref["dEL"]) < 1e-8
    ctx.vmc_steps(0, vbqmc.FP64, R, 3, spec.step, 11, step0=2)
    Ro, _, _, _ = orc.vmc(spec, R0, 3, spec.step, seed=11, step0=2, eloc=False)
    assert np.abs(R.cpu().numpy() - Ro).max() < 1e-12
    ctx.close()
