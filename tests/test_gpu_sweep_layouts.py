"""Sweeps over the forms of the sweep kernel's layout against the oracle's trajectories: proposal rows
for 4, 2 or 1 electrons at a time (by the number of nuclei, up to more than a warp has lanes), both
spins prepared together or one after the other (more than 32 electrons, or too large a region), spins
with the same and with different orbitals, an empty spin, one and several rounds of contraction chunks.

Double form: the proposals are computed with the oracle's rounding, so that trajectories agree to
1e-12 unless a uniform falls within the rounding of an acceptance probability (1e-13 a move).
Mixed form: the probability carries float errors of the orbital row and of the exponent (1e-4
at most), so that among the 64 x 3 x N <= 9216 moves of a case about one can be decided otherwise;
4 walkers of 64 may differ."""
import dataclasses

import numpy as np
import pytest

pytestmark = pytest.mark.gpu
torch = pytest.importorskip("torch")

from oracle import oracle as orc  # noqa: E402
from paper_2207_14715_gb300 import systems as S  # noqa: E402
from paper_2207_14715_gb300 import vbqmc  # noqa: E402


def _nuclei(count):
    """The open-shell system with distant further nuclei of its first element."""
    sp = S.small_open_shell()
    k = count - sp.Nn
    xyz = 4.0 + np.stack([np.arange(k), np.arange(k) % 3, np.arange(k) % 5], axis=1).astype(np.float64)
    return dataclasses.replace(sp, name="nuclei%d" % count, nuc_xyz=np.concatenate([np.asarray(sp.nuc_xyz), xyz]),
                               nuc_Z=np.concatenate([np.asarray(sp.nuc_Z), np.full(k, np.asarray(sp.nuc_Z)[0])]),
                               nuc_elem=np.concatenate([np.asarray(sp.nuc_elem), np.full(k, np.asarray(sp.nuc_elem)[0])]))


CASES = {
    "h2": S.h2_vb, "one_electron": lambda: S.one_electron(1.0, 1.2), "slater": S.slater_h2,
    "open_shell": S.small_open_shell, "nuclei8": lambda: _nuclei(8), "nuclei9": lambda: _nuclei(9),
    "nuclei17": lambda: _nuclei(17), "nuclei34": lambda: _nuclei(34), "ethylene": S.ethylene_vb,
    "p400": S.ethylene_vb_p400, "bovb": S.ethylene_bovb, "many": lambda: S.random_molecule(0), "dmc48": S.dmc48,
}


@pytest.mark.parametrize("precision", ["fp64", "mixed"])
@pytest.mark.parametrize("name", sorted(CASES))
def test_trajectories(name, precision):
    spec = CASES[name]()
    W, sweeps = (64, 3) if precision == "mixed" else (8, 3)
    R0 = S.initial_walkers(spec, W, 5)
    ctx = vbqmc.create(0)
    ctx.set_system(0, spec)
    R = torch.tensor(R0, dtype=torch.float64, device="cuda:0")
    nacc = torch.zeros(W, dtype=torch.int32, device="cuda:0")
    ctx.vmc_steps(0, vbqmc.FP64 if precision == "fp64" else vbqmc.MIXED, R, sweeps, spec.step, 11, step0=0, refresh=2,
                  nacc=nacc)
    torch.cuda.synchronize()
    Ro = orc.vmc(spec, R0, sweeps, spec.step, seed=11, step0=0, eloc=False)[0]
    off = np.abs(R.cpu().numpy() - Ro).reshape(W, -1).max(axis=1) > 1e-12
    assert off.sum() <= (4 if precision == "mixed" else 0), np.flatnonzero(off)
    assert 0 < int(nacc.sum()) <= W * sweeps * spec.N
