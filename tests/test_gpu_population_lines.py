"""Both sides of the dispatch lines by size that smaller tests leave out.

Populations: past two rounds of walkers over the SMs (48 electrons in the mixed form: 2 x 10 x 152 walkers of the
table evaluation, 2 x 9 x 152 of the sweep; ethylene-shaped system: 2 x 16 x 152) the kernels run in their
smallest full blocks; the first walkers of such a population alone are spread over the SMs.  A walker's
arithmetic is that of its own warp: equal bit for bit.

Linear method: 64-column tiles whose last one passes the stored columns (100 parameters: two tiles over
112), as every linear-method test within 1e-5 (float) or 2e-6 (double) of the matrix scale."""
import numpy as np
import pytest

pytestmark = pytest.mark.gpu
torch = pytest.importorskip("torch")

from paper_2207_14715_gb300 import systems as S  # noqa: E402
from paper_2207_14715_gb300 import vbqmc  # noqa: E402


def _run(spec, R0):
    W, P, dt = R0.shape[0], spec.n_params, vbqmc.deriv_dtype(vbqmc.MIXED)
    ctx = vbqmc.create(0)
    ctx.set_system(0, spec)
    R = R0.clone()
    z = lambda *shape, dtype=torch.float64: torch.zeros(shape, dtype=dtype, device="cuda:0")  # noqa: E731
    lp, sg, el, na = z(W), z(W), z(W), z(W, dtype=torch.int32)
    O, dE = (z(W, P, dtype=dt), z(W, P, dtype=dt)) if P else (None, None)
    ctx.vmc_steps(0, vbqmc.MIXED, R, 2, spec.step, 5, step0=0, refresh=0, nacc=na, logpsi=lp, sign=sg, eloc=el, O=O,
                  dEL=dE)
    torch.cuda.synchronize()
    ctx.close()
    return [t for t in (R, na, lp, sg, el, O, dE) if t is not None]


@pytest.mark.parametrize("name,W", [("dmc48", 3301), ("ethylene_vb", 5101)])
def test_many_rounds(name, W):
    spec = getattr(S, name)()
    R0 = torch.tensor(S.initial_walkers(spec, W, 3), device="cuda:0")
    whole = _run(spec, R0)
    for k in (1, 700, 2600):
        for a, b in zip(whole, _run(spec, R0[:k].contiguous())):
            assert torch.equal(a[:k], b)


@pytest.mark.parametrize("precision", [0, 1])
def test_ragged_64_column_tiles(orc, precision):
    M, P = 90000, 100
    rng = np.random.default_rng(1)
    O = rng.normal(size=(M, P)) + rng.normal(size=P)
    dE = rng.normal(size=(M, P)) * 0.3
    E = -10.0 + rng.normal(size=M) + 0.5 * O[:, 0]
    dt = vbqmc.deriv_dtype(precision)
    dev = lambda x, d=torch.float64: torch.tensor(x, dtype=d, device="cuda")  # noqa: E731
    Od, Dd = dev(O, dt), dev(dE, dt)
    ctx = vbqmc.create(0)
    got = ctx.accumulate_lin_matrices(precision, Od, Dd, dev(E))
    ref = orc.lin_matrices(Od.double().cpu().numpy(), Dd.double().cpu().numpy(), E, None)
    for k in ("S", "H", "gL", "gR"):
        err = np.abs(got[k].cpu().numpy() - ref[k]).max() / max(1.0, np.abs(ref[k]).max())
        assert err < (2e-6 if precision == 0 else 1e-5), (k, err)
    ctx.close()
