"""The walkers of a launch are spread over blocks by their number (one walker per warp): results of a
walker do not depend on how many others are in the call.  The first walkers of a large population
(several rounds over the SMs, the smallest blocks) are compared with the same walkers alone (spread over
idle SMs), bit for bit: a walker's arithmetic is that of its own warp."""
import pytest

pytestmark = pytest.mark.gpu
torch = pytest.importorskip("torch")

from paper_2207_14715_gb300 import systems as S  # noqa: E402
from paper_2207_14715_gb300 import vbqmc  # noqa: E402


def _run(spec, prec, R0):
    W, P, dt = R0.shape[0], spec.n_params, vbqmc.deriv_dtype(prec)
    ctx = vbqmc.create(0)
    ctx.set_system(0, spec)
    R = R0.clone()
    z = lambda *shape, dtype=torch.float64: torch.zeros(shape, dtype=dtype, device="cuda:0")  # noqa: E731
    lp, sg, el, na = z(W), z(W), z(W), z(W, dtype=torch.int32)
    O, dE = (z(W, P, dtype=dt), z(W, P, dtype=dt)) if P else (None, None)
    ctx.vmc_steps(0, prec, R, 2, spec.step, 5, step0=0, refresh=0, nacc=na, logpsi=lp, sign=sg, eloc=el, O=O, dEL=dE)
    torch.cuda.synchronize()
    return [t for t in (R, na, lp, sg, el, O, dE) if t is not None]


@pytest.mark.parametrize("precision", ["fp64", "mixed"])
@pytest.mark.parametrize("name,W", [("open_shell", 5333), ("ethylene", 2801), ("dmc48", 1301)])
def test_population_size(name, W, precision):
    spec = {"open_shell": S.small_open_shell, "ethylene": S.ethylene_vb, "dmc48": S.dmc48}[name]()
    prec = vbqmc.FP64 if precision == "fp64" else vbqmc.MIXED
    R0 = torch.tensor(S.initial_walkers(spec, W, 3), device="cuda:0")
    whole = _run(spec, prec, R0)
    for k in (1, 2, 153, 1000):
        for a, b in zip(whole, _run(spec, prec, R0[:k].contiguous())):
            assert torch.equal(a[:k], b)
