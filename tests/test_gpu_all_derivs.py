"""Parameter and nucleus derivatives from one evaluation: the same kernels on the same inputs as the two
separate calls, so every output is equal bit for bit; either kind can be left out; errors as before."""
import pytest

pytestmark = pytest.mark.gpu
torch = pytest.importorskip("torch")

from paper_2207_14715_gb300 import systems as S  # noqa: E402
from paper_2207_14715_gb300 import vbqmc  # noqa: E402


@pytest.mark.parametrize("precision", ["fp64", "mixed"])
@pytest.mark.parametrize("name,W", [("h2_vb", 1), ("small_open_shell", 311), ("ethylene_vb_p400", 153)])
def test_one_evaluation(name, W, precision):
    spec = getattr(S, name)()
    prec = vbqmc.FP64 if precision == "fp64" else vbqmc.MIXED
    ctx = vbqmc.create(0)
    ctx.set_system(0, spec)
    R = torch.tensor(S.initial_walkers(spec, W, 3), device="cuda:0")
    z = lambda *s, dtype=torch.float64: torch.zeros(s, dtype=dtype, device="cuda:0")  # noqa: E731
    P, dt = spec.n_params, vbqmc.deriv_dtype(prec)
    e, n, b = ([z(W), z(W), z(W)] for _ in range(3))
    O, dE, O2, dE2 = (z(W, P, dtype=dt) if P else None for _ in range(4))
    dl, dR, dl2, dR2 = (z(W, spec.Nn, 3) for _ in range(4))
    ctx.eval_walkers(0, prec, R, *e, O=O, dEL=dE)
    ctx.eval_nuclear_derivs(0, prec, R, *n, dl, dR)
    ctx.eval_nuclear_derivs(0, prec, R, *b, dl2, dR2, O=O2, dEL=dE2)
    torch.cuda.synchronize()
    for x, y in list(zip(e, b)) + list(zip(n, b)) + [(dl, dl2), (dR, dR2)] + ([(O, O2), (dE, dE2)] if P else []):
        assert torch.equal(x, y)
    if P:
        with pytest.raises(vbqmc.VbqmcError):
            ctx.eval_nuclear_derivs(0, prec, R, *b, dl2, dR2, dEL=dE2)
