"""Linear-method accumulation of samples with more block partials than are summed in one go (4096: past 2^20
samples for the column sums, past 2^21 for w Ot E as well), whose sums run over segments first, on either
side of both lines, against the oracle.  Tolerance as for every linear-method test: 1e-5 of the matrix
scale for float inputs, 2e-6 for double inputs."""
import numpy as np
import pytest

pytestmark = pytest.mark.gpu
torch = pytest.importorskip("torch")


@pytest.mark.parametrize("M", [1 << 20, (1 << 20) + 1, (1 << 21) + 1, 2500003])
@pytest.mark.parametrize("precision", [0, 1])
def test_segments_match_oracle(orc, M, precision):
    if not torch.cuda.is_available():
        pytest.skip("no CUDA device")
    from paper_2207_14715_gb300 import build, vbqmc
    build.build()
    P = 5
    rng = np.random.default_rng(M % 1000)
    O = rng.normal(size=(M, P)) + rng.normal(size=P)
    dE = rng.normal(size=(M, P)) * 0.3
    E = -10.0 + rng.normal(size=M) + 0.5 * O[:, 0]
    w = rng.uniform(0.2, 1.8, M)
    dt = vbqmc.deriv_dtype(precision)
    dev = lambda x, d=torch.float64: torch.tensor(x, dtype=d, device="cuda")  # noqa: E731
    Od, Dd = dev(O, dt), dev(dE, dt)
    ctx = vbqmc.create(0)
    got = ctx.accumulate_lin_matrices(precision, Od, Dd, dev(E), dev(w))
    ref = orc.lin_matrices(Od.double().cpu().numpy(), Dd.double().cpu().numpy(), E, w)
    for k in ("S", "H", "gL", "gR"):
        err = np.abs(got[k].cpu().numpy() - ref[k]).max() / max(1.0, np.abs(ref[k]).max())
        assert err < (2e-6 if precision == 0 else 1e-5), (k, err)
    ctx.close()
