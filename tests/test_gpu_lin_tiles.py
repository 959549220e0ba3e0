"""Linear-method accumulation at the edges of its output tiles (32, 64 or 112 columns by the size
of the sample), of the centring blocks (1 to 8 tiles of 64 samples) and of the stored columns,
against the oracle.  Tolerance as for every linear-method test: centred values rounded to float
and split into halves, 1e-5 of the matrix scale for float inputs, 2e-6 for double inputs."""
import numpy as np
import pytest

pytestmark = pytest.mark.gpu
torch = pytest.importorskip("torch")


@pytest.fixture(scope="module")
def vb():
    if not torch.cuda.is_available():
        pytest.skip("no CUDA device")
    from paper_2207_14715_gb300 import build, vbqmc
    build.build()
    ctx = vbqmc.create(0)
    yield vbqmc, ctx
    ctx.close()


# 32-column tiles: P at a tile's edge, and past the last 112-column boundary (99, 113); 64-column
# tiles: 8000 x 400; 112-column tiles: 19000 x 400; samples at the edges of a 64-sample tile
@pytest.mark.parametrize("M,P,weights", [(63, 31, False), (65, 33, True), (129, 99, True), (4096, 113, False),
                                         (15001, 216, True), (8000, 400, False), (19000, 400, True)])
@pytest.mark.parametrize("precision", [0, 1])
def test_tiles_match_oracle(vb, orc, M, P, weights, precision):
    mod, ctx = vb
    rng = np.random.default_rng(M + P)
    O = rng.normal(size=(M, P)) + rng.normal(size=P)
    dE = rng.normal(size=(M, P)) * 0.3
    E = -10.0 + rng.normal(size=M) + 0.5 * O[:, 0]
    w = rng.uniform(0.2, 1.8, M) if weights else None
    dt = mod.deriv_dtype(precision)
    dev = lambda x, d=torch.float64: None if x is None else torch.tensor(x, dtype=d, device="cuda")
    Od, Dd = dev(O, dt), dev(dE, dt)
    got = ctx.accumulate_lin_matrices(precision, Od, Dd, dev(E), dev(w))
    ref = orc.lin_matrices(Od.double().cpu().numpy(), Dd.double().cpu().numpy(), E, w)
    for k in ("S", "H", "gL", "gR"):
        err = np.abs(got[k].cpu().numpy() - ref[k]).max() / max(1.0, np.abs(ref[k]).max())
        assert err < (2e-6 if precision == 0 else 1e-5), (k, err)
