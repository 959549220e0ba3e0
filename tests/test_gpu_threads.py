"""Host threads, each with a context, stream and walkers of its own, call the same system with different
populations at the same time.  A launch's shared memory depends on its population, the kernel's limit
does not: no call of either thread fails, and each thread's results are those of the same calls alone,
bit for bit.  In processes of their own, where the threads' first launches of every kernel coincide: with a
limit that follows the population, the larger one's first call failed in nine processes of ten (while a
kernel is being loaded, the other thread sets its own)."""
import os
import subprocess
import sys

import pytest

pytestmark = pytest.mark.gpu
torch = pytest.importorskip("torch")

ROOT = os.path.dirname(os.path.dirname(os.path.abspath(__file__)))

# populations with blocks of different sizes in the sweep and evaluation kernels: one below a round of
# walkers over the SMs (spread over small blocks), one of one to two rounds (full blocks)
SCRIPT = r"""
import sys, threading
sys.setswitchinterval(1e-5)
import torch
from paper_2207_14715_gb300 import systems as S, vbqmc

class Run:
    def __init__(self, spec, tables, prec, W):
        z = lambda *s, dtype=torch.float64: torch.zeros(s, dtype=dtype, device="cuda:0")
        self.args = spec, tables, prec, W
        self.R = torch.tensor(S.initial_walkers(spec, W, 3), device="cuda:0")
        dt = vbqmc.deriv_dtype(prec)
        self.out = [z(W), z(W), z(W), z(W, spec.n_params, dtype=dt), z(W, spec.n_params, dtype=dt)]
        self.errors = []

    def __call__(self, barrier=None):
        spec, tables, prec, W = self.args
        with torch.cuda.stream(torch.cuda.Stream()):
            ctx = vbqmc.create(0)
            ctx.set_system(0, spec)
            if tables:
                ctx.use_tables(0, True)
            if barrier:
                barrier.wait(timeout=60)
            for k in range(40):
                try:
                    ctx.eval_walkers(0, prec, self.R, *self.out[:3], O=self.out[3], dEL=self.out[4])
                    ctx.vmc_steps(0, prec, self.R, 1, spec.step, 5, step0=k)
                except vbqmc.VbqmcError as e:
                    self.errors.append((k, str(e)))
            torch.cuda.current_stream().synchronize()

ok = True
for name, tables, prec in [(n, t, p) for n, t in (("small_open_shell", 0), ("h2_vb", 1)) for p in (vbqmc.MIXED, vbqmc.FP64)]:
    spec = getattr(S, name)()
    both, barrier = [Run(spec, tables, prec, W) for W in (150, 2400)], threading.Barrier(2)
    torch.cuda.synchronize()
    threads = [threading.Thread(target=r, args=(barrier,)) for r in both]
    for t in threads: t.start()
    for t in threads: t.join()
    for b in both:
        if b.errors:
            print(name, prec, b.args[3], len(b.errors), b.errors[0])
            ok = False
            continue
        a = Run(*b.args)
        a()
        for x, y in zip([a.R] + a.out, [b.R] + b.out):
            ok &= torch.equal(x, y)
print("all equal" if ok else "failed")
"""


@pytest.mark.parametrize("process", range(3))
def test_threads_with_different_populations(process):
    if not torch.cuda.is_available():
        pytest.skip("no CUDA device")
    r = subprocess.run([sys.executable, "-c", SCRIPT], capture_output=True, text=True, cwd=ROOT, timeout=300,
                       env=dict(os.environ, PYTHONPATH=ROOT))
    assert r.returncode == 0 and r.stdout.strip() == "all equal", r.stdout + r.stderr[-2000:]
