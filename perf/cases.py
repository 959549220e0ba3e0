"""Performance cases of the VB-QMC library: what a user's program has it do, through the public
entry points, with the inputs such a program holds and 64-bit reference results.

Every case is a dict of plain values.  kind:
  step      one VMC walker-step: a sweep from the carried walker state, then ln|Psi|, E_L and every
            parameter derivative (the sampling loop of a wave-function optimisation)
  eval      evaluation of walkers that come without a state: fresh Slater factorisation, gradient,
            derivatives and the new state (walkers read from a file or moved by the caller)
  sweeps    sweeps alone (equilibration, decorrelation between measurements)
  dmc       fixed-node diffusion Monte Carlo steps
  forces    ln|Psi|, E_L and their derivatives with respect to the nuclei
  lin       linear-method matrices of a sample; "noalloc": through the allocation-free entry
  gradient  energy and its gradient in parameters and nuclei through the autograd face
  batch     one step of many small uneven molecules at once

The 64-bit results (exact) come from plain torch arithmetic on the system description: basis,
determinant expansion, Jastrow factor, local energy, derivatives and Metropolis moves are written
out below from the method's formulas (arXiv:2207.14715) and share nothing with the library.
"""
import functools
import itertools
import math

import numpy as np
import torch

from paper_2207_14715_gb300 import autograd, systems, vbqmc

PRECISION = {"mixed": vbqmc.MIXED, "fp64": vbqmc.FP64}
DEV = "cuda"


# ---------------------------------------------------------------------------------------
# cases
# ---------------------------------------------------------------------------------------
def listed():
    return [
        # smallest call: two electrons, launches and latency count
        dict(name="step_h2_1024_mixed", kind="step", system="h2", walkers=1024, precision="mixed"),
        # the benchmark's workload: 16 electrons, 216 parameters, default walker population
        dict(name="step_ethylene_16384_mixed", kind="step", system="ethylene", walkers=16384, precision="mixed"),
        # the same in full double precision (reference runs, checks of the mixed form); ragged
        dict(name="step_ethylene_3001_fp64", kind="step", system="ethylene", walkers=3001, precision="fp64"),
        # walkers without a state: LU of every determinant, gradient, state and derivatives
        dict(name="eval_ethylene_6001_mixed", kind="eval", system="ethylene", walkers=6001, precision="mixed"),
        # equilibration of a population, refactorised now and then
        dict(name="sweeps_ethylene_4096_mixed", kind="sweeps", system="ethylene", walkers=4096, sweeps=10,
             refresh=5, precision="mixed"),
        # decorrelating sweep of the 48-electron system (256 determinants on reference tables)
        dict(name="sweeps_dmc48_8192_mixed", kind="sweeps", system="dmc48", walkers=8192, sweeps=1, refresh=10,
             precision="mixed"),
        # diffusion Monte Carlo of the 48-electron system
        dict(name="dmc_dmc48_4096_mixed", kind="dmc", system="dmc48", walkers=4096, steps=2, precision="mixed"),
        # forces on the nuclei of a sample
        dict(name="forces_ethylene_2500_mixed", kind="forces", system="ethylene", walkers=2500, precision="mixed"),
        # linear-method matrices at the benchmark's size, and a small double one with sample weights
        # through the allocation-free entry
        dict(name="lin_1048576x400_mixed", kind="lin", samples=1 << 20, params=400, precision="mixed",
             weights=False, noalloc=False),
        dict(name="lin_15001x216_fp64", kind="lin", samples=15001, params=216, precision="fp64", weights=True,
             noalloc=True),
        # gradient of the energy for an optimiser that is driven from torch
        dict(name="gradient_ethylene_2048_mixed", kind="gradient", system="ethylene", walkers=2048,
             precision="mixed"),
        # many small molecules of uneven size in one batch
        dict(name="batch_16_molecules_mixed", kind="batch", molecules=16, workload=7, precision="mixed"),
    ]


def _log_int(rng, lo, hi):
    return int(round(math.exp(rng.uniform(math.log(lo), math.log(hi)))))


def draw(rng):
    kind = rng.choice(["step", "step", "eval", "sweeps", "sweeps", "dmc", "forces", "lin", "lin", "gradient", "batch"])
    prec = "mixed" if rng.random() < 0.7 else "fp64"
    most = {"mixed": 16384, "fp64": 3001}[prec]
    if kind in ("step", "eval"):
        return dict(kind=kind, system=rng.choice(["h2", "open_shell", "ethylene", "slater_h2", "bovb"]),
                    walkers=_log_int(rng, 200, most if kind == "step" else most // 2), precision=prec)
    if kind == "sweeps":
        if rng.random() < 0.5:
            return dict(kind=kind, system="dmc48", walkers=_log_int(rng, 500, 8192), sweeps=1, refresh=10,
                        precision="mixed")
        return dict(kind=kind, system=rng.choice(["h2", "open_shell", "ethylene"]),
                    walkers=_log_int(rng, 200, 4096 if prec == "mixed" else 1024), sweeps=rng.choice([2, 5, 10]),
                    refresh=rng.choice([1, 5, 10]), precision=prec)
    if kind == "dmc":
        big = rng.random() < 0.5
        return dict(kind=kind, system="dmc48" if big else "ethylene", walkers=_log_int(rng, 1000, 4096),
                    steps=rng.choice([1, 2]), precision="mixed")
    if kind in ("forces", "gradient"):
        return dict(kind=kind, system=rng.choice(["h2", "open_shell", "ethylene"]),
                    walkers=_log_int(rng, 200, 2500 if prec == "mixed" else 600), precision=prec)
    if kind == "lin":
        p = _log_int(rng, 20, 400)
        noalloc = rng.random() < 0.3
        m = _log_int(rng, 1000, 15000 if noalloc else (1 << 20 if prec == "mixed" else 1 << 18))
        return dict(kind=kind, samples=m, params=min(p, 216) if noalloc else p, precision=prec,
                    weights=rng.random() < 0.5, noalloc=noalloc)
    return dict(kind="batch", molecules=rng.randrange(4, 17), workload=rng.randrange(1, 1000), precision="mixed")


def _system(name):
    return {"h2": systems.h2_vb, "open_shell": systems.small_open_shell, "ethylene": systems.ethylene_vb,
            "slater_h2": systems.slater_h2, "bovb": systems.ethylene_bovb, "dmc48": systems.dmc48}[name]()


@functools.lru_cache(maxsize=8)
def _molecules(count, workload):
    """Molecules and walker counts of a batch.  Of the random molecules, those whose orbitals carry
    their electrons: some have an atom with tight functions only, where every Slater matrix of a
    starting configuration is singular to working precision and E_L is noise in any arithmetic."""
    rng, specs = np.random.default_rng(workload), []
    for i in itertools.count():
        sp = systems.random_molecule(workload * 1000 + i)
        psi = _Psi(sp)
        A = psi.slater(psi.orbitals(_walkers(sp, 32, 0), psi.X, False)[0])[0]
        A = torch.cat([a[:, 0] for a in A]).cpu()
        A = A / A.norm(dim=1, keepdim=True)
        if torch.linalg.cond(A / A.norm(dim=2, keepdim=True)).quantile(0.9) < 1000:
            specs.append(sp)
        if len(specs) == count:
            return specs, [32 * int(round(math.exp(rng.uniform(math.log(8), math.log(32))))) for _ in specs]


def _workload(case):
    return _molecules(case["molecules"], case["workload"])


# ---------------------------------------------------------------------------------------
# what a user's program has in hand, and one pass
# ---------------------------------------------------------------------------------------
def _zeros(*shape, dtype=torch.float64):
    return torch.zeros(shape, dtype=dtype, device=DEV)


def _walkers(spec, W, seed):
    return torch.tensor(systems.initial_walkers(spec, W, seed), device=DEV)


def _lin_inputs(case, seed):
    g = torch.Generator(device=DEV)
    g.manual_seed(seed)
    M, P = case["samples"], case["params"]
    dt = torch.float32 if case["precision"] == "mixed" else torch.float64
    mean = torch.randn(P, generator=g, device=DEV, dtype=dt)
    O = torch.randn((M, P), generator=g, device=DEV, dtype=dt).add_(mean)
    dE = torch.randn((M, P), generator=g, device=DEV, dtype=dt).mul_(0.3)
    E = -10.0 + torch.randn(M, generator=g, device=DEV, dtype=torch.float64)
    w = 0.5 + torch.rand(M, generator=g, device=DEV, dtype=torch.float64) if case["weights"] else None
    return O, dE, E, w


def prepare(case, seed):
    s = dict(case=case, seed=seed, kind=case["kind"], prec=PRECISION[case["precision"]])
    if s["kind"] == "lin":
        s["O"], s["dE"], s["E"], s["w"] = _lin_inputs(case, seed)
        s["ctx"] = vbqmc.create(0)
        P = case["params"]
        if case["noalloc"]:
            s["out"] = dict(E0=_zeros(1), gL=_zeros(P), gR=_zeros(P), S=_zeros(P, P), H=_zeros(P, P))
        return s
    ctx = s["ctx"] = vbqmc.create(0)
    dt = vbqmc.deriv_dtype(s["prec"])
    if s["kind"] == "batch":
        specs, Ws = _workload(case)
        for k, sp in enumerate(specs):
            ctx.set_system(k, sp)
        flat = {}

        def rows(name, sizes, dtype=torch.float64):  # one buffer, a piece of it for each system
            flat[name] = torch.zeros(sum(w * m for w, m in zip(Ws, sizes)), dtype=dtype, device=DEV)
            return list(flat[name].split([w * m for w, m in zip(Ws, sizes)]))

        one = [1] * len(specs)
        R = rows("R", [3 * sp.N for sp in specs])
        for k, sp in enumerate(specs):
            R[k].copy_(_walkers(sp, Ws[k], seed * 1000 + k).reshape(-1))
        s["R"] = [r.view(w, sp.N, 3) for r, w, sp in zip(R, Ws, specs)]
        s["args"] = dict(state=rows("state", [ctx.walker_state_size(k) for k in range(len(specs))]),
                         nacc=rows("nacc", one, torch.int32), logpsi=rows("logpsi", one), sign=rows("sign", one),
                         eloc=rows("eloc", one), O=rows("O", [sp.n_params for sp in specs], dt),
                         dEL=rows("dEL", [sp.n_params for sp in specs], dt))
        s["batch"] = vbqmc.Batch(ctx, list(range(len(specs))), Ws, s["prec"])
        s["flat"], s["specs"], s["k"] = flat, specs, 0
        return s
    spec = s["spec"] = _system(case["system"])
    W, P = case["walkers"], spec.n_params
    ctx.set_system(0, spec)
    s["lp"], s["sg"], s["el"] = _zeros(W), _zeros(W), _zeros(W)
    R = s["R"] = _walkers(spec, W, seed)
    s["k"] = 0
    if s["kind"] in ("step", "eval"):
        s["O"], s["dE"] = _zeros(W, P, dtype=dt), _zeros(W, P, dtype=dt)
        s["state"] = _zeros(W, ctx.walker_state_size(0))
        if s["kind"] == "step":
            s["nacc"] = _zeros(W, dtype=torch.int32)
            s["k"] = 7  # the third step of a fresh run refactorises (every tenth does)
            ctx.eval_walkers(0, s["prec"], R, s["lp"], s["sg"], s["el"], state_out=s["state"])
        else:
            s["grad"] = _zeros(W, spec.N, 3)
    elif s["kind"] == "sweeps":
        s["nacc"] = _zeros(W, dtype=torch.int32)
    elif s["kind"] == "dmc":
        # a run starts from equilibrated walkers and their mean energy (double form)
        ctx.vmc_steps(0, vbqmc.FP64, R, 6 if case["system"] == "dmc48" else 20, spec.step, seed, step0=1 << 20)
        ctx.eval_walkers(0, vbqmc.FP64, R, s["lp"], s["sg"], s["el"])
        s["E_T"] = float(s["el"].median().item())
        s["R"] = torch.zeros((2 * W, spec.N, 3), dtype=torch.float64, device=DEV)
        s["R"][:W] = R
        s["W"] = W
    elif s["kind"] == "forces":
        s["dlp"], s["dER"] = _zeros(W, spec.Nn, 3), _zeros(W, spec.Nn, 3)
    elif s["kind"] == "gradient":
        s["p"] = torch.tensor(autograd.parameter_vector(spec), requires_grad=True)
        s["X"] = torch.tensor(np.asarray(spec.nuc_xyz, np.float64), requires_grad=True)
    return s


def run(s):
    kind, prec, ctx, case = s["kind"], s["prec"], s["ctx"], s["case"]
    if kind == "lin":
        if case["noalloc"]:
            o = s["out"]
            vbqmc.accumulate_lin_matrices_noalloc(prec, s["O"], s["dE"], s["E"], s["w"], o["E0"], o["gL"], o["gR"],
                                                  o["S"], o["H"])
            return o
        return ctx.accumulate_lin_matrices(prec, s["O"], s["dE"], s["E"], weights=s["w"])
    if kind == "batch":
        s["batch"].vmc_steps(s["R"], 1, 0.3, s["seed"], step0=s["k"], refresh=0, state_valid=s["k"] > 0,
                             **s["args"])
        s["k"] += 1
        return {k: v for k, v in s["flat"].items() if k != "state"}
    spec, R = s["spec"], s["R"]
    if kind == "step":
        ctx.vmc_steps(0, prec, R, 1, spec.step, s["seed"], step0=s["k"], refresh=10, state=s["state"],
                      state_valid=True, nacc=s["nacc"], logpsi=s["lp"], sign=s["sg"], eloc=s["el"],
                      O=s["O"] if spec.n_params else None, dEL=s["dE"] if spec.n_params else None)
        s["k"] += 1
        return dict(R=R, state=s["state"], nacc=s["nacc"], logpsi=s["lp"], sign=s["sg"], eloc=s["el"], O=s["O"],
                    dEL=s["dE"])
    if kind == "eval":
        ctx.eval_walkers(0, prec, R, s["lp"], s["sg"], s["el"], grad=s["grad"],
                         O=s["O"] if spec.n_params else None, dEL=s["dE"] if spec.n_params else None,
                         state_out=s["state"])
        return dict(logpsi=s["lp"], sign=s["sg"], eloc=s["el"], grad=s["grad"], O=s["O"], dEL=s["dE"],
                    state=s["state"])
    if kind == "sweeps":
        ctx.vmc_steps(0, prec, R, case["sweeps"], spec.step, s["seed"], step0=s["k"], refresh=case["refresh"],
                      nacc=s["nacc"])
        s["k"] += case["sweeps"]
        return dict(R=R, nacc=s["nacc"])
    if kind == "dmc":
        W = case["walkers"]
        s["W"], s["E_T"], h = ctx.dmc_steps(0, prec, R, s["W"], case["steps"], 0.005, s["E_T"], W, s["seed"],
                                            step0=s["k"])
        s["k"] += case["steps"]
        return dict(R=R, W=s["W"], E_T=s["E_T"], **h)
    if kind == "forces":
        ctx.eval_nuclear_derivs(0, prec, R, s["lp"], s["sg"], s["el"], s["dlp"], s["dER"])
        return dict(logpsi=s["lp"], sign=s["sg"], eloc=s["el"], dlogpsi=s["dlp"], dEL=s["dER"])
    lp, el = autograd.evaluate(ctx, 0, spec, R, prec, params=s["p"], nuclei=s["X"])
    e = el.detach()
    loss = el.mean() + 2.0 * ((e - e.mean()) * lp).mean()  # its gradient is that of the VMC energy
    wanted = [t for t in (s["p"], s["X"]) if t.numel()]
    return dict(logpsi=lp.detach(), eloc=e, grads=torch.autograd.grad(loss, wanted))


# ---------------------------------------------------------------------------------------
# bytes and flops that no implementation can do without
# ---------------------------------------------------------------------------------------
def _counts(spec):
    """Flops per walker of a sweep, an evaluation, all parameter derivatives and all nucleus derivatives."""
    N, Nn, n = spec.N, spec.Nn, spec.n_up
    nnz = (spec.orb_coef != 0).sum(1)
    det = sorted(set(map(int, spec.inact)) | set(map(int, spec.pairs.ravel())) | set(map(int, spec.unp)))
    ev = sorted(set(det) | set(map(int, spec.kappa_kl[:, 0])))
    U = len({d for up, dn, _, _ in _terms(spec) for d in (("u",) + up, ("d",) + dn)})
    een = 23 * 12 if spec.een_on else 0
    pairs = N * (N - 1) // 2
    sweep = N * (3 * spec.M + nnz[det].sum() + (U / 2) * 2 * n + 0.5 * (U / 2) * 4 * n * n + (N + Nn) * 20 + N * Nn * een / 6)
    evaluate = N * (10 * spec.M + 2 * 5 * nnz[det].sum()) + U * 2 * n * n + pairs * 60 + N * Nn * 30 + pairs * Nn * een
    derivs = N * 10 * nnz[ev].sum() + U * 4 * n ** 3 + pairs * Nn * een + len(spec.kappa_kl) * 8 * n if spec.n_params else 0
    forces = pairs * Nn * een * 4 + N * nnz[det].sum() * 24 + Nn * U * n * n * 18
    return float(sweep), float(evaluate), float(derivs), float(forces), U * 2 * n ** 3


def work(case):
    b = 4 if case["precision"] == "mixed" else 8
    if case["kind"] == "lin":
        M, P = case["samples"], case["params"]
        return {"bytes": 2 * M * P * b + 8 * M * (2 if case["weights"] else 1) + 16 * P * P, "flops": 4.0 * M * P * P}
    if case["kind"] == "batch":
        specs, Ws = _workload(case)
        fl = by = 0.0
        for sp, W in zip(specs, Ws):
            sw, ev, de, _, lu = _counts(sp)
            fl += W * (sw + ev + de + lu)
            by += W * (48 * sp.N + 28 + 2 * b * sp.n_params)
        return {"bytes": by, "flops": fl}
    spec, W = _system(case["system"]), case["walkers"]
    sw, ev, de, fo, lu = _counts(spec)
    r, P = 24 * spec.N, spec.n_params
    state = 8 * (2 * spec.n_up ** 2) * max(1, spec.Nvb)
    by, fl = {"step": (2 * r + 2 * state + 24 + 2 * b * P, sw + ev + de + lu / 10),
              "eval": (2 * r + state + 24 + 2 * b * P, ev + de + lu),
              "sweeps": (2 * r, case.get("sweeps", 1) * sw + lu),
              "dmc": (2 * r * case.get("steps", 1), (case.get("steps", 1) + 1) * (ev + lu)),
              "forces": (r + 24 + 48 * spec.Nn, ev + lu + fo),
              "gradient": (r + 16, 2 * (ev + lu) + de + fo)}[case["kind"]]
    return {"bytes": float(W * by), "flops": float(W * fl)}


# ---------------------------------------------------------------------------------------
# 64-bit results
# ---------------------------------------------------------------------------------------
CART = {0: [(0, 0, 0)], 1: [(1, 0, 0), (0, 1, 0), (0, 0, 1)],
        2: [(2, 0, 0), (0, 2, 0), (0, 0, 2), (1, 1, 0), (1, 0, 1), (0, 1, 1)]}
EEN = [(p, k, l, (p - k - l) // 2) for p in range(2, 6) for k in range(p)
       for l in range((p - k if k else p - k - 2) + 1) if (p - k - l) % 2 == 0]


def _sorted_sign(v):
    inv = sum(1 for i, j in itertools.combinations(range(len(v)), 2) if v[i] > v[j])
    return tuple(sorted(v)), -1 if inv & 1 else 1


def _terms(spec):
    """(up orbitals, down orbitals, structure, sign) of every determinant of every structure."""
    out = []
    for I in range(spec.Nvb):
        ina = [int(x) for x in spec.inact[spec.inact_off[I]:spec.inact_off[I + 1]]]
        prs = [tuple(map(int, p)) for p in spec.pairs[spec.pair_off[I]:spec.pair_off[I + 1]]]
        unp = [int(x) for x in spec.unp[spec.unp_off[I]:spec.unp_off[I + 1]]]
        for flip in itertools.product(*[(0,) if i == j else (0, 1) for i, j in prs]):
            ops, sgn = [(o, sp) for o in ina for sp in (0, 1)], 1
            for (i, j), f in zip(prs, flip):
                ops += [(i, f), (j, 1 - f)]
                sgn = -sgn if f else sgn
            ops += [(o, 0) for o in unp]
            downs = 0
            for _, sp in ops:  # every up operator moves left of the down operators before it
                if sp:
                    downs += 1
                elif downs & 1:
                    sgn = -sgn
            up, su = _sorted_sign([o for o, sp in ops if not sp])
            dn, sd = _sorted_sign([o for o, sp in ops if sp])
            if len(set(up)) == len(up) and len(set(dn)) == len(dn):
                out.append((up, dn, I, sgn * su * sd))
    return out


def _een_basis():
    """Null space (reduced row echelon form, free columns in order) of the e-e-n cusp conditions."""
    rows = [[k if k and p - k == q else 0 for p, k, l, m in EEN] for q in range(1, 6)]
    rows += [[(l + m if k + m == q else 0) + (m if k + l + m == q else 0) for p, k, l, m in EEN] for q in range(7)]
    A, piv, r = np.array(rows, float), [], 0
    for c in range(len(EEN)):
        if r == len(A) or abs(A[r:, c]).max() < 1e-9:
            continue
        b = r + int(abs(A[r:, c]).argmax())
        A[[r, b]] = A[[b, r]]
        A[r] /= A[r, c]
        for i in range(len(A)):
            if i != r:
                A[i] -= A[i, c] * A[r]
        piv.append(c)
        r += 1
    free = [c for c in range(len(EEN)) if c not in piv]
    B = np.zeros((len(EEN), len(free)))
    for f, c in enumerate(free):
        B[c, f] = 1.0
        B[piv, f] = -A[:len(piv), c]
    return B


def _f64(x):
    return torch.tensor(np.ascontiguousarray(x), dtype=torch.float64, device=DEV)


class _Psi:
    """The trial wave function of a system in plain torch, in 64 bits."""

    def __init__(self, spec):
        self.spec = spec
        kind = spec.sh_kind if spec.sh_kind is not None else np.zeros(len(spec.sh_l), int)
        cen, zet, sla, cart, nrm = [], [], [], [], []
        dfac = lambda n: math.prod(range(n, 0, -2)) if n > 0 else 1
        for c, l, z, kd in zip(spec.sh_center, spec.sh_l, spec.sh_zeta, kind):
            l, z = int(l), float(z)
            for a in CART[l]:
                d = math.prod(dfac(2 * x - 1) for x in a)
                if kd:
                    nn = math.sqrt((2 * z) ** (2 * l + 3) * dfac(2 * l + 1) / (4 * math.pi * math.factorial(2 * l + 2) * d))
                else:
                    nn = (2 * z / math.pi) ** 0.75 * (4 * z) ** (l / 2) / math.sqrt(d) if z else 1.0
                cen.append(int(c)), zet.append(z), sla.append(float(kd)), cart.append(a), nrm.append(nn)
        self.cen = torch.tensor(cen, device=DEV)
        self.zet, self.sla, self.nrm = _f64(zet), _f64(sla) > 0, _f64(nrm)
        self.cart = torch.tensor(cart, device=DEV)
        self.C = _f64(spec.orb_coef)
        terms = _terms(spec)
        ups, dns = sorted({t[0] for t in terms}), sorted({t[1] for t in terms})
        self.cols = [torch.tensor(ups, device=DEV).reshape(len(ups), -1), torch.tensor(dns, device=DEV).reshape(len(dns), -1)]
        self.td = torch.tensor([(ups.index(t[0]), dns.index(t[1])) for t in terms], device=DEV)
        self.tI = torch.tensor([t[2] for t in terms], device=DEV)
        self.tsign = _f64([t[3] for t in terms])
        self.c_vb = _f64(spec.c_vb)
        self.Z, self.X = _f64(spec.nuc_Z), _f64(spec.nuc_xyz)
        self.elem = torch.tensor(np.asarray(spec.nuc_elem, np.int64), device=DEV)
        self.B = _f64(_een_basis())
        self.jas = (_f64(spec.jas_a), _f64(spec.jas_b), _f64(spec.theta()))
        up = torch.arange(spec.N, device=DEV) < spec.n_up
        self.b1 = torch.where(up[:, None] == up[None, :], spec.b1_par, spec.b1_anti).to(torch.float64)

    def orbitals(self, R, X, derivs):
        """phi [w, e, orbital], and its gradient [.., 3] and Laplacian."""
        d = R[:, :, None, :] - X[self.cen]
        r2 = (d * d).sum(-1)
        r = torch.where(self.sla, r2, 1.0).sqrt()
        e = self.nrm * torch.exp(-self.zet * torch.where(self.sla, r, r2))
        a = self.cart
        f0 = torch.where(a == 0, 1.0, torch.where(a == 1, d, d * d))
        P = f0.prod(-1)
        if not derivs:
            return (e * P) @ self.C.T, None, None
        f1 = torch.where(a == 0, 0.0, torch.where(a == 1, 1.0, 2 * d))
        oth = torch.stack([f0[..., 1] * f0[..., 2], f0[..., 0] * f0[..., 2], f0[..., 0] * f0[..., 1]], -1)
        t = torch.where(self.sla, self.zet / r, 2 * self.zet)
        l = a.sum(-1)
        base = torch.where(self.sla, self.zet ** 2 - 2 * self.zet * (l + 1) / r, 4 * self.zet ** 2 * r2 - self.zet * (6 + 4 * l))
        lapP = (torch.where(a == 2, 2.0, 0.0) * oth).sum(-1)
        g = e[..., None] * (f1 * oth - t[..., None] * d * P[..., None])
        return ((e * P) @ self.C.T, torch.einsum("wemd,om->weod", g, self.C), (e * (lapP + P * base)) @ self.C.T)

    def pade(self, r, a1, a, q):
        """f(R) = a1 R/(1 + a R) + sum q_p R^p, R = r/(1 + kappa r): f, f', f'' in r."""
        k = self.spec.kappa
        den = 1 / (1 + k * r)
        x, x1, x2 = r * den, den ** 2, -2 * k * den ** 3
        p = 1 / (1 + a * x)
        f = a1 * x * p + sum(q[n] * x ** (n + 2) for n in range(4))
        fx = a1 * p * p + sum((n + 2) * q[n] * x ** (n + 1) for n in range(4))
        fxx = -2 * a1 * a * p ** 3 + sum((n + 2) * (n + 1) * q[n] * x ** n for n in range(4))
        return f, fx * x1, fxx * x1 * x1 + fx * x2

    def radial(self, R, X, ja, jb):
        """e-n and e-e terms of ln J with gradient [w, e, 3] and Laplacian [w, e], and the potential."""
        N = self.spec.N
        dn = R[:, :, None, :] - X
        rn = (dn * dn).sum(-1).sqrt()
        eye = torch.eye(N, device=DEV, dtype=torch.bool)
        off = (~eye).to(torch.float64)
        de = R[:, :, None, :] - R[:, None, :, :]
        re = torch.where(eye, 1.0, (de * de).sum(-1)).sqrt()
        a = ja[self.elem]
        f, f1, f2 = self.pade(rn, a[:, 0], a[:, 1], [a[:, 2 + n] for n in range(4)])
        lnj, G, L = f.sum((1, 2)), ((f1 / rn)[..., None] * dn).sum(2), (f2 + 2 * f1 / rn).sum(2)
        f, f1, f2 = self.pade(re, self.b1, jb[1], [jb[2 + n] for n in range(4)])
        lnj = lnj + 0.5 * (f * off).sum((1, 2))
        G = G + ((f1 / re * off)[..., None] * de).sum(2)
        L = L + ((f2 + 2 * f1 / re) * off).sum(2)
        V = (off / re).sum((1, 2)) / 2 - (self.Z / rn).sum((1, 2))
        dd = (X[:, None] - X[None]) + torch.eye(len(X), device=DEV)[..., None]
        ZZ = self.Z[:, None] * self.Z[None] * (1 - torch.eye(len(X), device=DEV))
        return lnj, G, L, V + 0.5 * (ZZ / dd.norm(dim=-1)).sum()

    def een(self, R, X, derivs):
        """Every e-e-n term per (electron, nucleus): its share of ln J [w, e, a], gradient [w, 3, e, a] and
        Laplacian [w, e, a], without coefficient.  sum_{i<j} u^k (s_i^A s_j^B + s_i^B s_j^A) goes through the
        sums over the partners j of u_ij^k s_j^q, grad u_ij^k s_j^q and lap u_ij^k s_j^q."""
        k, N = self.spec.kappa, self.spec.N
        dn = R[:, :, None, :] - X
        rn = (dn * dn).sum(-1).sqrt()
        en = (dn / rn[..., None]).permute(0, 3, 1, 2)
        eye = torch.eye(N, device=DEV, dtype=torch.bool)
        off = (~eye).to(torch.float64)
        de = R[:, :, None, :] - R[:, None, :, :]
        re = torch.where(eye, 1.0, (de * de).sum(-1)).sqrt()
        ee = (de / re[..., None]).permute(0, 3, 1, 2)
        pw = lambda x, n: x ** n if n > 0 else torch.ones_like(x)
        d1 = lambda x, n: n * pw(x, n - 1)
        d2 = lambda x, n: n * (n - 1) * pw(x, n - 2) if n > 1 else torch.zeros_like(x)
        u, s = 1 / (1 + k * re), 1 / (1 + k * rn)
        u1, u2, s1, s2 = -k * u * u, 2 * k * k * u ** 3, -k * s * s, 2 * k * k * s ** 3
        sums = {}

        def partner(n, q):  # [w, 5, e, a]: value, gradient, Laplacian (value alone without derivs)
            if (n, q) not in sums:
                U = (pw(u, n) * off)[:, None]
                if derivs:
                    g = d1(u, n) * u1 * off
                    h = (d2(u, n) * u1 ** 2 + d1(u, n) * u2) * off + 2 / re * g
                    U = torch.cat([U, g[:, None] * ee, h[:, None]], 1)
                sums[n, q] = U @ pw(s, q)[:, None]
            return sums[n, q]

        for t, (_, n, l, m) in enumerate(EEN):
            val = grad = lap = 0.0
            for A, B in ((l + m, m), (m, l + m)):
                y = partner(n, B)
                val = val + 0.5 * pw(s, A) * y[:, 0]
                if derivs:
                    S1 = d1(s, A) * s1
                    S2 = d2(s, A) * s1 ** 2 + d1(s, A) * s2 + 2 / rn * S1
                    grad = grad + pw(s, A)[:, None] * y[:, 1:4] + (S1 * y[:, 0])[:, None] * en
                    lap = lap + pw(s, A) * y[:, 4] + S2 * y[:, 0] + 2 * S1 * (y[:, 1:4] * en).sum(1)
            yield t, val, grad, lap

    def jastrow(self, R, X, derivs=True):
        """ln J, its gradient [w, e, 3] and Laplacian [w, e], and the potential energy."""
        lnj, G, L, V = self.radial(R, X, *self.jas[:2])
        if self.spec.een_on:
            c = (self.B @ self.jas[2].T)[:, self.elem]  # [term, nucleus]
            for t, val, grad, lap in self.een(R, X, derivs):
                lnj = lnj + (val @ c[t]).sum(1)
                if derivs:
                    G, L = G + (grad @ c[t]).transpose(1, 2), L + lap @ c[t]
        return lnj, G, L, V

    def slater(self, phi):
        """Per spin: matrices [w, det, electron, slot], sign and ln|det|; then the structure sum."""
        n = self.spec.n_up
        sg, ln, As = [], [], []
        for sp, cols in enumerate(self.cols):
            ph = phi[:, :n] if sp == 0 else phi[:, n:]
            A = ph[:, :, cols].permute(0, 2, 1, 3)
            s, l = torch.linalg.slogdet(A) if cols.shape[1] else (phi.new_ones(A.shape[:2]), phi.new_zeros(A.shape[:2]))
            sg.append(s), ln.append(l), As.append(A)
        lt = ln[0][:, self.td[:, 0]] + ln[1][:, self.td[:, 1]]
        top = lt.max(1, keepdim=True).values
        D = self.tsign * sg[0][:, self.td[:, 0]] * sg[1][:, self.td[:, 1]] * torch.exp(lt - top)  # signed, per term
        Phi = (D * self.c_vb[self.tI]).sum(1)
        return As, D / Phi[:, None], top[:, 0] + Phi.abs().log(), Phi.sign()

    def value(self, R):
        lnj = self.jastrow(R, self.X, False)[0]
        return lnj + self.slater(self.orbitals(R, self.X, False)[0])[2]

    def local(self, R, X=None, derivs=False):
        """ln|Psi|, sign, E_L, gradient; with derivs also O and dE_L/dp."""
        X = self.X if X is None else X
        n, sp = self.spec.n_up, self.spec
        lnj, G, LJ, V = self.jastrow(R, X)
        phi, gr, lap = self.orbitals(R, X, True)
        L = lap + 2 * torch.einsum("wed,weod->weo", G, gr)
        As, D, lnPhi, sign = self.slater(phi)
        wt = D * self.c_vb[self.tI]
        inv, tr, Wu, grad = [], [], [], []
        for q, cols in enumerate(self.cols):
            sl = slice(0, n) if q == 0 else slice(n, sp.N)
            B = torch.linalg.inv(As[q]) if cols.shape[1] else As[q].transpose(2, 3)
            Lq = L[:, sl][:, :, cols].permute(0, 2, 1, 3)
            tr.append(torch.einsum("wuoe,wueo->wu", B, Lq))
            Wu.append(wt.new_zeros(len(wt), len(cols)).index_add(1, self.td[:, q], wt))
            grad.append(torch.einsum("wu,wuoe,weuod->wed", Wu[q], B, gr[:, sl][:, :, cols]))
            inv.append(B)
        tt = tr[0][:, self.td[:, 0]] + tr[1][:, self.td[:, 1]]
        K = (wt * tt).sum(1)
        grad = G + torch.cat(grad, 1)
        eloc = -0.5 * (LJ.sum(1) + (G * G).sum((1, 2)) + K) + V
        out = [lnj + lnPhi, sign, eloc, grad]
        if not derivs:
            return out
        O, dE = [], []
        for I in map(int, sp.cparam):
            m = (self.tI == I).to(torch.float64)
            o = (D * m).sum(1)
            O.append(o), dE.append(-0.5 * ((D * m * tt).sum(1) - o * K))
        if sp.jas_param:
            ja, jb, _ = self.jas
            basis = [(0, i) for e in range(sp.n_elem) for i in range(6 * e + 1, 6 * e + 6)] + [(1, i) for i in range(1, 6)]
            for which, i in basis:
                tan = [torch.zeros_like(x) for x in (ja, jb)]
                tan[which].view(-1)[i] = 1.0
                _, (o, g1, l1, _) = torch.func.jvp(lambda *j: self.radial(R, X, *j), (ja, jb), tuple(tan))
                O.append(o), dE.append(-0.5 * (l1.sum(1) + 2 * (g1 * grad).sum((1, 2))))
            if sp.een_on:
                raw = [(val.sum(1), -0.5 * (lp.sum(1) + 2 * torch.einsum("wdia,wid->wa", g1, grad)))
                       for _, val, g1, lp in self.een(R, X, True)]
                for E in range(sp.n_elem):
                    mine = (self.elem == E).to(torch.float64)
                    for out_, k in ((O, 0), (dE, 1)):
                        out_ += list((torch.stack([x[k] @ mine for x in raw], 1) @ self.B).T)
        if len(sp.kappa_kl):
            acc = [phi.new_zeros(len(phi), len(sp.kappa_kl)) for _ in range(2)]
            for q, cols in enumerate(self.cols):
                sl = slice(0, n) if q == 0 else slice(n, sp.N)
                B, ph, Lp = inv[q], phi[:, None, sl], L[:, None, sl]
                Tu = wt.new_zeros(len(wt), len(cols)).index_add(1, self.td[:, q], wt * tt)
                x = B @ ph  # [w, det, slot, orbital]
                y = B @ Lp - B @ L[:, sl][:, :, cols].permute(0, 2, 1, 3) @ x
                has = [c.tolist() for c in cols]
                hit = [(j, u, h.index(l), k) for j, (k, l) in enumerate(sp.kappa_kl.tolist()) for u, h in enumerate(has)
                       if l in h and k not in h]
                j, u, o, k = torch.tensor(hit, device=DEV).reshape(-1, 4).T
                acc[0].index_add_(1, j, Wu[q][:, u] * x[:, u, o, k])
                acc[1].index_add_(1, j, Tu[:, u] * x[:, u, o, k] + Wu[q][:, u] * y[:, u, o, k])
            O += list(acc[0].T)
            dE += list((-0.5 * (acc[1] - acc[0] * K[:, None])).T)
        e = R.new_zeros(len(R), 0)
        return out + [torch.stack(O, 1) if O else e, torch.stack(dE, 1) if dE else e]

    def forces(self, R):
        dl, dE = [], []
        for i in range(self.X.numel()):
            t = torch.zeros_like(self.X)
            t.view(-1)[i] = 1.0
            _, (l, e) = torch.func.jvp(lambda x: tuple(self.local(R, x)[k] for k in (0, 2)), (self.X,), (t,))
            dl.append(l), dE.append(e)
        return [torch.stack(v, 1).reshape(len(R), -1, 3) for v in (dl, dE)]

    def sweep(self, R, seed, step0, nsweeps, step, tag=0, first=0):
        R = R.clone()
        w = torch.arange(first, first + len(R), device=DEV)
        old = self.value(R)
        for k in range(nsweeps):
            for e in range(self.spec.N):
                u = torch.stack(_uniforms(w, step0 + k, e, tag, 0, seed) + _uniforms(w, step0 + k, e, tag, 1, seed), 1)
                new = R.clone()
                new[:, e] = R[:, e] + step * (2 * u[:, :3] - 1)
                v = self.value(new)
                ok = u[:, 3] < torch.exp(2 * (v - old))
                R, old = torch.where(ok[:, None, None], new, R), torch.where(ok, v, old)
        return R


def _uniforms(w, step, slot, tag, purpose, seed):
    """Philox4x32-10, counter (walker, step, slot, tag << 8 | purpose), key = seed: two uniforms."""
    m32 = 0xFFFFFFFF
    c = [w, torch.full_like(w, step), torch.full_like(w, slot), torch.full_like(w, (tag << 8) | purpose)]
    k = [seed & m32, (seed >> 32) & m32]

    def mul(a, x):  # 64-bit product in halves, without overflow of signed integers
        lo, hi = a * (x & 0xFFFF), a * (x >> 16)
        s = lo + ((hi & 0xFFFF) << 16)
        return (hi >> 16) + (s >> 32), s & m32

    for _ in range(10):
        h0, l0 = mul(0xD2511F53, c[0])
        h1, l1 = mul(0xCD9E8D57, c[2])
        c = [h1 ^ c[1] ^ k[0], l1, h0 ^ c[3] ^ k[1], l0]
        k = [(k[0] + 0x9E3779B9) & m32, (k[1] + 0xBB67AE85) & m32]
    return [((hi << 21) | (lo >> 11)).to(torch.float64) * 2.0 ** -53 for lo, hi in ((c[0], c[1]), (c[2], c[3]))]


def _chunked(f, R, size):
    parts = [f(R[i:i + size], i) for i in range(0, len(R), size)]
    return [torch.cat(p) for p in zip(*parts)]


def exact(case, seed):
    if case["kind"] == "lin":
        O, dE, E, w = _lin_inputs(case, seed)
        w = torch.ones_like(E) if w is None else w
        sw = w.sum()
        P = case["params"]
        mu = sum((w[i:j, None] * O[i:j].double()).sum(0) for i, j in _ranges(len(E))) / sw
        S, H = _zeros(P, P), _zeros(P, P)
        oe, de = _zeros(P), _zeros(P)
        for i, j in _ranges(len(E)):
            o, d, e, q = O[i:j].double() - mu, dE[i:j].double(), E[i:j], w[i:j, None]
            S += (q * o).T @ o
            H += (q * o).T @ (e[:, None] * o + d)
            oe += (q * o * e[:, None]).sum(0)
            de += (q * d).sum(0)
        return dict(E0=((w * E).sum() / sw).reshape(1), gL=2 * oe / sw, gR=2 * (oe + de) / sw, S=S / sw, H=H / sw)
    if case["kind"] == "dmc" or case.get("system") == "dmc48":
        # populations follow from decisions of whole runs; 48 electrons take too long in plain torch
        return None
    if case["kind"] == "batch":
        specs, Ws = _workload(case)
        flat = {n: [] for n in ("R", "logpsi", "sign", "eloc", "O", "dEL")}
        for k, sp in enumerate(specs):
            psi = _Psi(sp)
            R = psi.sweep(_walkers(sp, Ws[k], seed * 1000 + k), seed, 0, 1, 0.3, tag=k)
            lp, sg, el, _, O, dEL = _chunked(lambda r, i: psi.local(r, derivs=True), R, 512)
            for n, v in zip(flat, (R, lp, sg, el, O, dEL)):
                flat[n].append(v.reshape(-1))
        return dict({n: torch.cat(v) for n, v in flat.items()}, nacc=None)
    spec = _system(case["system"])
    psi, R = _Psi(spec), _walkers(spec, case["walkers"], seed)
    if case["kind"] in ("step", "sweeps"):
        ns, k0 = (1, 7) if case["kind"] == "step" else (case["sweeps"], 0)
        R, = _chunked(lambda r, i: [psi.sweep(r, seed, k0, ns, spec.step, first=i)], R, 4096)
        if case["kind"] == "sweeps":
            return dict(R=R, nacc=None)
    if case["kind"] == "forces":
        lp, sg, el, _ = _chunked(lambda r, i: psi.local(r), R, 1024)
        dl, dE = _chunked(lambda r, i: psi.forces(r), R, 512)
        return dict(logpsi=lp, sign=sg, eloc=el, dlogpsi=dl, dEL=dE)
    lp, sg, el, grad, O, dEL = _chunked(lambda r, i: psi.local(r, derivs=True), R, 1024)
    if case["kind"] == "gradient":
        dl, dE = _chunked(lambda r, i: psi.forces(r), R, 512)
        a = 2 * (el - el.mean()) / len(el)
        grads = [torch.einsum("w,w...->...", a, o) + d.mean(0) for o, d in ((O, dEL), (dl, dE)) if o.numel()]
        return dict(logpsi=lp, eloc=el, grads=grads)
    if case["kind"] == "eval":
        return dict(logpsi=lp, sign=sg, eloc=el, grad=grad, O=O, dEL=dEL, state=None)
    return dict(R=R, state=None, nacc=None, logpsi=lp, sign=sg, eloc=el, O=O, dEL=dEL)


def _ranges(n, size=1 << 16):
    return [(i, min(n, i + size)) for i in range(0, n, size)]
