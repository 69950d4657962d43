"""What users of the library have it compute: single applies, time evolution, stationary
states, spectra and a training gradient of the warm-start network, through the Python
binding, with the inputs made from a seed and the same results worked out in plain torch.

Families of cases (``kind``):

* ``apply``    y = M x on random ADO vectors (a user's own integrator or eigensolver);
* ``evolve``   RK4 in place, from a pure initial state or continuing a run;
* ``steady``   stationary states, one parameter set or a sweep of sets of uneven depth;
* ``spectrum`` densities of states, all frequencies from the shift-invariant solver;
* ``mlp``      loss gradient of the learned warm start on one batch.

Every model is one of the package's own workloads: the spin-boson model (one Drude-Lorentz
bath, 3 exponents), the single-impurity Anderson model (two leads, 24 exponents with two Pade
poles, 56 with six), the charge-cavity model (d = 24) and random dense operators. Exponents
come from the formulas below, as from a user who brings their own, and serve both sides.
"""
from __future__ import annotations

import itertools
import math

import numpy as np
import torch

import paper_2306_07522_gb300 as heom

DEV = "cuda"


# ------------------------------------------------------------------ the cases
def listed():
    return [
        # transient of the smallest model: 35 ADOs of 2 x 2, t = 10 in steps of 0.01, populations
        # saved every 10 steps; almost no arithmetic, so launches and latency are what counts
        dict(name="evolve_spin_boson_f64", kind="evolve", model="spin_boson", tier=4, sets=1,
             batch=1, dtype="c128", steps=1000, save=10),
        # charge-cavity dynamics in single precision: 790 ADOs of 24 x 24, one column, t = 2
        dict(name="evolve_cavity_f32", kind="evolve", model="cavity", tier=2, sets=1, batch=1,
             dtype="c64", steps=200, save=20),
        # transients over a bias sweep of 37 parameter sets (an odd number), double precision
        dict(name="evolve_sweep_f64", kind="evolve", model="siam", tier=2, sets=37, batch=37,
             dtype="c128", steps=50, save=10),
        # one apply on many columns of one model: 2,325 ADOs x 1,024 columns (305 MB a vector)
        dict(name="apply_wide_f32", kind="apply", model="siam", tier=3, sets=1, batch=1024,
             dtype="c64"),
        # the 56-exponent Anderson model at four tiers: 396,607 ADOs, one column
        dict(name="apply_large_f32", kind="apply", model="siam56", tier=4, sets=1, batch=1,
             dtype="c64"),
        dict(name="apply_large_f64", kind="apply", model="siam56", tier=4, sets=1, batch=1,
             dtype="c128"),
        # operators without zeros (user-supplied): d = 24, 222 ADOs, 64 columns
        dict(name="apply_dense_f32", kind="apply", model="dense24", tier=2, sets=1, batch=64,
             dtype="c64"),
        # one stationary state in double precision: 2,325 ADOs, one column
        dict(name="steady_one_f64", kind="steady", model="siam", tier=3, sets=1, prec="fp64"),
        # stationary states of a parameter sweep in mixed precision, the sets truncated at
        # tiers 2, 3 and 4 of one 12,951-ADO hierarchy (the batched-spectra workload's first half)
        dict(name="steady_sweep_mixed", kind="steady", model="siam", tier=4, sets=32,
             prec="mixed"),
        # density of states of one model at 1,000 frequencies
        dict(name="spectrum_one", kind="spectrum", model="siam", tier=3, sets=1, omegas=1000),
        # densities of states of a sweep of uneven depth (the batched-spectra workload's second
        # half, on a quarter of its sets and frequencies)
        dict(name="spectrum_sweep", kind="spectrum", model="siam", tier=4, sets=16, omegas=1024),
        # gradient of the warm-start network (5 -> 3 x 256 -> 784) on a batch of 4,096 states
        dict(name="mlp_gradient", kind="mlp", hidden=256, layers=3, outputs=784, batch=4096),
    ]


def _logint(rng, lo, hi):
    return max(lo, min(hi, int(round(math.exp(rng.uniform(math.log(lo), math.log(hi)))))))


def draw(rng):
    """One more case: a family at random, then its sizes over the range the listed ones span."""
    kind = rng.choice(["evolve", "evolve", "apply", "apply", "apply", "steady", "spectrum", "mlp"])
    if kind == "evolve":
        model = rng.choice(["spin_boson", "siam", "cavity"])
        if model == "spin_boson":  # 10 to 165 ADOs
            return dict(kind=kind, model=model, tier=rng.randint(2, 8), sets=1, batch=1,
                        dtype=rng.choice(["c128", "c64"]), steps=_logint(rng, 100, 1000), save=10)
        if model == "siam":  # 25 to 2,325 ADOs, a sweep of up to 64 sets
            tier = rng.randint(1, 3)
            sets = _logint(rng, 1, 64 if tier < 3 else 8)
            return dict(kind=kind, model=model, tier=tier, sets=sets, batch=sets * rng.randint(1, 2),
                        dtype=rng.choice(["c128", "c64"]), steps=_logint(rng, 10, 50), save=5)
        return dict(kind=kind, model=model, tier=rng.randint(1, 2), sets=1, batch=rng.randint(1, 3),
                    dtype="c64", steps=_logint(rng, 20, 150), save=10)
    if kind == "apply":
        model = rng.choice(["siam", "siam", "siam56", "cavity", "dense16", "dense24"])
        dtype = rng.choice(["c64", "c64", "c128"])
        if model == "siam":  # odd and even widths, one set or one per column
            tier = rng.randint(1, 4)
            batch = _logint(rng, 1, 1024 if tier < 4 else 96)
            if dtype == "c128":
                batch = min(batch, 200 if tier < 4 else 40)
            sets = batch if rng.random() < 0.25 else 1
            return dict(kind=kind, model=model, tier=tier, sets=sets, batch=batch, dtype=dtype)
        if model == "siam56":  # 57 to 396,607 ADOs
            return dict(kind=kind, model=model, tier=rng.randint(1, 4), sets=1, batch=1, dtype=dtype)
        if model == "cavity":
            return dict(kind=kind, model=model, tier=rng.randint(1, 2), sets=1,
                        batch=_logint(rng, 1, 64), dtype="c64")
        return dict(kind=kind, model=model, tier=rng.randint(1, 2), sets=1, batch=_logint(rng, 1, 64),
                    dtype="c64")
    if kind == "steady":
        if rng.random() < 0.5:
            return dict(kind=kind, model="siam", tier=rng.randint(2, 3), sets=1,
                        prec=rng.choice(["fp64", "mixed"]))
        return dict(kind=kind, model="siam", tier=rng.randint(2, 4), sets=_logint(rng, 2, 32),
                    prec="mixed")
    if kind == "spectrum":
        tier = rng.randint(2, 4)
        sets = _logint(rng, 1, 16) if rng.random() < 0.6 else 1
        return dict(kind=kind, model="siam", tier=tier, sets=sets, omegas=_logint(rng, 64, 1024))
    return dict(kind=kind, hidden=_logint(rng, 64, 256), layers=rng.randint(1, 3),
                outputs=_logint(rng, 100, 784), batch=_logint(rng, 64, 4096))


# ------------------------------------------------------------------ models and exponents
def _pade(n, fermi):
    """[N-1/N] Pade constants kappa, zeta of the Fermi (Bose) function (Hu, Xu, Yan 2010)."""
    b = (lambda m: 2.0 * m - 1.0) if fermi else (lambda m: 2.0 * m + 1.0)

    def roots(size, shift):
        t = np.zeros((size, size))
        for m in range(1, size):
            t[m - 1, m] = t[m, m - 1] = 1.0 / math.sqrt(b(m + shift) * b(m + shift + 1))
        lam = np.linalg.eigvalsh(t)
        return 2.0 / np.sort(lam[lam > 1e-12])[::-1]

    zeta = roots(2 * n, 0)
    zt = roots(2 * n - 1, 1) if n > 1 else np.zeros(0)
    kappa = np.array([0.5 * n * b(n + 1) * np.prod(zt ** 2 - zeta[j] ** 2) /
                      np.prod(np.delete(zeta, j) ** 2 - zeta[j] ** 2) for j in range(n)])
    return kappa, zeta


def _lead(Gamma, W, mu, kT, poles):
    """Exponents of a Lorentzian lead: nu = +1 then nu = -1, as coefficient and rate lists."""
    kappa, zeta = _pade(poles, True)
    x = 1j * W / kT
    fermi = 0.5 - np.sum(2.0 * kappa * x / (x * x + zeta * zeta))
    coef, rate = [], []
    for nu in (1, -1):
        coef += [0.5 * Gamma * W * fermi]
        rate += [W - nu * 1j * mu]
        coef += list(-1j * kappa * kT * Gamma * W ** 2 / (W ** 2 - (zeta * kT) ** 2))
        rate += list(zeta * kT - nu * 1j * mu)
    return np.array(coef), np.array(rate)


def _drude(lam, W, kT, poles, matsubara):
    if matsubara:
        kappa, zeta = np.ones(poles), 2 * np.pi * np.arange(1, poles + 1)
    else:
        kappa, zeta = _pade(poles, False)
    zk = zeta * kT
    coef = np.concatenate([[lam * W * (1.0 / math.tan(W / (2.0 * kT)) - 1j)],
                           -2.0 * kappa * kT * 2.0 * lam * W * zk / (W ** 2 - zk ** 2)])
    return coef.astype(complex), np.concatenate([[W], zk]).astype(complex)


_SM = np.array([[0, 1], [0, 0]], dtype=complex)  # |1> -> |0>
_SZ = np.diag([1.0, -1.0]).astype(complex)
_SX = np.array([[0, 1], [1, 0]], dtype=complex)


def _fermion_bath(op, coef, rate):
    h = len(coef) // 2
    return dict(kind="F", op=op, coef=coef, rate=rate, nu=np.array([1] * h + [-1] * h, np.int32),
                partner=np.array(list(range(h, 2 * h)) + list(range(h)), np.int32))


def _problems(case, seed, parity):
    """One raw problem per parameter set (same structure, parameters drawn from the seed) and
    each set's fermionic tier."""
    rng = np.random.default_rng([7522, seed])
    model, out = case["model"], []
    if model.startswith("dense"):
        d = int(model[5:])
        z = lambda *s: rng.standard_normal(s) + 1j * rng.standard_normal(s)  # noqa: E731
        H, V = z(d, d), z(d, d)
        baths = [dict(kind="RI", op=0.5 * (V + V.conj().T), coef=0.3 * z(2),
                      rate=rng.uniform(0.2, 2.0, 2) + 1j * rng.uniform(-0.5, 0.5, 2)),
                 _fermion_bath(0.5 * z(d, d), 0.3 * z(8),
                               rng.uniform(0.2, 2.0, 8) + 1j * rng.uniform(-0.5, 0.5, 8))]
        return [dict(d=d, H=0.5 * (H + H.conj().T), baths=baths, tier_b=case["tier"],
                     tier_f=case["tier"], parity=parity)], [case["tier"]]
    # parameter draws; kT keeps away from 0.68 .. 0.87, where two exponents of these leads meet
    tiers = sorted((int(t) for t in rng.integers(min(2, case["tier"]), case["tier"] + 1, case["sets"])), reverse=True)
    tiers[0] = case["tier"]
    if case["kind"] not in ("steady", "spectrum"):
        tiers = [case["tier"]] * case["sets"]
    for s in range(case["sets"]):
        U, kT, mu = rng.uniform(4.0, 12.0), rng.uniform(0.35, 0.6), rng.uniform(0.0, 2.0)
        if model == "spin_boson":
            coef, rate = _drude(rng.uniform(0.05, 0.15), 0.5, kT, 2, True)
            out.append(dict(d=2, H=0.5 * rng.uniform(0.8, 1.2) * _SX, parity=parity,
                            baths=[dict(kind="RI", op=_SZ, coef=coef, rate=rate)],
                            tier_b=case["tier"], tier_f=0))
        elif model == "cavity":
            a1 = np.diag(np.sqrt(np.arange(1.0, 12.0)), 1).astype(complex)
            dop, a = np.kron(_SM, np.eye(12)), np.kron(np.eye(2), a1)
            nd, x = dop.conj().T @ dop, a + a.conj().T
            H = -3.0 * nd + a.conj().T @ a + rng.uniform(0.3, 0.5) * nd @ x
            coef, rate = _drude(0.01, 0.2, 0.5, 2, False)
            baths = [dict(kind="RI", op=x, coef=coef, rate=rate)]
            baths += [_fermion_bath(dop, *_lead(1.0, 10.0, m, 0.5, 2)) for m in (1.0 + mu, -1.0 - mu)]
            out.append(dict(d=24, H=H, baths=baths, tier_b=case["tier"], tier_f=case["tier"],
                            parity=parity))
        else:
            up, dn = np.kron(_SM, np.eye(2)), np.kron(_SZ, _SM)
            nu, nd = up.conj().T @ up, dn.conj().T @ dn
            gamma, poles = (1.0, 6) if model == "siam56" else (2.0, 2)
            baths = [_fermion_bath(op, *_lead(gamma, 10.0, m, kT, poles))
                     for m in (mu, -mu) for op in (up, dn)]
            out.append(dict(d=4, H=-5.0 * (nu + nd) + U * nu @ nd, baths=baths, tier_b=0,
                            tier_f=case["tier"], parity=parity))
    return out, tiers


def _hierarchy(case, seed, parity=1):
    """The library's hierarchy holding every parameter set of the case."""
    probs, tiers = _problems(case, seed, parity)
    h = heom.build_hierarchy(probs[0])
    if len(probs) > 1:
        heom.set_params(h, np.array([p["H"] for p in probs]),
                        np.array([np.concatenate([b["coef"] for b in p["baths"]]) for p in probs]),
                        np.array([np.concatenate([b["rate"] for b in p["baths"]]) for p in probs]))
        if min(tiers) < max(tiers):
            heom.set_truncation(h, [0] * len(probs), tiers)
    return h, probs


# ------------------------------------------------------------------ prepare and run
_DTYPE = {"c64": torch.complex64, "c128": torch.complex128}
_OMEGA = 20.0  # spectra run over [-20, 20]
_TOL = 1e-10   # both solvers' tolerance


def _vector(case, seed, shape):
    gen = torch.Generator(device=DEV).manual_seed(2306 + seed)
    return torch.randn(shape, dtype=torch.complex128, device=DEV, generator=gen).to(_DTYPE[case["dtype"]])


def _initial(case, seed, n_ado, d):
    """A random pure state in the reduced density matrix of every column, other ADOs zero."""
    gen = torch.Generator(device=DEV).manual_seed(99 + seed)
    psi = torch.randn((d, case["batch"]), dtype=torch.complex128, device=DEV, generator=gen)
    if case["model"] == "cavity":  # amplitudes fall off towards the Fock cutoff
        psi *= 0.5 ** torch.arange(12, device=DEV, dtype=torch.float64).repeat(2)[:, None]
    psi /= psi.norm(dim=0)
    x = torch.zeros((n_ado, d, d, case["batch"]), dtype=torch.complex128, device=DEV)
    x[0] = psi[:, None, :] * psi[None, :, :].conj()
    return x.to(_DTYPE[case["dtype"]])


def _shaped(case, x):
    return x[..., 0].contiguous() if case["batch"] == 1 else x


def _mlp_arrays(case, seed):
    rng = np.random.default_rng([11, seed])
    w = [5] + [case["hidden"]] * case["layers"] + [case["outputs"]]
    params = []
    for i, o in zip(w[:-1], w[1:]):
        params += [rng.uniform(-1, 1, i * o) * math.sqrt(6.0 / (i + o)), 0.1 * rng.standard_normal(o)]
    n = case["batch"]
    x = np.stack([rng.uniform(0, 12, n), rng.uniform(-8, -2, n), rng.uniform(1, 3, n),
                  rng.uniform(0.2, 1, n), rng.uniform(0, 3, n)], axis=1)
    t = 0.3 * rng.standard_normal((n, w[-1])) + np.sin(x @ rng.standard_normal((5, w[-1])))
    f32 = lambda a: np.asarray(a, np.float32)  # noqa: E731
    norms = (f32(x.mean(0)), f32(x.std(0)), f32(t.mean(0)), f32(t.std(0)))
    return w, f32(np.concatenate(params)), f32(x), f32(t), norms


def prepare(case, seed):
    kind = case["kind"]
    if kind == "mlp":
        w, params, x, t, norms = _mlp_arrays(case, seed)
        net = heom.Mlp(w, seed=seed)
        net.set_params(params)
        net.set_standardisation(*norms)
        return dict(kind=kind, net=net, x=torch.from_numpy(x).to(DEV), t=torch.from_numpy(t).to(DEV))
    h, probs = _hierarchy(case, seed)
    if kind == "apply":
        x = _shaped(case, _vector(case, seed, (h.n_ado, h.d, h.d, case["batch"])))
        return dict(kind=kind, h=h, x=x, y=torch.empty_like(x))
    if kind == "evolve":
        return dict(kind=kind, h=h, x=_shaped(case, _initial(case, seed, h.n_ado, h.d)),
                    steps=case["steps"], save=case["save"])
    shape = (h.n_ado, h.d, h.d) + ((case["sets"],) if case["sets"] > 1 else ())
    x = torch.zeros(shape, dtype=torch.complex128, device=DEV)
    if kind == "steady":
        return dict(kind=kind, h=h, x=x, prec=heom.FP64 if case["prec"] == "fp64" else heom.MIXED)
    # a spectrum starts from the even sector's stationary states
    heom.steady(h, x, tol=_TOL, max_iter=4000, prec=heom.MIXED if case["sets"] > 1 else heom.FP64)
    odd, _ = _hierarchy(case, seed, -1)
    return dict(kind=kind, h=odd, x=x, op=np.kron(_SM, np.eye(2)),
                omega=np.linspace(-_OMEGA, _OMEGA, case["omegas"]))


def run(state):
    kind = state["kind"]
    if kind == "apply":
        return heom.apply(state["h"], state["x"], state["y"])
    if kind == "evolve":
        traj = heom.evolve(state["h"], state["x"], 0.01, state["steps"], state["save"])
        return {"traj": traj, "ados": state["x"]}
    if kind == "steady":
        heom.steady(state["h"], state["x"], tol=_TOL, max_iter=4000, prec=state["prec"])
        return state["x"]
    if kind == "spectrum":
        # max_iter bounds the Krylov basis (12,951 ADOs x 32 columns: 212 MB a step)
        A, _, _ = heom.spectrum(state["h"], state["x"], state["op"], state["omega"], tol=_TOL,
                                max_iter=240, prec=heom.SHIFTED)
        return A
    grad, loss = state["net"].gradients(state["x"], state["t"])
    return {"grad": grad, "loss": loss}


# ------------------------------------------------------------------ the work of one pass
def _counts(case):
    """ADOs and non-zero coefficients of M (all sets' structures are the same)."""
    prob = _problems(dict(case, sets=1), 0, 1)[0][0]
    d = prob["d"]
    kb = sum(len(b["coef"]) for b in prob["baths"] if b["kind"] != "F")
    kf = sum(len(b["coef"]) for b in prob["baths"] if b["kind"] == "F")
    nb = math.comb(kb + prob["tier_b"], prob["tier_b"])
    nf = sum(math.comb(kf, n) for n in range(min(prob["tier_f"], kf) + 1))
    # every coupling appears twice, as the raising of one ADO and the lowering of the other
    eb = sum(math.comb(kb + t - 1, t) * kb for t in range(prob["tier_b"])) if kb else 0
    ef = sum(math.comb(kf, n) * (kf - n) for n in range(min(prob["tier_f"], kf)))
    nnz = lambda k: np.mean([np.count_nonzero(b["op"]) for b in prob["baths"] if (b["kind"] == "F") == k])  # noqa: E731
    terms = 2 * 2 * d * ((nnz(False) * eb * nf if kb else 0) + (nnz(True) * ef * nb if kf else 0))
    hn = np.count_nonzero(prob["H"] - np.diag(np.diag(prob["H"])))
    return nb * nf, d, terms + nb * nf * (d * d + 2 * d * hn)


def work(case):
    if case["kind"] == "mlp":
        w = [5] + [case["hidden"]] * case["layers"] + [case["outputs"]]
        n = sum(i * o + o for i, o in zip(w[:-1], w[1:]))
        # forward and weight gradients of every layer, input gradients of all but the first
        mac = 3 * sum(i * o for i, o in zip(w[:-1], w[1:])) - w[0] * w[1]
        return {"bytes": 4 * (2 * n + case["batch"] * (w[0] + w[-1])), "flops": 2 * mac * case["batch"]}
    N, d, terms = _counts(case)
    if case["kind"] == "apply":
        s = 8 if case["dtype"] == "c64" else 16
        return {"bytes": 2 * N * d * d * case["batch"] * s, "flops": 8 * terms * case["batch"]}
    if case["kind"] == "evolve":
        s = 8 if case["dtype"] == "c64" else 16
        saves = case["steps"] // case["save"] + 1
        return {"bytes": (2 * N + saves) * d * d * case["batch"] * s,
                "flops": 4 * case["steps"] * 8 * terms * case["batch"]}
    # Krylov solvers: at least 50 applies to 1e-10, each reading and writing a vector (FP64);
    # a spectrum's basis of 50 vectors is read once per step for its projections
    cols = case["sets"] * (2 if case["kind"] == "spectrum" else 1)
    vec = N * d * d * cols * 16
    passes = 50 * 2 if case["kind"] == "steady" else 50 * 2 + 50 * 50 / 2
    return {"bytes": passes * vec, "flops": 50 * 8 * terms * cols}


# ------------------------------------------------------------------ the same in plain torch
def _ado_tables(prob):
    """Bosonic occupations, fermionic subsets (as bit masks) and tier-ordered ADO indices."""
    kb = sum(len(b["coef"]) for b in prob["baths"] if b["kind"] != "F")
    kf = sum(len(b["coef"]) for b in prob["baths"] if b["kind"] == "F")
    bos = []
    for t in range(prob["tier_b"] + 1 if kb else 1):
        level = [m for m in itertools.product(range(t, -1, -1), repeat=kb) if sum(m) == t]
        bos += sorted(level, reverse=True)
    one = np.uint64(1)
    fer = [np.zeros(1, np.uint64)]
    for n in range(1, min(prob["tier_f"], kf) + 1):
        idx = np.fromiter(itertools.chain.from_iterable(itertools.combinations(range(kf), n)),
                          np.uint64).reshape(-1, n)
        fer.append(np.bitwise_or.reduce(one << idx, axis=1))
    return np.array(bos, np.int64).reshape(len(bos), kb), np.concatenate(fer)


def _matrix(prob):
    """M of Eq. HEOM as (rows, cols, values), ADO blocks row-major, for one raw problem."""
    d, p = prob["d"], prob["parity"]
    bos, fer = _ado_tables(prob)
    nb, nf = len(bos), len(fer)
    n_f = np.array([bin(int(m)).count("1") for m in fer])
    order = np.argsort(fer)
    locate = lambda m: order[np.searchsorted(fer, m, sorter=order)]  # noqa: E731
    bos_at = {tuple(m): i for i, m in enumerate(bos)}
    rows, cols, vals = [], [], []
    e = np.arange(d)

    def couple(i, j, left, right, O):
        """(M X)_i += left O X_j + right X_j O for arrays of ADO pairs i, j and factors."""
        for r, l in zip(*np.nonzero(O)):
            for a, b, f in ((r * d + e, l * d + e, left), (e * d + l, e * d + r, right)):
                rows.append((i[:, None] * d * d + a).ravel())
                cols.append((j[:, None] * d * d + b).ravel())
                vals.append(np.repeat(f * O[r, l], d))

    kb = 0
    for b in (b for b in prob["baths"] if b["kind"] != "F"):
        for c, _ in zip(b["coef"], b["rate"]):
            up = [(i, bos_at[tuple(m + (np.arange(len(m)) == kb))], m[kb] + 1) for i, m in enumerate(bos)
                  if tuple(m + (np.arange(len(m)) == kb)) in bos_at]
            lo, hi, cnt = (np.array(v) for v in zip(*up))
            f = np.arange(nf)
            i, j = (lo[:, None] * nf + f).ravel(), (hi[:, None] * nf + f).ravel()
            couple(i, j, np.full(len(i), -1j), np.full(len(i), 1j), b["op"])       # raised
            m = np.repeat(cnt, nf)
            couple(j, i, -1j * m * c, 1j * m * np.conj(c), b["op"])                # lowered
            kb += 1
    q = 0
    ib = np.arange(nb)
    for b in (b for b in prob["baths"] if b["kind"] == "F"):
        O = {1: b["op"], -1: b["op"].conj().T}
        # d^nu with nu = +1 the creation operator
        dnu = {1: O[-1], -1: O[1]}
        for k in range(len(b["coef"])):
            bit, nu = np.uint64(1) << np.uint64(q), int(b["nu"][k])
            has = (fer & bit) != 0
            eps = 1 - 2 * (np.array([bin(int(m)).count("1") for m in fer & (bit - np.uint64(1))]) & 1)
            sigma = p * (1 - 2 * (n_f & 1))
            for lowered in (False, True):
                s = np.nonzero(has if lowered else ~has & (n_f < n_f.max()))[0]
                if not len(s):
                    continue
                t = locate(fer[s] ^ bit)
                le, ri = p * eps[s], p * eps[s] * sigma[s] * (1 if lowered else -1)
                A = b["coef"][k] if lowered else 1.0
                B = np.conj(b["coef"][int(b["partner"][k])]) if lowered else 1.0
                i, j = (ib[:, None] * nf + s).ravel(), (ib[:, None] * nf + t).ravel()
                couple(i, j, np.tile(-1j * A * le, nb), np.tile(-1j * B * ri, nb),
                       dnu[nu] if lowered else dnu[-nu])
            q += 1
    # damping and the commutator with H, on every ADO
    rb = np.concatenate([b["rate"] for b in prob["baths"] if b["kind"] != "F"] or [np.zeros(0)])
    rf = np.concatenate([b["rate"] for b in prob["baths"] if b["kind"] == "F"] or [np.zeros(0)])
    damp_f = sum((((fer >> np.uint64(k)) & np.uint64(1)).astype(float) * rf[k] for k in range(len(rf))),
                 np.zeros(nf, complex))
    damp = ((bos @ rb)[:, None] + damp_f).ravel()
    n = np.arange(nb * nf)
    diag = np.arange(nb * nf * d * d)
    rows.append(diag), cols.append(diag), vals.append(-np.repeat(damp, d * d).astype(complex))
    couple(n, n, np.full(len(n), -1j), np.full(len(n), 1j), np.asarray(prob["H"], complex))
    return nb * nf, np.concatenate(rows), np.concatenate(cols), np.concatenate(vals), n_f


def _csr(prob):
    n_ado, r, c, v, _ = _matrix(prob)
    n = n_ado * prob["d"] ** 2
    r, order = torch.from_numpy(r).to(DEV).sort()
    ptr = torch.searchsorted(r, torch.arange(n + 1, device=DEV))
    M = torch.sparse_csr_tensor(ptr, torch.from_numpy(c).to(DEV)[order],
                                torch.from_numpy(v).to(DEV)[order], size=(n, n))
    return n_ado, M


def _arnoldi(mul, b, steps):
    """Orthonormal basis (rows of V) and Hessenberg matrix of the Krylov space of b."""
    V = torch.zeros((steps + 1, len(b)), dtype=b.dtype, device=DEV)
    H = torch.zeros((steps + 1, steps), dtype=b.dtype, device=DEV)
    beta = b.norm()
    V[0] = b / beta
    for j in range(steps):
        w = mul(V[j])
        for _ in range(2):  # classical Gram-Schmidt, twice
            c = V[: j + 1].conj() @ w
            H[: j + 1, j] += c
            w = w - c @ V[: j + 1]
        H[j + 1, j] = w.norm()
        V[j + 1] = w / H[j + 1, j]
    return V, H, beta


def _least_squares(H, beta, shifts):
    """y of min || beta e1 - (H + s I) y || for every shift s: Givens rotations on rows."""
    S, m = len(shifts), H.shape[1]
    A = H[None].repeat(S, 1, 1)
    A[:, range(m), range(m)] += shifts[:, None]
    g = torch.zeros((S, m + 1), dtype=H.dtype, device=DEV)
    g[:, 0] = beta
    for j in range(m):
        a, b = A[:, j, j].clone(), A[:, j + 1, j].clone()
        r = (a.abs() ** 2 + b.abs() ** 2).sqrt()
        c, s = a.conj() / r, b.conj() / r
        for T in (A[:, :, j:], g[:, :, None]):
            x, y = T[:, j].clone(), T[:, j + 1].clone()
            T[:, j] = c[:, None] * x + s[:, None] * y
            T[:, j + 1] = (-b / r)[:, None] * x + (a / r)[:, None] * y
    return torch.linalg.solve_triangular(A[:, :m], g[:, :m, None], upper=True)[:, :, 0], g[:, m].abs()


def _stationary(prob):
    """Null vector of M with unit trace: restarted GMRES on M + e00 tr, diagonal preconditioner."""
    n_ado, M = _csr(prob)
    d, n = prob["d"], n_ado * prob["d"] ** 2
    _, r, c, v, _ = _matrix(prob)
    diag = torch.from_numpy(np.bincount(r[r == c], v[r == c].real, n) +
                            1j * np.bincount(r[r == c], v[r == c].imag, n)).to(DEV)
    diag[: d * d] -= 1.0
    tr = torch.arange(d, device=DEV) * (d + 1)

    def mul(x):
        y = M @ x
        y[0] += x[tr].sum()
        return y

    b = torch.zeros(n, dtype=torch.complex128, device=DEV)
    b[0] = 1.0
    x = torch.zeros_like(b)
    for _ in range(12):
        res = b - mul(x)
        if res.norm() < 1e-14:
            break
        V, H, beta = _arnoldi(lambda u: mul(u / diag), res, min(150, n - 1))
        y, _ = _least_squares(H, beta, torch.zeros(1, dtype=b.dtype, device=DEV))
        x = x + (y[0] @ V[:-1]) / diag
    return x / x[tr].sum(), n_ado


def _in_sets(prob, parts, n_ado, tiers):
    """Columns of truncated hierarchies (leading ADOs) embedded in the deepest one."""
    d = prob["d"]
    out = torch.zeros((n_ado, d, d, len(parts)), dtype=torch.complex128, device=DEV)
    for s, x in enumerate(parts):
        x = x.reshape(-1, d, d)
        out[: len(x), :, :, s] = x
    return out


def exact(case, seed):
    kind = case["kind"]
    if kind == "mlp":
        w, params, x, t, norms = _mlp_arrays(case, seed)
        f64 = lambda a: torch.from_numpy(a).to(DEV, torch.float64)  # noqa: E731
        flat = f64(params).requires_grad_(True)
        im, isd, om, osd = (f64(a) for a in norms)
        y, at = (f64(x) - im) / isd, 0
        for l, (i, o) in enumerate(zip(w[:-1], w[1:])):
            y = y @ flat[at: at + i * o].reshape(i, o) + flat[at + i * o: at + i * o + o]
            at += i * o + o
            y = torch.tanh(y) if l + 2 < len(w) else y
        loss = ((y - (f64(t) - om) / osd) ** 2).mean()
        loss.backward()
        return {"grad": flat.grad, "loss": float(loss)}
    probs, tiers = _problems(case, seed, 1)
    d = probs[0]["d"]
    per = case.get("batch", 0) // case["sets"]
    if kind in ("apply", "evolve"):
        out, traj = None, None
        for s, prob in enumerate(probs):
            n_ado, M = _csr(prob)
            if out is None:
                shape = (n_ado, d, d, case["batch"])
                x0 = (_vector if kind == "apply" else _initial)(
                    *((case, seed, shape) if kind == "apply" else (case, seed, n_ado, d)))
                out = torch.zeros(shape, dtype=torch.complex128, device=DEV)
            x = x0[..., s * per:(s + 1) * per].to(torch.complex128).reshape(-1, per).contiguous()
            if kind == "apply":
                out[..., s * per:(s + 1) * per] = (M @ x).reshape(n_ado, d, d, per)
                continue
            snaps = [x[: d * d].clone()]
            for k in range(1, case["steps"] + 1):
                k1 = M @ x
                k2 = M @ (x + 0.005 * k1)
                k3 = M @ (x + 0.005 * k2)
                k4 = M @ (x + 0.01 * k3)
                x = x + (0.01 / 6.0) * (k1 + 2 * k2 + 2 * k3 + k4)
                if k % case["save"] == 0:
                    snaps.append(x[: d * d].clone())
            out[..., s * per:(s + 1) * per] = x.reshape(n_ado, d, d, per)
            if traj is None:
                traj = torch.zeros((len(snaps), d, d, case["batch"]), dtype=torch.complex128, device=DEV)
            traj[..., s * per:(s + 1) * per] = torch.stack(snaps).reshape(-1, d, d, per)
        if kind == "apply":
            return _shaped(case, out)
        return {"traj": _shaped(case, traj), "ados": _shaped(case, out)}
    states = [_stationary(dict(p, tier_f=t)) for p, t in zip(probs, tiers)]
    if kind == "steady":
        x = _in_sets(probs[0], [s[0] for s in states], states[0][1], tiers)
        return x[..., 0].contiguous() if case["sets"] == 1 else x
    # spectrum: pi A(w) = -Re{Tr[d x_+] + Tr[d^dag x_-]}, (M +- i w) x_+- = (d^dag, d) rho
    op = torch.from_numpy(np.kron(_SM, np.eye(2))).to(DEV)
    om = torch.linspace(-_OMEGA, _OMEGA, case["omegas"], dtype=torch.float64, device=DEV)
    rows = []
    for (x, n_ado), prob, t in zip(states, _problems(case, seed, -1)[0], tiers):
        _, M = _csr(dict(prob, tier_f=t))
        acc = torch.zeros(len(om), dtype=torch.float64, device=DEV)
        for left, read, sign in ((op.conj().T, op, 1.0), (op, op.conj().T, -1.0)):
            b = (left @ x.reshape(-1, d, d)).reshape(-1)
            V, H, beta = _arnoldi(lambda u: M @ u, b, min(260, len(b) - 1))
            top = V[:-1, : d * d].reshape(-1, d, d)
            trace = torch.einsum("il,kli->k", read, top)
            y = torch.cat([_least_squares(H, beta, part)[0]
                           for part in (sign * 1j * om).split(256)])
            acc -= (y @ trace).real
        rows.append(acc / math.pi)
    return torch.stack(rows).cpu().numpy() if case["sets"] > 1 else rows[0].cpu().numpy()
