"""The work this library is measured on, through its Python binding.

Five kinds of call, over the range a user meets:
  apply   one M psi or M^dag psi (FP64 or mixed), the building block of any
          solver or observable a user writes on top;
  cg      one solve of (M M^dag) x = chi (observables, user-side integrators);
  traj    one HMC trajectory, what a Markov chain is made of;
  batch   one trajectory of many uneven chains in one launch (a scan over
          couplings and temperatures);
  brs     one application of the printed Eq. (2.2) stencil.
Sizes are those of the named workloads in synth.py and of bench.py's modes;
launch shapes are the library's automatic ones unless a case says otherwise.
Fields are Gaussian with variance delta U / 8: rough enough that a solve takes
the hundreds of iterations of a thermalised field, smooth enough that M stays
away from singular (an i.i.d. draw of the full variance does not).
"""
import math

import numpy as np
import torch

from paper_2210_06874_gb300 import hmc

FIELD_SCALE = math.sqrt(1.0 / 8.0)


def listed():
    return [
        # the smallest calls: what a call costs when the arithmetic is nothing
        dict(name="apply_fp64_l3_nt8", kind="apply", L=3, Nt=8, U=2.0, beta=2.0, mu=0.0,
             prec="fp64", dagger=False),
        # one operator application on the largest named lattice, both precisions
        # and both directions
        dict(name="apply_mixed_l24_nt96", kind="apply", L=24, Nt=96, U=4.0, beta=12.0, mu=0.0,
             prec="mixed", dagger=False),
        dict(name="apply_fp64_dag_l24_nt96", kind="apply", L=24, Nt=96, U=4.0, beta=12.0, mu=0.0,
             prec="fp64", dagger=True),
        # a solve in plain FP64 (the path a user checks the mixed one against)
        dict(name="cg_fp64_l12_nt64", kind="cg", L=12, Nt=64, U=3.8, beta=8.0, prec="fp64",
             tuned=False),
        # the same lattice on the mixed path, automatic launch shape
        dict(name="cg_mixed_l12_nt64", kind="cg", L=12, Nt=64, U=3.8, beta=8.0, prec="mixed",
             tuned=False),
        # the largest lattice in the launch shape the autotuner picks for it
        # (split-K tiles, clusters of 6, reliable updates at 0.003)
        dict(name="cg_mixed_tuned_l24_nt96", kind="cg", L=24, Nt=96, U=4.0, beta=12.0,
             prec="mixed", tuned=True),
        # Markov chains: the FP64 workload, the small mixed one with both
        # integrators' step counts in reach, and the largest
        dict(name="traj_fp64_l3_nt8", kind="traj", L=3, Nt=8, U=2.0, beta=2.0, n_md=10, tau=1.0,
             omelyan=False, prec="fp64"),
        dict(name="traj_mixed_l6_nt32", kind="traj", L=6, Nt=32, U=3.5, beta=4.0, n_md=20,
             tau=1.0, omelyan=False, prec="mixed"),
        dict(name="traj_mixed_l24_nt96", kind="traj", L=24, Nt=96, U=4.0, beta=12.0, n_md=10,
             tau=1.0 / 3.0, omelyan=False, prec="mixed"),
        # a scan: many chains of uneven size, short trajectories
        dict(name="batch_mixed_128", kind="batch", chains=128, L_max=12, Nt_max=64, n_md=4,
             tau=0.2),
        # the printed operator on the paper's largest lattice, and an odd one
        dict(name="brs_fp32_l102_nt256", kind="brs", L=102, Nt=256, prec="mixed", dagger=False),
        dict(name="brs_fp64_dag_l51_nt100", kind="brs", L=51, Nt=100, prec="fp64", dagger=True),
    ]


def _log_int(rng, lo, hi):
    return max(lo, min(hi, int(round(math.exp(rng.uniform(math.log(lo), math.log(hi)))))))


def draw(rng):
    kind = rng.choice(["apply", "apply", "cg", "cg", "traj", "traj", "batch", "brs"])
    U = round(rng.uniform(2.0, 5.0), 3)
    delta = rng.choice([0.125, 0.125, 0.25, 1.0 / 6.0])
    if kind == "apply":
        L, Nt = _log_int(rng, 2, 24), _log_int(rng, 3, 96)
        return dict(kind=kind, L=L, Nt=Nt, U=U, beta=delta * Nt,
                    mu=rng.choice([0.0, 0.0, round(rng.uniform(-0.5, 0.5), 3)]),
                    prec=rng.choice(["fp64", "mixed"]), dagger=rng.random() < 0.5)
    if kind == "cg":
        prec = rng.choice(["fp64", "mixed", "mixed"])
        L, Nt = _log_int(rng, 2, 12 if prec == "fp64" else 24), _log_int(rng, 4, 72)
        return dict(kind=kind, L=L, Nt=Nt, U=U, beta=0.125 * Nt, prec=prec, tuned=False)
    if kind == "traj":
        prec = rng.choice(["fp64", "mixed", "mixed"])
        L, Nt = _log_int(rng, 2, 5 if prec == "fp64" else 16), _log_int(rng, 4, 16 if prec == "fp64" else 64)
        n_md = rng.randint(3, 10)
        return dict(kind=kind, L=L, Nt=Nt, U=U, beta=0.125 * Nt, n_md=n_md, tau=n_md / 30.0,
                    omelyan=rng.random() < 0.3, prec=prec)
    if kind == "batch":
        return dict(kind=kind, chains=_log_int(rng, 8, 128), L_max=rng.choice([6, 9, 12]),
                    Nt_max=rng.choice([32, 48, 64]), n_md=rng.randint(2, 4), tau=0.2)
    return dict(kind=kind, L=_log_int(rng, 10, 102), Nt=_log_int(rng, 16, 256),
                prec=rng.choice(["fp64", "mixed"]), dagger=rng.random() < 0.5)


# ---------------------------------------------------------------- inputs
def _prec(case):
    return hmc.PREC_FP64 if case["prec"] == "fp64" else hmc.PREC_MIXED


def _cdtype(case):
    return torch.complex128 if case["prec"] == "fp64" else torch.complex64


def _gen(seed):
    return torch.Generator(device="cuda").manual_seed(int(seed))


def _field(g, Nt, V, variance, scale=FIELD_SCALE):
    return (scale * math.sqrt(variance)) * torch.randn(Nt, V, generator=g, dtype=torch.float64,
                                                       device="cuda")


def _vector(g, Nt, V, dtype=torch.complex128):
    return torch.view_as_complex(
        torch.randn(Nt, V, 2, generator=g, dtype=torch.float64, device="cuda")).to(dtype)


CG_TOL = 1e-11      # of a direct solve
MD_TOL = 1e-10      # of the solves inside trajectories, as in the named workloads


def _chains(case, seed):
    """Sizes and couplings of a batch's chains: the sets of the batched
    workload up to the case's largest, the first chain the largest itself."""
    r = np.random.default_rng(1000 + case["chains"])
    Ls = [v for v in (3, 6, 9, 12) if v <= case["L_max"]]
    Nts = [v for v in (16, 32, 48, 64) if v <= case["Nt_max"]]
    L, Nt = r.choice(Ls, case["chains"]), r.choice(Nts, case["chains"])
    L[0], Nt[0] = case["L_max"], case["Nt_max"]
    U = np.random.default_rng(seed).uniform(2.0, 5.0, case["chains"])
    return [(int(a), int(b), float(u)) for a, b, u in zip(L, Nt, U)]


def _inputs(case, seed):
    """The tensors of a case, from the seed alone."""
    g, kind = _gen(seed), case["kind"]
    if kind == "batch":
        return [_field(g, Nt, 2 * L * L, 0.125 * U) for L, Nt, U in _chains(case, seed)]
    L, Nt, V = case["L"], case["Nt"], 2 * case["L"] ** 2
    if kind == "brs":
        return _field(g, Nt, V, 0.5, 1.0), _vector(g, Nt, V, _cdtype(case))
    variance = case["beta"] / Nt * case["U"]
    if kind == "traj":
        return _field(g, Nt, V, variance)
    return (_field(g, Nt, V, variance, 1.0 if kind == "apply" else FIELD_SCALE),
            _vector(g, Nt, V, _cdtype(case) if kind == "apply" else torch.complex128))


def prepare(case, seed):
    kind, x = case["kind"], _inputs(case, seed)
    s = dict(case=case, seed=int(seed))
    if kind == "batch":
        plist = [hmc.Params(L=L, Nt=Nt, U=U, beta=0.125 * Nt, n_md=case["n_md"],
                            traj_length=case["tau"], cg_tol=MD_TOL, cg_max_iter=200000,
                            precision=hmc.PREC_MIXED) for L, Nt, U in _chains(case, seed)]
        s["batch"] = hmc.Batch(plist)
        s["start"] = torch.cat([f.reshape(-1) for f in x])
        s["phi"] = s["start"].clone()
    elif kind == "brs":
        phi, s["psi"] = x
        c64, c32 = hmc.brs_phases(case["L"], case["Nt"], phi)
        s["cis"] = c64 if case["prec"] == "fp64" else c32
        s["out"] = torch.empty_like(s["psi"])
    else:
        p = dict(L=case["L"], Nt=case["Nt"], U=case["U"], beta=case["beta"],
                 precision=_prec(case))
        if kind == "apply":
            s["ctx"] = hmc.Context(hmc.Params(mu=case["mu"], **p))
            s["phi"], s["psi"] = x
            s["out"] = torch.empty_like(s["psi"])
        elif kind == "cg":
            if case["tuned"]:
                p.update(operand_mode=5, inner_ctas=6, ru_delta=0.003)
            s["ctx"] = hmc.Context(hmc.Params(**p))
            s["phi"], s["chi"] = x
            s["x"] = torch.empty_like(s["chi"])
        else:
            s["ctx"] = hmc.Context(hmc.Params(n_md=case["n_md"], traj_length=case["tau"],
                                              cg_tol=MD_TOL, integrator=int(case["omelyan"]), **p))
            s["start"] = x
            s["phi"] = x.clone()
    return s


def run(s):
    case = s["case"]
    kind = case["kind"]
    if kind == "apply":
        f = s["ctx"].apply_Mdag if case["dagger"] else s["ctx"].apply_M
        return f(s["phi"], s["psi"], out=s["out"], prec=_prec(case))
    if kind == "brs":
        return hmc.apply_brs(case["L"], case["Nt"], 0.125, s["cis"], s["psi"], out=s["out"],
                             dagger=case["dagger"])
    if kind == "cg":
        x, _ = s["ctx"].cg_solve(s["phi"], s["chi"], tol=CG_TOL, prec=_prec(case), x=s["x"])
        return x
    # every pass takes the chain's first step from its start field, so every
    # pass is the same work
    s["phi"].copy_(s["start"])
    if kind == "traj":
        o = s["ctx"].trajectory(s["phi"], s["seed"], 0)
        return dict(phi=s["phi"], H0=o.H0, H1=o.H1, u=o.u, accept=o.accept)
    outs = s["batch"].trajectory(s["phi"], s["seed"], 0)
    return dict(phi=s["phi"], H0=np.array([o.H0 for o in outs]),
                H1=np.array([o.H1 for o in outs]), accept=np.array([o.accept for o in outs]))


# ---------------------------------------------------------------- floors
def _apply_flops(N, fp64):
    """One application on N sites: the exponential of the sparse hopping to
    the result's precision is a polynomial of degree about 11 (FP64) or 6
    (FP32) in h, each degree two additions and a multiply-add per real
    component; the phase, sign and subtraction add about 10."""
    return N * ((11 if fp64 else 6) * 8 + 10.0)


def _iterations(N, beta, digits):
    """Typical CG iterations on these fields (they grow with beta and with
    the digits asked for, and cannot exceed the unknowns by much)."""
    return min(N, 8.5 * beta * digits)


def work(case):
    kind = case["kind"]
    if kind == "batch":
        tot = dict(bytes=0.0, flops=0.0)
        for L, Nt, _ in _chains(case, 0):
            w = work(dict(kind="traj", L=L, Nt=Nt, beta=0.125 * Nt, n_md=case["n_md"],
                          omelyan=False, prec="mixed"))
            tot = {k: tot[k] + w[k] for k in tot}
        return tot
    N = 2.0 * case["L"] ** 2 * case["Nt"]
    fp64 = case["prec"] == "fp64"
    if kind == "brs":
        return dict(bytes=N * (48 if fp64 else 24), flops=N * 16)
    if kind == "apply":
        return dict(bytes=N * (8 + (32 if fp64 else 16)), flops=_apply_flops(N, fp64))
    per_iter = 2 * _apply_flops(N, fp64) + 20 * N
    if kind == "cg":
        return dict(bytes=N * (8 + 32), flops=per_iter * _iterations(N, case["beta"], 11))
    solves = case["n_md"] * (2 if case["omelyan"] else 1) + 1
    return dict(bytes=N * 16, flops=per_iter * _iterations(N, case["beta"], 10) * solves)


# ---------------------------------------------------------------- 64-bit values
def _neighbours(L):
    """Indices in the other sublattice (cell m1 L + m2) of each A site's and
    each B site's three neighbours."""
    m1, m2 = np.divmod(np.arange(L * L), L)
    a = [m1 * L + m2, (m1 - 1) % L * L + m2, m1 * L + (m2 - 1) % L]
    b = [m1 * L + m2, (m1 + 1) % L * L + m2, m1 * L + (m2 + 1) % L]
    return a, b


def _transfer(L, dk, f=1.0):
    LL = L * L
    h = np.zeros((2 * LL, 2 * LL))
    for nb in _neighbours(L)[0]:
        np.add.at(h, (np.arange(LL), LL + nb), 1.0)
        np.add.at(h, (LL + nb, np.arange(LL)), 1.0)
    w, v = np.linalg.eigh(h)
    return torch.from_numpy(f * (v * np.exp(dk * w)) @ v.T).cuda()


class _Operator:
    def __init__(self, E, phi):
        self.E, self.D = E, torch.polar(torch.ones_like(phi), phi)
        self.s = torch.ones(phi.shape[0], 1, dtype=phi.dtype, device=phi.device)
        self.s[0] = -1.0

    def _hop(self, v):     # E v on every slice
        return torch.view_as_complex(
            torch.einsum("xy,tyc->txc", self.E, torch.view_as_real(v)).contiguous())

    def M(self, v):
        return v - self.s * self._hop(torch.roll(self.D * v, 1, 0))

    def Mdag(self, v):
        return v - torch.roll(self.s, -1, 0) * self.D.conj() * self._hop(torch.roll(v, -1, 0))

    def solve(self, chi, tol=2e-15, most=20000):
        """CG to rounding, restarted from the true residual until it stops
        improving."""
        x, best = torch.zeros_like(chi), math.inf
        target = tol * float(torch.linalg.vector_norm(chi))
        for _ in range(4):
            r = chi - self.M(self.Mdag(x))
            p, rr = r.clone(), float(torch.linalg.vector_norm(r)) ** 2
            if not rr or math.sqrt(rr) > 0.5 * best:
                break
            best = math.sqrt(rr)
            for _ in range(most):
                q = self.Mdag(p)
                a = rr / float(torch.linalg.vector_norm(q)) ** 2
                x, r = x + a * p, r - a * self.M(q)
                new = float(torch.linalg.vector_norm(r)) ** 2
                if math.sqrt(new) <= target:
                    break
                p, rr = r + (new / rr) * p, new
        return x


def _philox(seed, stream, n):
    """Philox4x32-10 (Salmon et al. 2011) of counters (e, stream, 0, 0)."""
    m = np.uint64(0xFFFFFFFF)
    sh = np.uint64(32)
    c = [np.arange(n, dtype=np.uint64), np.full(n, stream, np.uint64), np.zeros(n, np.uint64),
         np.zeros(n, np.uint64)]
    k0, k1 = seed & 0xFFFFFFFF, seed >> 32
    for _ in range(10):
        p0, p1 = c[0] * np.uint64(0xD2511F53), c[2] * np.uint64(0xCD9E8D57)
        c = [(p1 >> sh) ^ c[1] ^ np.uint64(k0), p1 & m, (p0 >> sh) ^ c[3] ^ np.uint64(k1), p0 & m]
        k0, k1 = (k0 + 0x9E3779B9) & 0xFFFFFFFF, (k1 + 0xBB67AE85) & 0xFFFFFFFF
    return [(((a << sh) | b) >> np.uint64(11)).astype(np.float64) * 2.0 ** -53 + 2.0 ** -54
            for a, b in ((c[0], c[1]), (c[2], c[3]))]


def _exact_traj(case, phi, seed):
    Nt, V, dl, U = case["Nt"], 2 * case["L"] ** 2, case["beta"] / case["Nt"], case["U"]
    E = _transfer(case["L"], dl)

    def normals(stream):
        u, w = _philox(seed, stream, Nt * V)
        r = np.sqrt(-2.0 * np.log(u))
        return [torch.from_numpy((r * f(2.0 * np.pi * w)).reshape(Nt, V)).cuda()
                for f in (np.cos, np.sin)]

    pi = normals(0)[0]
    a, b = normals(1)
    rho = torch.complex(a, b) / math.sqrt(2.0)
    chi, start = _Operator(E, phi).M(rho), phi.clone()

    def energy(fermions):
        return float((phi * phi).sum() / (2 * dl * U) + (pi * pi).sum() / 2) + fermions

    def kick(c):
        nonlocal pi
        op = _Operator(E, phi)
        x = op.solve(chi)
        F = phi / (dl * U) + 2.0 * (x * op.Mdag(x).conj()).imag
        pi = pi - c * eps * dl * F
        return float((chi.conj() * x).sum().real)

    H0 = energy(float((rho.abs() ** 2).sum()))
    eps, n, lam = case["tau"] / case["n_md"], case["n_md"], 0.1931833275037836
    kicks = [0.5] + [1.0] * (n - 1) + [0.5]
    if case["omelyan"]:
        kicks = [lam] + [1 - 2 * lam, 2 * lam] * (n - 1) + [1 - 2 * lam, lam]
    last = kick(kicks[0])
    for c in kicks[1:]:
        phi = phi + (0.5 if case["omelyan"] else 1.0) * eps * dl * pi
        last = kick(c)
    H1 = energy(last)
    u = float(_philox(seed, 2, 1)[0][0])
    return dict(phi=phi if u < math.exp(min(0.0, H0 - H1)) else start, H0=H0, H1=H1, u=u,
                accept=None)


def exact(case, seed):
    kind = case["kind"]
    if kind == "batch":
        return None        # a whole scan takes minutes in plain torch
    x = _inputs(case, seed)
    if kind == "brs":
        phi, v = x
        c, v = torch.polar(torch.ones_like(phi), phi), v.to(torch.complex128)
        if case["prec"] != "fp64":
            c = c.to(torch.complex64).to(torch.complex128)    # the table the call is given
        LL, dag = case["L"] ** 2, case["dagger"]
        a, b = _neighbours(case["L"])
        A, B, cA, cB = v[:, :LL], v[:, LL:], c[:, :LL], c[:, LL:]
        sg = torch.ones(case["Nt"], 1, dtype=torch.float64, device=v.device)
        sg[-1] = -1.0                                          # t + 1 wraps
        up, dn = (lambda w: sg * torch.roll(w, -1, 0)), (lambda w: torch.roll(sg * w, 1, 0))
        hA = 0.125 * sum(B[:, torch.from_numpy(i).to(v.device)] for i in a)
        hB = 0.125 * sum(A[:, torch.from_numpy(i).to(v.device)] for i in b)
        if dag:
            oA, oB = dn(A) - cA.conj() * A - hA, B - torch.roll(cB, -1, 0) * up(B) - hB
        else:
            oA, oB = up(A) - cA * A - hA, B - cB.conj() * dn(B) - hB
        return torch.cat([oA, oB], 1)
    dl = case["beta"] / case["Nt"]
    if kind == "traj":
        return None if case["L"] > 8 else _exact_traj(case, x, int(seed))
    phi, v = x
    op = _Operator(_transfer(case["L"], dl, math.exp(-dl * case.get("mu", 0.0))), phi)
    if kind == "cg":
        return op.solve(v)
    v = v.to(torch.complex128)
    return op.Mdag(v) if case["dagger"] else op.M(v)
