"""Measured cases of the G0W0 path: the calls a program makes through the binding, over the sizes it makes them at.

A case names the call ("path"), the shape of the system (k mesh, atoms, functions per atom, bands,
frequencies) and the options (precision, treatment of q -> 0). Inputs are drawn on the GPU by the
recipe of the package's synthetic systems (orthonormal eigenvectors, decaying two-centre
coefficients, positive definite Coulomb matrices with one dominant eigenvalue at q = 0, time
reversal unless the mesh is shifted), from the seed alone.

The split precisions compute with FP32 accuracy in FP64 containers; their results are kept in
single precision, as a program that stores them would. The FP64 method's results stay FP64.
"""
import ctypes
import math
import random

import numpy as np
import torch

from paper_2011_01400_gb300 import gw
from paper_2011_01400_gb300.synth import surrogate_init

SI = dict(atoms=2, basis=39, aux=200, bands=78, occ=4, freq=32, lo=0, hi=8)      # Si-like 2-atom cell
ZNO = dict(atoms=4, basis=75, aux=400, bands=300, occ=36, freq=32, lo=32, hi=40)  # ZnO-like 4-atom cell
SMALL = dict(atoms=2, basis=16, aux=48, bands=32, occ=4, freq=16, lo=2, hi=6)     # small insulator
CELL = 270.25                                                                     # cell volume (bohr^3)
EXACT_FLOPS = 1.3e13                                                              # what 64 bits do in ~15 s


def listed():
    return [
        # chi0 of one q of the production mesh: the step a program repeats for every q
        dict(SI, name="chi0_si", path="chi0", n1=6, n2=6, n3=6, q=1, prec="3xfp16", head=0),
        # chi0 of a larger cell with many transitions per k, at the most accurate split, on a sparse grid
        dict(ZNO, name="chi0_zno", path="chi0", n1=2, n2=2, n3=1, q=1, prec="3xbf16", head=0, freq=16),
        # the plain FP64 method on a small system: what results are checked against
        dict(SMALL, name="chi0_small_fp64", path="chi0", n1=2, n2=2, n3=2, q=1, prec="fp64", head=0),
        # the Gamma point of the screening with head and wings, and an ordinary q of a large cell
        dict(SI, name="screen_si_gamma", path="screen", n1=2, n2=2, n3=2, q=0, prec="3xfp16", head=1),
        dict(ZNO, name="screen_zno", path="screen", n1=2, n2=1, n3=1, q=1, prec="3xfp16", head=0, aux=300, freq=16),
        # Sigma_c of one q with a given W^c, all k of the production mesh
        dict(SI, name="sigma_si", path="sigma", n1=6, n2=6, n3=6, q=1, prec="3xfp16", head=0, k_hi=216),
        # one point of a band structure: the q term of one off-mesh k of a large cell
        dict(ZNO, name="sigma_zno_line", path="sigma", n1=2, n2=2, n3=2, q=3, prec="3xtf32", head=0, k_hi=1),
        # the exchange part, once per system
        dict(SI, name="exchange_si", path="exchange", n1=4, n2=4, n3=4, q=0, prec="3xfp16", head=0),
        # a complete run from inputs to quasiparticle energies: the smallest system, where launches and
        # latency count, and an ordinary one
        dict(SMALL, name="pass_small", path="pass", n1=2, n2=2, n3=2, q=0, prec="3xbf16", head=1),
        dict(SI, name="pass_si", path="pass", n1=4, n2=4, n3=4, q=0, prec="3xfp16", head=2),
        # screening many materials: independent systems of uneven size in one call
        dict(name="batch_uneven", path="batch", systems=8, shapes=30000, prec="3xfp16"),
        # one gradient evaluation of the frequency surrogate on a data set
        dict(name="net_grad", path="net", n_in=12, hidden=256, n_out=48, rows=16384),
    ]


def draw(rng):
    most = max(work(c)["flops"] for c in listed())
    while True:
        c = _draw(rng)
        if work(c)["flops"] <= most:
            return c


def _draw(rng):
    def log(lo, hi):
        return int(round(math.exp(rng.uniform(math.log(lo), math.log(hi)))))

    path = rng.choice(["chi0", "screen", "sigma", "exchange", "pass", "batch", "net", "chi0", "screen", "sigma", "pass"])
    if path == "net":
        return dict(path="net", n_in=rng.randint(4, 16), hidden=rng.choice([64, 128, 200, 256]),
                    n_out=rng.randint(12, 48), rows=log(500, 20000))
    if path == "batch":
        return dict(path="batch", systems=rng.randint(2, 8), shapes=rng.randrange(10 ** 6), prec=rng.choice(["3xfp16", "3xbf16"]))
    prec = rng.choice(["3xfp16", "3xfp16", "3xbf16", "3xtf32"])
    c = dict(path=path, prec=prec, atoms=2, basis=rng.randint(10, 40), aux=log(24, 240), occ=rng.randint(2, 8),
             freq=rng.randint(8, 40), q=0, head=0)
    if path in ("chi0", "sigma", "screen") and rng.random() < 0.3:                # larger cells
        c.update(atoms=4, basis=rng.randint(40, 75), aux=log(100, 300), occ=rng.randint(16, 36), freq=rng.randint(8, 16))
    c["bands"] = rng.randint(max(c["occ"] + 6, c["atoms"] * c["basis"] // 2), c["atoms"] * c["basis"])
    width = rng.randint(2, 5)
    c["lo"], c["hi"] = max(0, c["occ"] - width), min(c["bands"], c["occ"] + width)
    top = 2 if c["atoms"] == 4 or path == "screen" else 4 if path in ("pass", "exchange") else 6
    c["n1"], c["n2"], c["n3"] = (rng.randint(1 if i else 2, top) for i in range(3))
    if path == "chi0" and c["atoms"] == 2 and c["aux"] <= 64 and rng.random() < 0.5:
        c["prec"] = "fp64"
    nk = c["n1"] * c["n2"] * c["n3"]
    if path in ("chi0", "screen", "sigma"):
        c["q"] = rng.randrange(nk)
    if path == "screen":
        c["head"] = rng.choice([0, 1])
    if path == "pass":
        c["head"] = rng.choice([0, 1, 2])
    if path == "sigma":
        c["k_hi"] = rng.choice([1, nk])
    return c


# ---------------------------------------------------------------------------------------------
# inputs
# ---------------------------------------------------------------------------------------------

_C = torch.complex128
_D = torch.float64


def _minus(n, k):
    i3, i2, i1 = k % n[2], k // n[2] % n[1], k // (n[1] * n[2])
    return (-i1 % n[0] * n[1] + -i2 % n[1]) * n[2] + -i3 % n[2]


def _plus(n, k, q):
    i1, i2, i3 = k // (n[1] * n[2]) + q // (n[1] * n[2]), k // n[2] % n[1] + q // n[2] % n[1], k % n[2] + q % n[2]
    return (i1 % n[0] * n[1] + i2 % n[1]) * n[2] + i3 % n[2]


def _gauss(g, *shape):
    return torch.complex(torch.randn(shape, generator=g, device="cuda", dtype=_D),
                         torch.randn(shape, generator=g, device="cuda", dtype=_D)) / math.sqrt(2.0)


def _mirror(x, n, sign=1):
    """x(-k) = sign conj(x(k)) over the leading k axis, exactly."""
    mk = torch.tensor([_minus(n, k) for k in range(x.shape[0])], device="cuda")
    k = torch.arange(x.shape[0], device="cuda")
    shape = (-1,) + (1,) * (x.dim() - 1)
    y = x[mk]
    other = sign * (y.conj() if y.is_complex() else y)
    same = (x + other) / 2 if x.is_complex() else x
    return torch.where((k < mk).view(shape), x, torch.where((k > mk).view(shape), other, same)).resolve_conj().contiguous()


def _orthonormal(x):
    """Columns of x made orthonormal (twice, by the Cholesky factor of the overlap)."""
    for _ in range(2):
        low = torch.linalg.cholesky(x.mH @ x)
        x = torch.linalg.solve_triangular(low.mH, x, upper=True, left=False)
    return x


class _System:
    """Inputs of one system on the GPU, in the layouts of the binding's gw_problem."""

    def __init__(self, c, seed):
        g = torch.Generator(device="cuda")
        g.manual_seed(seed)
        self.c = c
        self.n = n = (c["n1"], c["n2"], c["n3"])
        self.nk = nk = n[0] * n[1] * n[2]
        self.nb, self.nx = c["atoms"] * c["basis"], c["atoms"] * c["aux"]
        self.shifted = c["path"] == "sigma" and c["k_hi"] < nk
        self.k0 = (0.11, 0.07, 0.23) if self.shifted else (0.0, 0.0, 0.0)
        occ, bands = c["occ"], c["bands"]
        e = torch.rand((nk, bands), generator=g, device="cuda", dtype=_D)
        e = torch.cat([(-0.8 + 0.6 * e[:, :occ]).sort(1).values, (0.05 + 2.95 * e[:, occ:]).sort(1).values], 1)
        v = _gauss(g, nk, self.nb, bands)
        pm = None
        if c["head"]:
            pm = _gauss(g, nk, 3, bands, bands)
            pm = 0.5 * (pm + pm.mH) / math.sqrt(2.0)
        if not self.shifted:
            e, v = _mirror(e, n), _mirror(v, n)
            pm = None if pm is None else _mirror(pm, n, -1)
        self.eps, self.evec, self.pmom = e, _orthonormal(v).contiguous(), pm
        self.R = np.array([(0, 0, 0), (1, 0, 0), (-1, 0, 0), (0, 1, 0), (0, -1, 0), (0, 0, 1), (0, 0, -1)], dtype=np.int32)
        decay = torch.tensor(np.exp(-0.5 * np.sqrt((self.R ** 2.0).sum(1))), device="cuda")
        size = 0.206 * math.sqrt(self.nb / (self.nx * c["basis"]))
        self.ctil = size * torch.randn((c["atoms"], 7, c["aux"], c["basis"], self.nb), generator=g, device="cuda", dtype=_D)
        self.ctil *= decay.view(1, 7, 1, 1, 1)
        a = _gauss(g, nk, self.nx, self.nx)
        a = a if self.shifted else _mirror(a, n)
        v = a @ a.mH
        v /= self.nx
        v.diagonal(dim1=1, dim2=2).add_(0.1)
        x = torch.randn(self.nx, generator=g, device="cuda", dtype=_D)
        x /= x.norm()
        v[0] += 40.0 * torch.outer(x, x)       # the eigenvalue that stands for G = 0, ten times the others
        v = 0.5 * (v + v.mH)
        self.V = v if self.shifted else _mirror(v, n)
        self.basis_atom = np.repeat(np.arange(c["atoms"], dtype=np.int32), c["basis"])
        self.aux_atom = np.repeat(np.arange(c["atoms"], dtype=np.int32), c["aux"])
        self.generator = g

    def problem(self):
        c, i32 = self.c, ctypes.POINTER(ctypes.c_int32)
        p = gw.gw_problem()
        p.nk[:] = list(self.n)
        p.n_atoms, p.n_basis, p.n_bands, p.n_occ, p.n_aux = c["atoms"], self.nb, c["bands"], c["occ"], self.nx
        p.basis_atom, p.aux_atom = self.basis_atom.ctypes.data_as(i32), self.aux_atom.ctypes.data_as(i32)
        p.n_R, p.R = len(self.R), self.R.ctypes.data_as(i32)
        p.eps, p.evec, p.ctil_R, p.V = (t.data_ptr() for t in (self.eps, self.evec, self.ctil, self.V))
        p.pmom = None if self.pmom is None else self.pmom.data_ptr()
        p.omega_cell = CELL
        p.qhat[:] = [1.0, 0.0, 0.0]
        p.head_wings, p.n_freq, p.omega0 = c["head"], c["freq"], 1.0
        p.sigma_lo, p.sigma_hi, p.spin, p.mu = c["lo"], c["hi"], 2.0, math.nan
        p.prec = gw.PREC[c["prec"]]
        p.time_reversal = int(not self.shifted)
        p.k_offset[:] = list(self.k0)
        return p

    def screened(self):
        """A W^c(q, i w) [freq][N][N] as the method gives it: poles of random strength in the range of the
        transition energies, screened by the Coulomb matrix of this q."""
        lam, u = torch.linalg.eigh(self.V[self.c["q"]])
        root = (u * lam.sqrt()) @ u.mH
        poles = 0.3 + 3.4 * torch.rand(2 * self.nx, generator=self.generator, device="cuda", dtype=_D)
        b = root @ _gauss(self.generator, self.nx, 2 * self.nx) / math.sqrt(2 * self.nx)
        eye = torch.eye(self.nx, device="cuda", dtype=_D)
        out = torch.empty((self.c["freq"], self.nx, self.nx), device="cuda", dtype=_C)
        for j, w in enumerate(_grid(self.c["freq"])[0]):
            x = torch.linalg.inv(eye + (b * (2 * poles / (w * w + poles * poles))) @ b.mH) - eye
            x = root @ x @ root
            out[j] = 0.5 * (x + x.mH)
        return out


def _batch_shapes(c):
    """Uneven systems: 20-80 bands, 120-400 auxiliary functions, 2 to 3 points per mesh axis, 16-32 frequencies."""
    r = random.Random(c["shapes"])
    out = []
    for _ in range(c["systems"]):
        basis, occ, m = r.randint(10, 40), r.randint(4, 8), r.randint(2, 3)
        out.append(dict(path="pass", prec=c["prec"], atoms=2, basis=basis, aux=r.randint(60, 200), bands=2 * basis, occ=occ,
                        freq=r.randint(16, 32), lo=occ - 2, hi=occ + 2, n1=m, n2=m, n3=r.randint(2, m), q=0, head=r.choice([0, 1])))
    return out


class _State:
    """Inputs, and the plan a program keeps for them (released with it)."""
    plan = None

    def __del__(self):
        if self.plan is not None:
            gw.gw_plan_destroy(self.plan)


class _Net:
    model = None

    def __del__(self):
        if self.model is not None:
            gw.gw_surrogate_destroy(self.model)


def _net_inputs(case, seed):
    g = torch.Generator(device="cuda")
    g.manual_seed(seed)
    params = torch.from_numpy(surrogate_init(case["n_in"], case["hidden"], case["n_out"], seed=seed, out_gain=1.0)).cuda()
    # mode curves: sums of decaying Lorentzians on the coarse and the fine frequencies, scaled by the first value
    f = torch.tensor(_grid(case["n_in"] + case["n_out"])[0], device="cuda")
    pole = 0.3 + 3.4 * torch.rand((case["rows"], 4, 1), generator=g, device="cuda", dtype=_D)
    amp = torch.rand((case["rows"], 4, 1), generator=g, device="cuda", dtype=_D)
    d = -(amp * 2 * pole / (f * f + pole * pole)).sum(1)
    d = (d / d[:, :1].abs()).float()
    step = (case["n_in"] + case["n_out"]) // case["n_in"]
    coarse = [i * step for i in range(case["n_in"])]
    fine = [i for i in range(case["n_in"] + case["n_out"]) if i not in set(coarse)]
    return params, d[:, coarse].contiguous(), d[:, fine].contiguous()


def prepare(case, seed):
    if case["path"] == "net":
        s = _Net()
        s.case = case
        s.params, s.x, s.y = _net_inputs(case, seed)
        s.model = gw.gw_surrogate_create(case["n_in"], case["hidden"], case["n_out"], s.params)
        s.grad = torch.empty_like(s.params)
        return s
    s = _State()
    s.case = case
    if case["path"] == "batch":
        s.systems = [_System(c, seed * 1000 + i) for i, c in enumerate(_batch_shapes(case))]
        s.accs = [_sigma_buffer(t) for t in s.systems]
        torch.cuda.synchronize()
        s.plan = gw.gw_plan_create([t.problem() for t in s.systems])
        return s
    s.system = _System(case, seed)
    s.wc = s.system.screened() if case["path"] == "sigma" else None
    s.problem = s.system.problem()
    if case["path"] != "pass":
        s.plan = gw.gw_plan_create(s.problem)
    if case["path"] in ("chi0", "screen"):
        s.out = torch.empty((case["freq"], s.system.nx, s.system.nx), device="cuda", dtype=_C)
    elif case["path"] == "exchange":
        s.out = torch.empty((s.system.nk, case["hi"] - case["lo"]), device="cuda", dtype=_D)
    else:
        s.out = _sigma_buffer(s.system)
    if case["path"] == "screen":
        gw.gw_chi0(s.plan, 0, case["q"])
    return s


def _sigma_buffer(system):
    c = system.c
    return torch.zeros((system.nk, c["hi"] - c["lo"], c["freq"]), device="cuda", dtype=_C)


def _kept(x, prec):
    if prec == "fp64":
        return x
    return x.to(torch.complex64 if x.is_complex() else torch.float32)


def run(state):
    c = state.case
    if c["path"] == "chi0":
        gw.gw_chi0(state.plan, 0, c["q"], state.out)
    elif c["path"] == "screen":
        gw.gw_screen(state.plan, 0, c["q"], state.out)
    elif c["path"] == "sigma":
        state.out.zero_()
        gw.gw_sigma_ext(state.plan, 0, c["q"], state.wc, 0, c["k_hi"], state.out)
    elif c["path"] == "exchange":
        gw.gw_sigma_x(state.plan, 0, state.out)
    elif c["path"] == "pass":
        state.out.zero_()
        plan = gw.gw_plan_create(state.problem)
        try:
            gw.gw_g0w0(plan, 0, state.out)
            e, gap, _ = gw.gw_qp(plan, 0, state.system.nk, c["hi"] - c["lo"], sigma=state.out)
        finally:
            gw.gw_plan_destroy(plan)
        return {"sigma": _kept(state.out, c["prec"]), "e_qp": e.astype(np.float32), "gap": np.float32(gap)}
    elif c["path"] == "batch":
        for a in state.accs:
            a.zero_()
        gw.gw_g0w0_batch(state.plan, state.accs)
        return [_kept(a, c["prec"]) for a in state.accs]
    else:
        loss = gw.gw_surrogate_loss_grad(state.model, state.x, state.y, state.grad)
        return {"loss": np.float32(loss), "grad": state.grad}
    return _kept(state.out, c["prec"])


# ---------------------------------------------------------------------------------------------
# the work a call cannot do without
# ---------------------------------------------------------------------------------------------


def work(case):
    if case["path"] == "net":
        p = case["hidden"] * (case["n_in"] + 2 * case["hidden"] + case["n_out"]) + case["n_in"] * case["n_out"]
        return {"bytes": 4 * (case["rows"] * (case["n_in"] + case["n_out"]) + 2 * p), "flops": 6 * case["rows"] * p}
    if case["path"] == "batch":
        each = [work(c) for c in _batch_shapes(case)]
        return {k: sum(w[k] for w in each) for k in ("bytes", "flops")}
    c = case
    nk, N, NB = c["n1"] * c["n2"] * c["n3"], c["atoms"] * c["aux"], c["atoms"] * c["basis"]
    coeff = 8 * 7 * c["atoms"] * c["aux"] * c["basis"] * NB + 16 * nk * NB * c["bands"] + 8 * nk * c["bands"]
    mats = 16 * c["freq"] * N * N
    pairs = nk * c["occ"] * (c["bands"] - c["occ"])
    chi0 = 4 * pairs * N * (N + 1) * c["freq"] + 16 * pairs * N * c["basis"]
    screen = 28 * N ** 3 * c["freq"]

    def sigma(k, bands):
        rows = k * (c["hi"] - c["lo"]) * bands
        return rows, 16 * rows * N * c["basis"]
    sig = 16 * nk * (c["hi"] - c["lo"]) * c["freq"]
    if c["path"] == "chi0":
        return {"bytes": coeff + mats, "flops": chi0}
    if c["path"] == "screen":
        return {"bytes": 2 * mats + 16 * N * N, "flops": screen}
    if c["path"] == "sigma":
        rows, m = sigma(c["k_hi"], c["bands"])
        return {"bytes": coeff + mats + sig, "flops": m + 4 * rows * N * (N + 1) * c["freq"]}
    if c["path"] == "exchange":
        rows, m = sigma(nk, c["occ"])
        return {"bytes": coeff + 16 * nk * N * N + sig // c["freq"], "flops": nk * (m + 4 * rows * N * (N + 1))}
    # a pass: the half transform, V^1/2 of each q, then each pair (q, -q) once and the targets k that are not mirrored
    n = (c["n1"], c["n2"], c["n3"])
    half = sum(1 for k in range(nk) if _minus(n, k) >= k)
    rows, m = sigma(nk if c["head"] == 1 else half, c["bands"])
    flops = 8 * nk * N * c["basis"] * NB * c["bands"] + 40 * half * N ** 3
    flops += half * (chi0 + screen) + nk * (m + 4 * rows * N * (N + 1) * c["freq"])
    return {"bytes": coeff + 16 * nk * N * N + 48 * nk * c["bands"] ** 2 * (c["head"] > 0) + sig, "flops": flops}


# ---------------------------------------------------------------------------------------------
# the same results by plain torch in 64 bits
# ---------------------------------------------------------------------------------------------


def _grid(n):
    x, w = np.polynomial.legendre.leggauss(n)
    return (1 + x) / (1 - x), 2 * w / (1 - x) ** 2


class _Plain:
    def __init__(self, s):
        self.s, self.c, self.half = s, s.c, {}
        self.omega, self.weight = _grid(s.c["freq"])
        self.mu = float(0.5 * (s.eps[:, s.c["occ"] - 1].max() + s.eps[:, s.c["occ"]].min()))

    def t1(self, k):
        """sum_R e^{2 pi i k R} sum_j C(R)_{mu i j} c_jb(k): [atom][aux][basis][bands]"""
        if k not in self.half:
            s, n = self.s, self.s.n
            f = np.array([k // (n[1] * n[2]) / n[0], k // n[2] % n[1] / n[1], k % n[2] / n[2]]) + np.array(s.k0)
            ph = torch.tensor(np.exp(2j * np.pi * (s.R @ f)), device="cuda")
            mat = torch.complex(torch.tensordot(ph.real, s.ctil, dims=([0], [1])), torch.tensordot(ph.imag, s.ctil, dims=([0], [1])))
            self.half[k] = mat @ s.evec[k]
        return self.half[k]

    def rows(self, k, kq, up, low):
        """M_{mu, a, b}, a of the bands `up` at kq, b of the bands `low` at k: [N][a][b]"""
        s, out = self.s, []
        tq, tk = self.t1(kq), self.t1(k)
        for a in range(self.c["atoms"]):
            i = slice(a * self.c["basis"], (a + 1) * self.c["basis"])
            out.append(tq[a][:, :, up].mH @ s.evec[k][i, low] + s.evec[kq][i, up].mH @ tk[a][:, :, low])
        return torch.cat(out)

    def bands(self):
        return slice(self.c["occ"], self.c["bands"]), slice(0, self.c["occ"])

    def chi0(self, q):
        s, (up, low) = self.s, self.bands()
        out = torch.zeros((len(self.omega), s.nx, s.nx), device="cuda", dtype=_C)
        step = max(1, int(3e8 // (s.nx * self.c["occ"] * (self.c["bands"] - self.c["occ"]))))
        for k0 in range(0, s.nk, step):
            m, d = [], []
            for k in range(k0, min(s.nk, k0 + step)):
                kq = _plus(s.n, k, q)
                m.append(self.rows(k, kq, up, low).reshape(s.nx, -1))
                d.append((s.eps[kq, up][:, None] - s.eps[k, low][None, :]).reshape(-1))
            m, d = torch.cat(m, 1), torch.cat(d)
            for j, w in enumerate(self.omega):
                out[j].addmm_(m * (2 * d / (w * w + d * d)), m.mH)
        return out.mul_(-2.0 / s.nk)

    def wc(self, q, chi):
        s, c = self.s, self.c
        lam, u = torch.linalg.eigh(s.V[q])
        root = (u * lam.sqrt()) @ u.mH
        eye = torch.eye(s.nx, device="cuda", dtype=_C)
        head = q == 0 and c["head"] == 1
        if head:
            x1 = u[:, -1] * (u[:, -1].abs()[u[:, -1].abs().argmax()] / u[u[:, -1].abs().argmax(), -1])
            body = (u[:, :-1] * lam[:-1].sqrt()) @ u[:, :-1].mH
            up, low = self.bands()
            d = s.eps[:, up][:, :, None] - s.eps[:, low][:, None, :]
            p = s.pmom[:, 0, low, up].mT                                # (p q^)_{ia}, laid out [k][a][i]
            mc = [self.rows(k, k, up, low).conj() for k in range(s.nk)]
        out = torch.empty_like(chi)
        for j, w in enumerate(self.omega):
            if head:
                e = eye - body @ chi[j] @ body
                f = 2 / (d * d + w * w)
                h = sum((mc[k] * (p[k] * f[k])).sum((1, 2)) for k in range(s.nk))
                row = -(2.0 / s.nk) * math.sqrt(4 * math.pi / CELL) * (h @ body)
                one = 4 * math.pi * 2.0 / (CELL * s.nk) * float((p.abs() ** 2 * f / d).sum())
                e = e + one * torch.outer(x1, x1.conj()) + torch.outer(x1, row) + torch.outer(row.conj(), x1.conj())
            else:
                e = eye - root @ chi[j] @ root
            out[j] = root @ (torch.linalg.inv(e) - eye) @ root
        return out

    def sigma(self, q, wc, ks, out):
        s, c = self.s, self.c
        om, g = (torch.tensor(v, device="cuda") for v in (self.omega, self.weight))
        for k in ks:
            kq = next(p for p in range(s.nk) if _plus(s.n, p, q) == k)
            a = self.rows(kq, k, slice(c["lo"], c["hi"]), slice(0, c["bands"])).reshape(s.nx, -1)
            S = torch.stack([((w.mT @ a) * a.conj()).sum(0).real for w in wc], -1).view(c["hi"] - c["lo"], c["bands"], -1)
            z = 1j * om[:, None] + (self.mu - s.eps[kq])[None, :]                       # [w][m]
            kern = g * 2 * z[:, :, None] / (z[:, :, None] ** 2 + om ** 2)               # [w][m][j]
            out[k] -= torch.einsum("nmj,wmj->nw", S.to(_C), kern) / (2 * math.pi * s.nk)

    def qp(self, sigma):
        """Two-pole continuation (linear least squares) and Newton's method, per band and k."""
        c, z = self.c, 1j * self.omega
        e0 = self.s.eps[:, c["lo"]:c["hi"]].cpu().numpy()
        out, f = np.empty(e0.shape), sigma.cpu().numpy()
        for i in np.ndindex(e0.shape):
            A = np.stack([-f[i] * z, -f[i], z, np.ones_like(z)], 1)
            norm = np.linalg.norm(A, axis=0)
            q1, q0, p1, p0 = np.linalg.lstsq(A / norm, f[i] * z * z, rcond=None)[0] / norm
            E = e0[i]
            for _ in range(100):
                x = E - self.mu
                den = x * x + q1 * x + q0
                step = (E - e0[i] - ((p1 * x + p0) / den).real) / (1 - ((p1 * den - (p1 * x + p0) * (2 * x + q1)) / den ** 2).real)
                E -= step
                if abs(step) < 1e-12:
                    break
            else:
                return None, None
            out[i] = E
        gap = np.nan
        if c["lo"] < c["occ"] < c["hi"]:
            gap = out[:, c["occ"] - c["lo"]].min() - out[:, c["occ"] - 1 - c["lo"]].max()
        return out, np.float64(gap)

    def g0w0(self):
        out = torch.zeros_like(_sigma_buffer(self.s))
        for q in range(self.s.nk):
            self.sigma(q, self.wc(q, self.chi0(q)), range(self.s.nk), out)
        return out


def _plain_flops(case):
    """What exact() multiplies, in 64 bits, without the symmetries."""
    w = work(case)["flops"]
    return w * {"chi0": 2, "screen": 2, "sigma": 2, "exchange": 2, "pass": 8, "net": 0}[case["path"]] + (
        2 * work(dict(case, path="chi0"))["flops"] if case["path"] == "screen" else 0)


def exact(case, seed):
    if case["path"] == "net":
        return _net_exact(case, seed)
    if case["path"] == "batch":
        shapes = _batch_shapes(case)
        if sum(_plain_flops(c) for c in shapes) > EXACT_FLOPS:
            return None
        return [_Plain(_System(c, seed * 1000 + i)).g0w0() for i, c in enumerate(shapes)]
    if _plain_flops(case) > EXACT_FLOPS or (case["path"] == "pass" and case["head"] == 2):
        return None
    p = _Plain(_System(case, seed))
    s = p.s
    if case["path"] == "chi0":
        return p.chi0(case["q"])
    if case["path"] == "screen":
        return p.wc(case["q"], p.chi0(case["q"]))
    if case["path"] == "sigma":
        wc = s.screened()
        out = torch.zeros_like(_sigma_buffer(s))
        p.sigma(case["q"], wc, range(case["k_hi"]), out)
        return out
    if case["path"] == "exchange":
        out = torch.zeros((s.nk, case["hi"] - case["lo"]), device="cuda", dtype=_D)
        for q in range(s.nk):
            for kq in range(s.nk):
                a = p.rows(kq, _plus(s.n, kq, q), slice(case["lo"], case["hi"]), slice(0, case["occ"]))
                flat = a.reshape(s.nx, -1)
                out[_plus(s.n, kq, q)] -= ((s.V[q].mT @ flat) * flat.conj()).sum(0).real.view(a.shape[1:]).sum(1) / s.nk
        return out
    sigma = p.g0w0()
    e, gap = p.qp(sigma)
    return {"sigma": sigma, "e_qp": e, "gap": gap}


def _net_exact(case, seed):
    params, x, y = _net_inputs(case, seed)
    I, H, O = case["n_in"], case["hidden"], case["n_out"]
    shapes = [(H, I), (H,), (H, H), (H,), (H, H), (H,), (O, H), (O,), (O, I), (1,)]
    parts = [t.view(sh) for t, sh in zip(params.split([math.prod(sh) for sh in shapes]), shapes)]
    # the network's matrices enter as bfloat16, everything else as given
    parts = [(t.bfloat16() if i in (0, 2, 4, 6) else t).double().requires_grad_() for i, t in enumerate(parts)]
    with torch.enable_grad():
        h = x.double()
        for i in (0, 2, 4):
            h = torch.nn.functional.silu(h @ parts[i].T + parts[i + 1])
        f = parts[9] * (h @ parts[6].T + parts[7]) + x.double() @ parts[8].T
        loss = ((f - y.double()) ** 2).mean()
        grads = torch.autograd.grad(loss, parts[:9])
    return {"loss": np.float64(loss.item()), "grad": torch.cat([t.reshape(-1) for t in grads] + [torch.zeros(1, device="cuda", dtype=_D)])}
