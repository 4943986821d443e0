"""Accuracy of the FP64 inverse of eps~, measured against LAPACK's own error: evenly scaled matrices up to
kappa = 5e8, and eps~ = 1 + D K D with the auxiliary functions' scales D spread over several powers of ten (the error
of elimination does not depend on D). With V = 1 the screened interaction is the inverse itself."""
import numpy as np
import pytest

from paper_2011_01400_gb300.synth import make_system

pytestmark = pytest.mark.gpu


def refined_inverse(e):
    """LAPACK's inverse and one Newton step with its residual in extended precision: error (u kappa)^2 + u (u kappa)."""
    x = np.linalg.inv(e)
    res = (np.eye(len(e)) - e.astype(np.clongdouble) @ x.astype(np.clongdouble)).astype(complex)
    return x.astype(np.clongdouble) + x @ res


def errors(e, x):
    """(||x - ref||, bound) off the diagonal for e^-1 - 1 = x, rows and columns scaled to a diagonal of about one.
    Bound: four times LAPACK's error of the scaled matrix, and 2^-51 kappa ||ref|| for digit products."""
    d = 2.0 ** -np.round(np.log2(e.diagonal().real) / 2)
    es = d[:, None] * e * d
    ref = refined_inverse(es)
    lam = np.linalg.eigvalsh(es)
    off = 1.0 - np.eye(len(e))
    size = np.linalg.norm(ref.astype(complex))
    lapack = np.linalg.norm((np.linalg.inv(es) - ref).astype(complex))
    err = np.linalg.norm(((x / d[:, None] / d) - ref).astype(complex) * off)
    return err, 4.0 * lapack + 2.0 ** -51 * lam[-1] / lam[0] * size


def system(n_aux, spread):
    """Well conditioned K (416 pair rows), D log-uniform in [1, spread]."""
    cfg = dict(nk=(4, 1, 1), n_atoms=1, nb_per_atom=30, naux_per_atom=n_aux, n_bands=30, n_occ=4, n_freq=2,
               sigma=(1, 4), omega_cell=100.0)
    s = make_system(cfg, seed=n_aux, head_wings=0, c_scale=2.0 / np.sqrt(n_aux))
    s.V[:] = np.eye(n_aux)
    s.ctil_R[0] *= np.exp(np.random.default_rng(n_aux).uniform(0, np.log(spread), n_aux))[None, :, None, None]
    return s


def even_system(n_aux, strength):
    """K of 54 pair rows: eps~ has eigenvalues 1 and up to strength^2 times as many tenths."""
    cfg = dict(nk=(2, 1, 1), n_atoms=1, nb_per_atom=12, naux_per_atom=n_aux, n_bands=12, n_occ=3, n_freq=3,
               sigma=(1, 4), omega_cell=100.0)
    s = make_system(cfg, seed=n_aux, head_wings=0, c_scale=strength * 0.206 / np.sqrt(n_aux))
    s.V[:] = np.eye(n_aux)
    return s


@pytest.mark.parametrize("n_aux", [24, 64, 129, 200])
@pytest.mark.parametrize("spread", [1e2, 1e4, 1e6])
def test_spread_rows(n_aux, spread):
    torch = pytest.importorskip("torch")
    from paper_2011_01400_gb300 import gw
    s = system(n_aux, spread)
    pb = gw.Problem(s, "fp64")
    plan = gw.gw_plan_create(pb.prob)
    try:
        chi = torch.empty((2, n_aux, n_aux), dtype=torch.complex128, device="cuda")
        w = torch.empty_like(chi)
        gw.gw_chi0(plan, 0, 1, chi)
        gw.gw_screen(plan, 0, 1, w)
        chi, w = chi.cpu().numpy(), w.cpu().numpy()
    finally:
        gw.gw_plan_destroy(plan)
    for c, x in zip(chi, w):
        err, bound = errors(np.eye(n_aux) - c, x)
        assert err <= bound


@pytest.mark.parametrize("n_aux", [33, 65, 129, 200])
@pytest.mark.parametrize("strength", [1.0, 300.0, 2e4])
def test_even_rows(n_aux, strength):
    """The bound is 2 to 200 times the kernel's error, which is 200 times larger without the last order of digit
    products: from n_aux = 65 on every case fails then."""
    torch = pytest.importorskip("torch")
    from paper_2011_01400_gb300 import gw
    s = even_system(n_aux, strength)
    pb = gw.Problem(s, "fp64")
    plan = gw.gw_plan_create(pb.prob)
    try:
        chi = torch.empty((3, n_aux, n_aux), dtype=torch.complex128, device="cuda")
        w = torch.empty_like(chi)
        gw.gw_chi0(plan, 0, 1, chi)
        gw.gw_screen(plan, 0, 1, w)
        chi, w = chi.cpu().numpy(), w.cpu().numpy()
    finally:
        gw.gw_plan_destroy(plan)
    for c, x in zip(chi, w):
        err, bound = errors(np.eye(n_aux) - c, x)
        assert err <= bound
