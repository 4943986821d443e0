"""The inverse of eps~ = 1 + D K D with the auxiliary functions' scales D spread over several powers of ten: the
error of elimination does not depend on D. With V = 1 the screened interaction is the inverse itself."""
import numpy as np
import pytest

from paper_2011_01400_gb300.synth import make_system

pytestmark = pytest.mark.gpu


def refined_inverse(e):
    """Inverse to well below 2^-53: LAPACK's and Newton steps in extended precision."""
    x, el, one = np.linalg.inv(e).astype(np.clongdouble), e.astype(np.clongdouble), np.eye(len(e))
    for _ in range(3):
        x = x + x @ (one - el @ x)
    return x


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
