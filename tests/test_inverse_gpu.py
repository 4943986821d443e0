"""eps~^-1 - 1 of the batched FP64 inversion (block sweeps with exact split products on the tensor
cores) against LAPACK's inverse, at the edges of its pivot blocks (32) and tiles (64), for well and
badly conditioned eps~. With V = 1 the screened interaction is the inverse itself."""
import numpy as np
import pytest

from paper_2011_01400_gb300.synth import make_system

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("n_aux", [1, 2, 31, 32, 33, 63, 64, 65, 96, 127, 129, 200, 321])
@pytest.mark.parametrize("strength", [1.0, 300.0])
def test_inverse_against_lapack(n_aux, strength):
    torch = pytest.importorskip("torch")
    from paper_2011_01400_gb300 import gw
    cfg = dict(nk=(2, 1, 1), n_atoms=1, nb_per_atom=12, naux_per_atom=n_aux, n_bands=12, n_occ=3, n_freq=3,
               sigma=(1, 4), omega_cell=100.0)
    s = make_system(cfg, seed=n_aux, head_wings=0, c_scale=strength * 0.206 / np.sqrt(n_aux))
    s.V[:] = np.eye(n_aux)
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
        e = np.eye(n_aux) - c
        ref = np.linalg.inv(e)
        lam = np.linalg.eigvalsh(e)
        # forward error of an inverse of a positive definite matrix: a small multiple of N u kappa |A^-1|; then
        # x = A^-1 - 1 as stored, V^1/2 = 1 as the iteration leaves it (each side within a few u) and the
        # products with it round relative to x
        bound = (8.0 * n_aux * lam[-1] / lam[0] * np.linalg.norm(ref) + 64.0 * np.linalg.norm(x)) * 1.2e-16
        assert np.linalg.norm(x + np.eye(n_aux) - ref) <= bound
