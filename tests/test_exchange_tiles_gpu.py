"""Exchange self-energy at the edges of its 80 x 80 tiles and K chunks of 16 (triangular column blocks,
several q side by side) against the oracle."""
import numpy as np
import pytest

from oracle import gw_oracle as O
from paper_2011_01400_gb300.synth import make_system

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("n_aux", [1, 15, 79, 80, 81, 96, 161])
@pytest.mark.parametrize("nk", [(1, 1, 1), (3, 3, 1)])
@pytest.mark.parametrize("prec", ["fp64", "3xtf32"])
def test_exchange(n_aux, nk, prec):
    torch = pytest.importorskip("torch")
    from paper_2011_01400_gb300 import gw
    cfg = dict(nk=nk, n_atoms=1, nb_per_atom=8, naux_per_atom=n_aux, n_bands=8, n_occ=3, n_freq=4, sigma=(1, 6), omega_cell=100.0)
    s = make_system(cfg, seed=n_aux, head_wings=0)
    ref = O.sigma_x(s)
    pb = gw.Problem(s, prec)
    plan = gw.gw_plan_create(pb.prob)
    try:
        x = torch.empty((s.n_k, 5), dtype=torch.float64, device="cuda")
        gw.gw_sigma_x(plan, 0, x)
        x = x.cpu().numpy()
    finally:
        gw.gw_plan_destroy(plan)
    # FP32 rows (2 n_basis terms) and products of up to N terms, one sign: a random walk of roundings, factor 4
    tol = 1e-11 if prec == "fp64" else 4.0 * np.sqrt(n_aux + 16.0) * 2.0 ** -24
    assert np.abs(x - ref).max() <= tol * np.abs(ref).max()
