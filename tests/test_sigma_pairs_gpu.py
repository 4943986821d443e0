"""The Sigma_c contraction at the edges of its tiles (256 rows per pair of CTAs, 64 columns, K stages of 16
or 32): row counts below, at and above one pair, ragged column blocks, against the oracle."""
import numpy as np
import pytest

from oracle import gw_oracle as O
from paper_2011_01400_gb300.synth import make_system

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("n_aux", [2, 30, 64, 66, 128, 190])
@pytest.mark.parametrize("bands,win", [(7, (1, 2)), (16, (0, 8)), (32, (2, 10)), (33, (0, 9))])   # 7, 128, 256, 297 rows per k
@pytest.mark.parametrize("prec", ["3xfp16", "3xtf32"])
def test_sigma_rows(n_aux, bands, win, prec):
    torch = pytest.importorskip("torch")
    from paper_2011_01400_gb300 import gw
    cfg = dict(nk=(2, 1, 1), n_atoms=1, nb_per_atom=33, naux_per_atom=n_aux, n_bands=bands, n_occ=3, n_freq=5, sigma=win,
               omega_cell=100.0)
    s = make_system(cfg, seed=bands, head_wings=0)
    om, g = O.freq_grid(5, s.omega0)
    w = O.screen(s, 1, O.chi0(s, 1, om), om)[1]
    ref = O.sigma_q(s, 1, w, om, g, O.mu_midgap(s))
    pb = gw.Problem(s, prec)
    plan = gw.gw_plan_create(pb.prob)
    try:
        d_w = torch.from_numpy(np.ascontiguousarray(w)).cuda()
        for lo, hi in ((0, 2), (1, 2)):
            acc = torch.zeros(ref.shape, dtype=torch.complex128, device="cuda")
            gw.gw_sigma_ext(plan, 0, 1, d_w, lo, hi, acc)
            a = acc.cpu().numpy()
            # two BF16 or TF32 pieces per operand (2^-16 of the products at most) and FP32 sums
            assert np.linalg.norm(a[lo:hi] - ref[lo:hi]) <= 4.0 * 2.0 ** -16 * np.linalg.norm(ref[lo:hi])
            assert not a[:lo].any()
    finally:
        gw.gw_plan_destroy(plan)
