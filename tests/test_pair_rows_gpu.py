"""Band-pair rows at the edges of their tiles (4 x 4 bands per thread, blocks of at most 256 threads, 2
basis functions per chunk, 16- and 8-byte copies): chi0 and a Sigma_c term of one q against the oracle."""
import numpy as np
import pytest

from oracle import gw_oracle as O
from paper_2011_01400_gb300.synth import make_system

pytestmark = pytest.mark.gpu


# atoms, basis per atom, ABFs per atom, bands, occupied, window
@pytest.mark.parametrize("na,nb,nx,bands,occ,win", [
    (1, 7, 4, 7, 1, (0, 1)),       # odd pitch, one occupied band
    (2, 33, 7, 66, 1, (0, 5)),     # 65 unoccupied bands
    (2, 37, 5, 73, 5, (1, 8)),     # 8-byte copies, 68 bands
    (3, 10, 2, 30, 9, (7, 16)),    # three atoms, nine occupied bands
    (1, 75, 10, 75, 37, (30, 39)), # wide on both sides
    (2, 40, 9, 80, 8, (0, 80)),    # every band in the window
    (2, 70, 3, 140, 4, (2, 6)),    # several blocks along the wide side
])
def test_pair_rows(na, nb, nx, bands, occ, win):
    torch = pytest.importorskip("torch")
    from paper_2011_01400_gb300 import gw
    cfg = dict(nk=(2, 1, 1), n_atoms=na, nb_per_atom=nb, naux_per_atom=nx, n_bands=bands, n_occ=occ, n_freq=6, sigma=win,
               omega_cell=100.0)
    s = make_system(cfg, seed=bands, head_wings=0)
    om, g = O.freq_grid(6, s.omega0)
    ref = O.chi0(s, 1, om)
    w = O.screen(s, 1, ref, om)[1]
    sig = O.sigma_q(s, 1, w, om, g, O.mu_midgap(s))
    pb = gw.Problem(s, "3xbf16")
    plan = gw.gw_plan_create(pb.prob)
    try:
        chi = torch.empty(ref.shape, dtype=torch.complex128, device="cuda")
        gw.gw_chi0(plan, 0, 1, chi)
        acc = torch.zeros(sig.shape, dtype=torch.complex128, device="cuda")
        gw.gw_sigma_ext(plan, 0, 1, torch.from_numpy(w).cuda(), 0, 2, acc)
        chi, acc = chi.cpu().numpy(), acc.cpu().numpy()
    finally:
        gw.gw_plan_destroy(plan)
    # the split method's own bounds: 1e-6 per frequency for chi0, two BF16 pieces per operand for Sigma_c
    for a, b in zip(chi, ref):
        assert np.linalg.norm(a - b) <= 1e-6 * np.linalg.norm(b)
    assert np.linalg.norm(acc - sig) <= 4.0 * 2.0 ** -16 * np.linalg.norm(sig)
