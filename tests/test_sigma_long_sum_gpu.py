"""The Sigma_c contraction over many ABFs: its truncating accumulators are drained every 512 ABFs, so the error does
not grow with the number of ABFs. Random signs, and terms of one sign, where the truncation adds up."""
import numpy as np
import pytest

from oracle import gw_oracle as O
from paper_2011_01400_gb300.synth import make_system

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("one_sign", [False, True])
@pytest.mark.parametrize("prec,pieces,adds", [("3xtf32", 2.0 ** -20, 128), ("3xfp16", 2.0 ** -16, 64)])
# 512 ABFs are one segment (16 or 32 stages), 514 and 544 one stage more
@pytest.mark.parametrize("n_aux", [510, 512, 514, 544, 1000, 1600])
def test_error_of_the_accumulator(one_sign, prec, pieces, adds, n_aux):
    torch = pytest.importorskip("torch")
    from paper_2011_01400_gb300 import gw
    cfg = dict(nk=(1, 1, 1), n_atoms=1, nb_per_atom=8, naux_per_atom=n_aux, n_bands=8, n_occ=3, n_freq=2, sigma=(1, 4),
               omega_cell=100.0)
    s = make_system(cfg, seed=n_aux, head_wings=0, trs=False)
    rng = np.random.default_rng(n_aux)
    b = rng.standard_normal((n_aux, 40)) + 1j * rng.standard_normal((n_aux, 40))
    if one_sign:
        s.ctil_R[0][:] = np.abs(s.ctil_R[0])
        s.evec[:] = np.abs(s.evec)
        b = np.abs(b)
    om, g = O.freq_grid(2, s.omega0)
    w = np.stack([b @ b.conj().T / (n_aux * (1.0 + x * x)) for x in om]).astype(np.complex128)
    ref = O.sigma_q(s, 0, w, om, g, O.mu_midgap(s))
    pb = gw.Problem(s, prec)
    plan = gw.gw_plan_create(pb.prob)
    try:
        acc = torch.zeros(ref.shape, dtype=torch.complex128, device="cuda")
        d_w = torch.from_numpy(w).cuda()
        gw.gw_sigma_ext(plan, 0, 0, d_w, 0, 1, acc)
        acc = acc.cpu().numpy()
    finally:
        gw.gw_plan_destroy(plan)
    # two pieces per operand; each addition between two drains drops up to an ulp of the accumulator, half on average
    bound = pieces + adds * 2.0 ** -24
    err = np.linalg.norm(acc - ref) / np.linalg.norm(ref)
    print(f"{prec} {n_aux} one sign {one_sign}: {err:.2e} (bound {bound:.2e})")
    assert err <= bound
