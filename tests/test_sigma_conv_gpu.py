"""The Sigma_c term of one q (contraction, frequency convolution split over bands) against the oracle
for frequency counts from one to more than a block's share, few and many (k, band) pairs."""
import numpy as np
import pytest

from oracle import gw_oracle as O
from paper_2011_01400_gb300.synth import make_system

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("n_freq", [1, 7, 33, 129, 200, 256])
@pytest.mark.parametrize("prec", ["fp64", "3xfp16"])
def test_sigma_term(n_freq, prec):
    torch = pytest.importorskip("torch")
    from paper_2011_01400_gb300 import gw
    s = make_system("tiny", seed=5, n_freq=n_freq, head_wings=0)
    rng = np.random.default_rng(n_freq)
    w = rng.standard_normal((n_freq, s.n_aux, s.n_aux)) + 1j * rng.standard_normal((n_freq, s.n_aux, s.n_aux))
    w = -(w @ np.conj(w.transpose(0, 2, 1))) / s.n_aux
    # W^c falls off as 1/w^2 (a W that does not would weigh the cancellation of z^2 + w'^2 at w = w' >> 1, in the
    # oracle's 64 bits too)
    w /= (1.0 + O.freq_grid(n_freq, s.omega0)[0] ** 2)[:, None, None]
    pb = gw.Problem(s, prec)
    plan = gw.gw_plan_create(pb.prob)
    try:
        acc = torch.zeros((s.n_k, s.sigma_hi - s.sigma_lo, n_freq), dtype=torch.complex128, device="cuda")
        gw.gw_sigma_ext(plan, 0, 1, torch.from_numpy(np.ascontiguousarray(w)).cuda(), 0, s.n_k, acc)
        acc = acc.cpu().numpy()
        om, g = gw.gw_plan_freq(plan, n_freq)   # (node by node the two Gauss-Legendre grids differ by 1e-11 at large w)
    finally:
        gw.gw_plan_destroy(plan)
    ref = O.sigma_q(s, 1, w, om, g, O.mu_midgap(s))
    # split: two BF16 pieces per operand (2^-16 of the products) and FP32 sums over bands and frequencies
    tol = 1e-12 if prec == "fp64" else 4.0 * 2.0 ** -16
    assert np.linalg.norm(acc - ref) <= tol * np.linalg.norm(ref)
