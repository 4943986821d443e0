"""Imaginary frequencies far beyond the transition energies, as a caller's grid may hold them: finite results, those
of the ordinary frequencies as the oracle has them."""
import numpy as np
import pytest

from oracle import gw_oracle as O
from paper_2011_01400_gb300.synth import make_system

pytestmark = pytest.mark.gpu


# the convolution forms products up to w^4: beyond 1e9 they overflow FP32
@pytest.mark.parametrize("far", [9e8, 1e10, 1e13, 3e18])
@pytest.mark.parametrize("prec", ["3xfp16", "3xtf32"])
def test_convolution_with_a_far_frequency(far, prec):
    torch = pytest.importorskip("torch")
    from paper_2011_01400_gb300 import gw
    om, g = np.array([0.4, 3.0, 20.0, far]), np.array([0.4, 2.6, 17.0, 1.0])
    s = make_system("cfg0", seed=3, head_wings=0, n_freq=4)
    w = O.screen(s, 1, O.chi0(s, 1, om), om)[1]
    ref = O.sigma_q(s, 1, w, om, g, O.mu_midgap(s))
    pb = gw.Problem(s, prec, grid=(om, g))
    plan = gw.gw_plan_create(pb.prob)
    try:
        acc = torch.zeros(ref.shape, dtype=torch.complex128, device="cuda")
        d_w = torch.from_numpy(np.ascontiguousarray(w)).cuda()
        gw.gw_sigma_ext(plan, 0, 1, d_w, 0, s.n_k, acc)
        acc = acc.cpu().numpy()
    finally:
        gw.gw_plan_destroy(plan)
    for j in range(4):                          # two pieces per operand (2^-16 of the products at most), FP32 sums
        assert np.linalg.norm(acc[..., j] - ref[..., j]) <= 1e-4 * np.linalg.norm(ref[..., j])


# chi0 falls as 1 / w^2: below 2^-114 the power of two that takes it, or eps~^-1 - 1, to the FP16 range is no finite
# FP32 number. Three frequencies: every weight row is its own; five: the rows go through the frequency compression
@pytest.mark.parametrize("near", [(0.4, 3.0), (0.3, 1.0, 4.0, 20.0)])
@pytest.mark.parametrize("far", [2e17, 4e17, 3e18])
@pytest.mark.parametrize("prec", ["3xfp16", "3xbf16", "3xtf32"])
def test_far_frequency(near, far, prec):
    torch = pytest.importorskip("torch")
    from paper_2011_01400_gb300 import gw
    om = np.array(near + (far,))
    g = np.append(np.diff(np.append(0.0, near)), 1.0)
    s = make_system("cfg0", seed=3, head_wings=0, n_freq=len(om))
    chi = O.chi0(s, 1, om)
    w = O.screen(s, 1, chi, om)[1]
    ref = O.sigma_q(s, 1, w, om, g, O.mu_midgap(s))
    pb = gw.Problem(s, prec, grid=(om, g))
    plan = gw.gw_plan_create(pb.prob)
    try:
        out = torch.empty(chi.shape, dtype=torch.complex128, device="cuda")
        acc = torch.zeros(ref.shape, dtype=torch.complex128, device="cuda")
        gw.gw_chi0(plan, 0, 1)
        gw.gw_screen(plan, 0, 1, out)
        gw.gw_sigma(plan, 0, 1, acc)
        out, acc = out.cpu().numpy(), acc.cpu().numpy()
    finally:
        gw.gw_plan_destroy(plan)
    n = len(near)
    assert np.isfinite(out).all()
    for a, b in zip(out[:n], w[:n]):            # pieces of 22 bits, FP32 sums that truncate
        assert np.linalg.norm(a - b) <= 1e-4 * np.linalg.norm(b)
    assert np.abs(out[n]).max() <= 1e-30
    assert np.linalg.norm(acc[..., :n] - ref[..., :n]) <= 1e-4 * np.linalg.norm(ref[..., :n])
