"""GW_SIGMA_CONV64: Sigma_c of a split precision at every frequency of the grid, the largest ones too, where the FP32
convolution cancels."""
import numpy as np
import pytest

from oracle import gw_oracle as O
from paper_2011_01400_gb300.synth import make_system

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("n_freq", [16, 40])
def test_every_frequency(monkeypatch, n_freq):
    torch = pytest.importorskip("torch")
    from paper_2011_01400_gb300 import gw
    s = make_system("cfg0", seed=4, head_wings=0, n_freq=n_freq)
    om, g = O.freq_grid(n_freq, s.omega0)
    w = O.screen(s, 1, O.chi0(s, 1, om), om)[1]
    ref = O.sigma_q(s, 1, w, om, g, O.mu_midgap(s))
    d_w = torch.from_numpy(np.ascontiguousarray(w)).cuda()
    monkeypatch.setenv("GW_SIGMA_CONV64", "1")
    pb = gw.Problem(s, "3xtf32", grid=(om, g))
    plan = gw.gw_plan_create(pb.prob)
    try:
        acc = torch.zeros(ref.shape, dtype=torch.complex128, device="cuda")
        gw.gw_sigma_ext(plan, 0, 1, d_w, 0, s.n_k, acc)
        acc = acc.cpu().numpy()
    finally:
        gw.gw_plan_destroy(plan)
    # TF32 pieces (2^-20 of a product) and truncating FP32 sums of at most 128 terms (2^-17)
    for j in range(n_freq):
        assert np.linalg.norm(acc[..., j] - ref[..., j]) <= (2.0 ** -20 + 2.0 ** -17) * np.linalg.norm(ref[..., j])
