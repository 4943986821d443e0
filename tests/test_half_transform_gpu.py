"""The lattice sum of the LRI coefficients is taken in FP64 and rounded once: coefficients of opposite lattice vectors
that are 1e4 times larger than their sum leave chi0 of the split precisions as accurate as without them."""
import numpy as np
import pytest

from oracle import gw_oracle as O
from paper_2011_01400_gb300.synth import make_system

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("big", [0.0, 1e4])
@pytest.mark.parametrize("prec", ["3xfp16", "3xbf16", "3xtf32"])
def test_cancelling_lattice_vectors(big, prec):
    torch = pytest.importorskip("torch")
    from paper_2011_01400_gb300 import gw
    s = make_system("cfg0", seed=9, nk=(2, 1, 1), head_wings=0, n_freq=4)
    plus, minus = (next(i for i, r in enumerate(s.R) if tuple(r) == v) for v in ((1, 0, 0), (-1, 0, 0)))
    rng = np.random.default_rng(0)
    for c in s.ctil_R:
        a = big * np.abs(c).mean() * rng.standard_normal(c.shape[1:])
        c[plus] += a                        # e^(2 pi i k.R) = e^(-2 pi i k.R) at k = 0 and 1/2
        c[minus] -= a
    om = O.freq_grid(4)[0]
    ref = O.chi0(s, 1, om)
    pb = gw.Problem(s, prec)
    plan = gw.gw_plan_create(pb.prob)
    try:
        out = torch.empty(ref.shape, dtype=torch.complex128, device="cuda")
        gw.gw_chi0(plan, 0, 1, out)
        out = out.cpu().numpy()
    finally:
        gw.gw_plan_destroy(plan)
    for a, b in zip(out, ref):              # FP32 rows, pieces of 22 bits and more, truncating FP32 sums
        assert np.linalg.norm(a - b) <= 5e-6 * np.linalg.norm(b)
