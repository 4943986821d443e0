"""FP64 chi0 over many pair rows: the sum is taken in steps of 16 rows, so its rounding grows with the steps and not
with the rows."""
import numpy as np
import pytest

from oracle import gw_oracle as O
from paper_2011_01400_gb300.synth import make_system

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("nk", [(1, 1, 1), (3, 3, 3), (6, 5, 5)])
def test_error_of_long_sums(nk):
    torch = pytest.importorskip("torch")
    from paper_2011_01400_gb300 import gw
    s = make_system("cfg0", seed=2, nk=nk, naux_per_atom=20, n_freq=3, head_wings=0)
    om, q = O.freq_grid(3)[0], s.n_k - 1
    ref = O.chi0(s, q, om)
    pb = gw.Problem(s, "fp64")
    plan = gw.gw_plan_create(pb.prob)
    try:
        out = torch.empty(ref.shape, dtype=torch.complex128, device="cuda")
        gw.gw_chi0(plan, 0, q, out)
        out = out.cpu().numpy()
    finally:
        gw.gw_plan_destroy(plan)
    steps = s.n_k * s.n_occ * (s.n_bands - s.n_occ) / 16
    # additions to a growing sum of one sign (the diagonal): 0.6 u per sqrt(step) rms; the rows of M on both sides and
    # the oracle's own sum: 10 u
    assert np.linalg.norm(out - ref) <= (0.6 * np.sqrt(steps) + 10.0) * 2.0 ** -53 * np.linalg.norm(ref)
