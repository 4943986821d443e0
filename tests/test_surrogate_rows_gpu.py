"""Loss and gradient of the surrogate network at row counts where the gradient products split their
sum over rows (parts of at least 256 rows, multiples of 16) and at ragged layer widths, against the
FP64 oracle."""
import numpy as np
import pytest

from oracle import surrogate as S
from paper_2011_01400_gb300.synth import surrogate_init

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("rows,dims", [(255, (3, 17, 5)), (513, (12, 64, 48)), (1040, (5, 130, 9)), (4099, (12, 256, 48)),
                                       (9999, (1, 65, 1)), (20000, (16, 200, 33))])
def test_loss_grad_rows(rows, dims):
    torch = pytest.importorskip("torch")
    from paper_2011_01400_gb300 import gw
    rng = np.random.default_rng(rows)
    th = surrogate_init(*dims, seed=rows, out_gain=1.0)
    x = rng.standard_normal((rows, dims[0])).astype(np.float32)
    y = rng.standard_normal((rows, dims[2])).astype(np.float32)
    loss, grad = S.loss_grad(th, dims, x.astype(np.float64), y.astype(np.float64))
    m = gw.gw_surrogate_create(*dims, torch.from_numpy(th).cuda())
    try:
        g = torch.empty(th.size, device="cuda")
        got = gw.gw_surrogate_loss_grad(m, torch.from_numpy(x).cuda(), torch.from_numpy(y).cuda(), g)
    finally:
        gw.gw_surrogate_destroy(m)
    g = g.cpu().numpy().astype(np.float64)
    # fp32 sums of up to rows / parts + parts terms after three layers of up to H: a random walk of that
    # many roundings, with a factor 4
    n = rows + 3 * dims[1]
    tol = 4.0 * np.sqrt(n) * 2.0 ** -24
    assert abs(got - loss) <= tol * loss
    o = 0
    for name, shape in S.layout(*dims):
        k = int(np.prod(shape))
        if name != "s":
            assert np.linalg.norm(g[o:o + k] - grad[o:o + k]) <= tol * max(np.linalg.norm(grad[o:o + k]), 1e-3 * np.linalg.norm(grad)), name
        o += k
