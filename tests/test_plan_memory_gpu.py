"""Device memory of a split-precision plan whose matrices over the frequencies dominate: six FP64 ones (chi0, eps~, W^c,
work, tmp, the compressed chi0) and the four 16-bit (FP16, BF16) or 32-bit (TF32) planes of W^c that the contraction
reads."""
import pytest

from paper_2011_01400_gb300.synth import make_system

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("prec,size", [("3xfp16", 2), ("3xbf16", 2), ("3xtf32", 4)])
def test_planes(prec, size):
    torch = pytest.importorskip("torch")
    from paper_2011_01400_gb300 import gw
    n, nw = 512, 64
    s = make_system("cfg0", seed=1, nk=(1, 1, 1), n_freq=nw, n_atoms=1, nb_per_atom=12, naux_per_atom=n, n_bands=12,
                    head_wings=0)
    pb = gw.Problem(s, prec)
    gw.gw_plan_destroy(gw.gw_plan_create(pb.prob))        # the library's own code and tables are on the device
    torch.cuda.synchronize()
    free = torch.cuda.mem_get_info()[0]
    plan = gw.gw_plan_create(pb.prob)
    held = free - torch.cuda.mem_get_info()[0]
    gw.gw_plan_destroy(plan)
    mats, plane = 6 * 16 * nw * n * n, size * nw * n * 2 * n
    assert held <= mats + 4 * plane + 64 * 2 ** 20        # (pieces and tables of one q: 30 MB; a plane: 67 or 134 MB)


def test_allocations_of_a_new_plan():
    """One for the plan's buffers, one for the half transform's staging, three for the work lists of the products; the
    eigenvectors are converted once, into the plan."""
    pytest.importorskip("torch")
    from paper_2011_01400_gb300 import gw
    s = make_system("cfg0", seed=1, head_wings=0, trs=False)
    pb = gw.Problem(s, "3xfp16")
    n = gw.gw_device_allocations()
    plan = gw.gw_plan_create(pb.prob)
    n = gw.gw_device_allocations() - n
    gw.gw_plan_destroy(plan)
    assert n == 5
