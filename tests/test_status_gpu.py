"""A wait that expired in one stage's products ends in GW_ERR_TIMEOUT, whichever call is the first to look: the status
word is set from the host (GW_INJECT_TIMEOUT) after products that ran to their end; nothing stalls."""
import pytest

from paper_2011_01400_gb300.synth import make_system

torch = pytest.importorskip("torch")
pytestmark = pytest.mark.gpu


@pytest.fixture
def plan_of(monkeypatch):
    from paper_2011_01400_gb300 import gw
    kept = []

    def make(stage, prec="3xfp16"):
        s = make_system("cfg0", seed=1)
        pb = gw.Problem(s, prec)
        monkeypatch.setenv("GW_INJECT_TIMEOUT", stage)
        kept.append((pb, gw.gw_plan_create(pb.prob)))
        return s, kept[-1][1]

    yield make
    for _, plan in kept:
        gw.gw_plan_destroy(plan)


def expect_timeout(plan, call, *args, **kw):
    from paper_2011_01400_gb300 import gw
    with pytest.raises(gw.GwError) as e:
        call(plan, *args, **kw)
    assert e.value.status == gw.GW_ERR_TIMEOUT
    with pytest.raises(gw.GwError) as e:                # and the plan's use ends
        gw.gw_chi0(plan, 0, 0)
    assert e.value.status == gw.GW_ERR_STATE


def test_plan_creation_reports_its_products(plan_of):
    from paper_2011_01400_gb300 import gw
    with pytest.raises(gw.GwError) as e:
        plan_of("sqrt")
    assert e.value.status == gw.GW_ERR_TIMEOUT


@pytest.mark.parametrize("prec", ["3xfp16", "3xtf32"])
def test_screen_reports_its_first_products(plan_of, prec):
    from paper_2011_01400_gb300 import gw
    _, plan = plan_of("eps", prec)
    gw.gw_chi0(plan, 0, 1)
    expect_timeout(plan, gw.gw_screen, 0, 1)


@pytest.mark.parametrize("stage", ["eps", "sigma"])
def test_whole_pass_reports(plan_of, stage):
    from paper_2011_01400_gb300 import gw
    _, plan = plan_of(stage)
    expect_timeout(plan, gw.gw_g0w0, 0)


@pytest.mark.parametrize("ext", [False, True])
@pytest.mark.parametrize("then", ["gw_chi0", "gw_screen", "gw_g0w0", "gw_qp", "gw_qp_static"])
def test_sigma_is_reported_by_the_next_call_that_waits(plan_of, then, ext):
    from paper_2011_01400_gb300 import gw
    s, plan = plan_of("sigma")
    w = torch.empty((s.n_freq, s.n_aux, s.n_aux), dtype=torch.complex128, device="cuda")
    gw.gw_chi0(plan, 0, 1)
    gw.gw_screen(plan, 0, 1, w)
    if ext:
        gw.gw_sigma_ext(plan, 0, 1, w, 0, s.n_k, None)
    else:
        gw.gw_sigma(plan, 0, 1)
    args = {"gw_chi0": (0, 2), "gw_screen": (0, 1), "gw_g0w0": (0,)}
    expect_timeout(plan, getattr(gw, then), *args.get(then, (0, s.n_k, s.sigma_hi - s.sigma_lo)))


def test_without_a_stage_nothing_is_reported(plan_of):
    from paper_2011_01400_gb300 import gw
    s, plan = plan_of("")
    for q in range(2):
        gw.gw_chi0(plan, 0, q)
        gw.gw_screen(plan, 0, q)
        gw.gw_sigma(plan, 0, q)
    gw.gw_qp(plan, 0, s.n_k, s.sigma_hi - s.sigma_lo)
