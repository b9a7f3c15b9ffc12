"""Plans and workspaces (host-side planning on a device): which calls are
accepted, and that a workspace sized for one call serves the calls it is
documented for."""
import pytest
import torch

import paper_1908_02136_gb300 as kpp

pytestmark = pytest.mark.gpu

DEV = "cuda:0"


@pytest.fixture(autouse=True)
def on_device():
    kpp.kpp_tune_clear()
    with torch.cuda.device(DEV):
        torch.zeros(1, device=DEV)
        yield


# a d without a specialisation: the persistent any-d kernel has one CTA per SM
@pytest.mark.parametrize("ctas", [2, 5, 8, 32])
@pytest.mark.parametrize("d,K", [(50, 20), (100, 6), (784, 40)])
def test_ctas_per_sm_of_an_automatic_any_d_plan(d, K, ctas):
    N = 100_000
    st, plan = kpp.kpp_describe(N, d, K, kpp.F32, {"ctas_per_sm": ctas})
    assert st == kpp.OK and plan.form == kpp.FORM_STREAMED
    st, streamed = kpp.kpp_describe(N, d, K, kpp.F32,
                                    {"form": kpp.FORM_STREAMED, "ctas_per_sm": ctas})
    assert st == kpp.OK and plan.grid == streamed.grid
    x = torch.randn(N, d, device=DEV)
    ref = kpp.seed(x, K, 3, opts={"form": kpp.FORM_STREAMED})
    out = kpp.seed(x, K, 3, opts={"ctas_per_sm": ctas})
    assert torch.equal(ref[0], out[0]) and torch.equal(ref[1], out[1])
