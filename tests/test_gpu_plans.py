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


# row widths on both sides of every rule of the plans, sets that fit shared
# memory, L2 and neither
@pytest.mark.parametrize("dtype", [kpp.F32, kpp.BF16, kpp.FP8_E4M3])
@pytest.mark.parametrize("d", [2, 8, 10, 14, 19, 32, 33, 50, 70, 100, 128, 300, 785, 2000, 4000])
def test_a_workspace_sized_for_one_K_serves_every_K(d, dtype):
    for N in (1500, 3000, 20_000, 65_000, 300_007, 2_000_000, 9_000_000):
        Ks = [k for k in (1, 4, 7, 8, 15, 16, 20, 100, 1000, 2048, 5000) if k <= N]
        sizes = [kpp.kpp_workspace_size(N, d, K, dtype) for K in Ks]
        for K in Ks:
            st, plan = kpp.kpp_describe(N, d, K, dtype)
            assert st == kpp.OK
            assert min(sizes) >= plan.workspace_bytes, (N, K)


def test_workspace_sized_for_many_seeds_runs_few():
    N, d = 20_000, 14
    x = torch.randn(N, d, device=DEV)
    ws = kpp.workspace_for(N, d, 100, kpp.F32, x.device)
    ref = kpp.seed(x, 5, 3, opts={"form": kpp.FORM_STREAMED})
    out = kpp.seed(x, 5, 3, workspace=ws)
    assert torch.equal(ref[0], out[0]) and torch.equal(ref[1], out[1])


def test_workspace_sized_for_few_seeds_lets_many_skip_rows():
    """The labels of a plan with D^2 in the output array have their room
    whatever K the workspace was sized for."""
    N, d = 4_000_000, 32
    assert (kpp.kpp_workspace_size(N, d, 4, kpp.F32) ==
            kpp.kpp_workspace_size(N, d, 64, kpp.F32) >=
            kpp.kpp_describe(N, d, 64, kpp.F32)[1].workspace_bytes + 2 * N)


# every pass reading every row, without a cache and with one: the plain plans of
# a shape whose automatic plan skips rows
@pytest.mark.parametrize("N,d,dtype", [(300_000, 64, "f32"), (4_000_000, 16, "f32"),
                                       (300_000, 128, "bf16"), (4_000_000, 16, "fp8")])
def test_plans_that_read_every_row_can_be_asked_for(N, d, dtype):
    K = 24
    code = {"f32": kpp.F32, "bf16": kpp.BF16, "fp8": kpp.FP8_E4M3}[dtype]
    lists = 16 * 9216  # at least: the row rings and lists of the passes that skip rows
    st, auto = kpp.kpp_describe(N, d, K, code)
    assert st == kpp.OK and auto.smem_bytes > lists and auto.cached_rows_per_cta == 0
    x, scales = torch.randn(N, d, device=DEV), None
    if dtype == "bf16":
        x = kpp.quantize(x, dtype)
    elif dtype == "fp8":
        x, scales = kpp.quantize(x, dtype)
    ref = kpp.seed(x, K, 3, row_scales=scales, opts={"form": kpp.FORM_STREAMED})
    for cache in (-2, 1 << 30):
        opts = {"form": kpp.FORM_PERSISTENT, "smem_cache": cache}
        st, plan = kpp.kpp_describe(N, d, K, code, opts)
        assert st == kpp.OK
        assert kpp.kpp_workspace_size(N, d, K, code, opts) == plan.workspace_bytes  # no labels
        assert (plan.cached_rows_per_cta > 0) == (cache > 0)
        # D^2 stays in shared memory (4 bytes a row and the chunk sums), or all is empty
        assert plan.d2_in_smem == (plan.rows_per_cta * 4.25 < 220 * 1024)
        out = kpp.seed(x, K, 3, row_scales=scales, opts=opts)
        assert torch.equal(ref[0], out[0]) and torch.equal(ref[1], out[1])


def test_what_a_plan_skips_and_launches():
    """kpp_skips_rows and kpp_lloyd_launches on both sides of their rules."""
    for N, d, K, opts, skips in [(300_000, 64, 24, None, True), (300_000, 64, 7, None, False),
                                 (300_000, 64, 24, {"form": 2, "smem_cache": -2}, False),
                                 (300_000, 2, 24, None, False), (9_000, 2, 24, None, False),
                                 (6_000_000, 8, 100, {"form": 2, "smem_cache": 1 << 30}, False),
                                 (300_000, 50, 24, None, True), (5_000_000, 100, 6, None, False),
                                 (300_000, 64, 24, {"form": kpp.FORM_STREAMED}, False)]:
        assert kpp.kpp_skips_rows(N, d, K, kpp.F32, opts) == skips, (N, d, K, opts)
    assert not kpp.kpp_skips_rows(10, 8, 11, kpp.F32)
    # the update over ordered points: many points, many values, or many centre tiles
    for N, d, K, n in [(199_999, 8, 20, 4), (200_000, 8, 20, 6), (104_166, 96, 50, 4),
                       (104_167, 96, 50, 6), (7_812, 128, 2000, 4), (7_813, 128, 2000, 6)]:
        assert kpp.kpp_lloyd_launches(N, d, K) == n, (N, d, K)
    assert kpp.kpp_lloyd_launches(10, 200, 5) == 0
