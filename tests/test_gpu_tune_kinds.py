"""The autotuner between plans whose passes skip rows and plans that read every
row: on data without clusters, where nothing can be skipped, its choice is not
slower than the plan that reads every row; on clusters not slower than the
automatic one, however few passes it may time."""
import pytest
import torch

import paper_1908_02136_gb300 as kpp
from paper_1908_02136_gb300 import datagen

pytestmark = pytest.mark.gpu

DEV = "cuda:0"


@pytest.fixture(autouse=True)
def clean_table():
    kpp.kpp_tune_clear()
    yield
    kpp.kpp_tune_clear()


def _ms(x, K, opts):
    N, d = x.shape
    with torch.cuda.device(DEV):
        ws = kpp.workspace_for(N, d, K, kpp.F32, x.device, opts)
    out = kpp.seed(x, K, 3, opts=opts, workspace=ws)
    best = float("inf")
    for _ in range(4):
        a, b = torch.cuda.Event(True), torch.cuda.Event(True)
        a.record()
        kpp.seed(x, K, 3, opts=opts, workspace=ws, out=out, check=False)
        b.record()
        b.synchronize()
        best = min(best, a.elapsed_time(b))
    return best


@pytest.mark.parametrize("passes", [4, 16])
def test_choice_on_data_without_clusters(passes):
    N, d, K = 2_000_000, 64, 96
    x = torch.randn(N, d, device=DEV)
    best, _ = kpp.tune(x, K, passes=passes)
    plain = _ms(x, K, {"form": kpp.FORM_PERSISTENT, "smem_cache": 1 << 30})
    # the tuner's own margin is 1 %, runs of one plan differ by another
    assert _ms(x, K, best) <= 1.03 * plain


@pytest.mark.parametrize("passes", [4, 16])
def test_choice_on_clusters(passes):
    N, d, K = 2_000_000, 64, 256
    x = torch.from_numpy(datagen.gmm(N, d, K, seed=1)).to(DEV)
    auto = _ms(x, K, None)
    best, _ = kpp.tune(x, K, passes=passes)
    assert _ms(x, K, best) <= 1.03 * auto


def test_workspace_without_labels_times_plans_that_read_every_row():
    """A workspace that cannot hold the labels skips the plans that keep them."""
    import ctypes

    N, d, K = 2_000_000, 64, 64
    x = torch.from_numpy(datagen.gmm(N, d, K, seed=2)).to(DEV)
    idx = torch.empty(K, dtype=torch.int64, device=DEV)
    d2 = torch.empty(N, dtype=torch.float32, device=DEV)
    ws = torch.empty(1 << 20, dtype=torch.uint8, device=DEV)
    best = kpp.Options()
    with torch.cuda.device(DEV):
        st = kpp.kpp_tune(x.data_ptr(), None, N, d, K, kpp.F32, idx.data_ptr(), d2.data_ptr(),
                          ws.data_ptr(), ws.numel(),
                          ctypes.c_void_p(torch.cuda.current_stream().cuda_stream), 8, best)
        assert st == kpp.OK
        opts = {f: getattr(best, f) for f, _ in kpp.Options._fields_ if f != "reserved"}
        assert kpp.kpp_workspace_size(N, d, K, kpp.F32, opts) <= ws.numel()


@pytest.mark.parametrize("N,d,K,dtype", [(100_003, 50, 64, "f32"), (200_003, 100, 20, "bf16")])
def test_any_d_is_timed_recorded_and_returned(N, d, K, dtype):
    """The persistent any-d kernel, which no form names, takes part: what the
    tuner returns and records is what later automatic calls run."""
    code = {"f32": kpp.F32, "bf16": kpp.BF16}[dtype]
    x = torch.from_numpy(datagen.gmm(N, d, K, seed=d)).to(DEV)
    if dtype == "bf16":
        x = kpp.quantize(x, dtype)
    ref = kpp.seed(x, K, 3, opts={"form": kpp.FORM_STREAMED})
    for _ in range(2):  # a recorded choice does not stand in for the automatic one
        best, ms = kpp.tune(x, K, passes=8)
        with torch.cuda.device(DEV):
            st, plan = kpp.kpp_describe(N, d, K, code, best)
            assert st == kpp.OK
            assert plan.form == kpp.FORM_PERSISTENT and plan.lanes_per_row == 0 and ms > 0
            st, auto = kpp.kpp_describe(N, d, K, code)
            assert st == kpp.OK and auto.as_dict() == plan.as_dict()
    for opts in (best, None):
        out = kpp.seed(x, K, 3, opts=opts)
        assert torch.equal(ref[0], out[0]) and torch.equal(ref[1], out[1])


def test_a_recorded_streamed_choice_stands_for_any_d(tmp_path):
    """A line of the cache file for a d without a specialisation is used as it is."""
    import json
    import os
    import subprocess
    import sys

    root = os.path.dirname(os.path.dirname(os.path.abspath(__file__)))
    N, d, K = 100_003, 50, 64
    p = torch.cuda.get_device_properties(0)
    cache = tmp_path / "tune.txt"
    cache.write_text(f"kpp-tune 1 {p.name.replace(' ', '_')}/{p.multi_processor_count} 0 {d} {N} {K} "
                     f"{kpp.FORM_STREAMED} 0 2 0 0 0 0\n")
    code = ("import json, torch, paper_1908_02136_gb300 as kpp; torch.zeros(1, device='cuda:0');"
            f"st, p = kpp.kpp_describe({N}, {d}, {K}, kpp.F32); print(json.dumps([st, p.form]))")
    r = subprocess.run([sys.executable, "-c", code], capture_output=True, text=True, cwd=root,
                       env=dict(os.environ, KPP_TUNE_CACHE=str(cache)), timeout=300)
    assert r.returncode == 0, r.stderr[-2000:]
    assert json.loads(r.stdout.strip().splitlines()[-1]) == [kpp.OK, kpp.FORM_STREAMED]


def test_more_seeds_than_the_tuner_runs():
    """K = N: the whole seedings that decide stop at 4096 passes."""
    N, d = 20_011, 64
    x = torch.from_numpy(datagen.gmm(N, d, 64, seed=3)).to(DEV)
    best, ms = kpp.tune(x, N, passes=8)
    assert best["form"] in (kpp.FORM_STREAMED, kpp.FORM_PERSISTENT) and ms > 0
