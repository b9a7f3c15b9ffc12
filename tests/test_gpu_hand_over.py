"""Passes that find next to no row to skip hand over to the kernel that reads
every row (where their lists had pushed D^2 out of shared memory): the results
of the streamed form on data without clusters, in clusters, ordered by cluster,
with given seeds and with fewer distinct points than seeds; and the time of the
plan that reads every row where there is nothing to skip."""
import numpy as np
import pytest
import torch

import paper_1908_02136_gb300 as kpp
from paper_1908_02136_gb300 import datagen

pytestmark = pytest.mark.gpu

DEV = "cuda:0"
# D^2 (4.25 bytes a row) fits shared memory alone but not beside the lists
N = 1_900_003


def _points(kind, d, dtype):
    if kind == "clusters":
        x = torch.from_numpy(datagen.gmm(N, d, 64, seed=d)).to(DEV)
    elif kind == "ordered":  # blocks of whole clusters, few of them near the first seeds
        g = torch.Generator(device=DEV)
        g.manual_seed(d)
        x = torch.randn(N, d, generator=g, device=DEV)
        x += (torch.arange(N, device=DEV) * 64 // N * 50).float()[:, None]
    else:
        g = torch.Generator(device=DEV)
        g.manual_seed(d)
        x = torch.randn(N, d, generator=g, device=DEV)
    if dtype == "f32":
        return x, None
    if dtype == "bf16":
        return kpp.quantize(x, "bf16"), None
    return kpp.quantize(x, "fp8")


def _same(x, scales, dtype, K, hands=None, **kw):
    with torch.cuda.device(DEV):
        code = {"f32": kpp.F32, "bf16": kpp.BF16, "fp8": kpp.FP8_E4M3}[dtype]
        st, plan = kpp.kpp_describe(N, x.shape[1], K, code)
        assert st == kpp.OK and plan.form == kpp.FORM_PERSISTENT and not plan.d2_in_smem
        assert plan.rows_per_cta * 4.25 < 200 * 1024
        assert hands is None or plan.launches == 1 + hands
    kw.update(dtype=dtype, row_scales=scales, check=False)
    ref = kpp.seed(x, K, 7, opts={"form": kpp.FORM_STREAMED}, **kw)
    out = kpp.seed(x, K, 7, **kw)
    torch.cuda.synchronize()
    assert torch.equal(ref[0], out[0])
    assert torch.equal(ref[1].view(torch.int32), out[1].view(torch.int32))
    a, b = float(ref[2][0]), float(out[2][0])
    assert a == b or abs(a - b) <= 1e-13 * abs(a)
    return out


# from 20 GB of rows in all passes; the pass that decides is 9, then 17, ... (K / 16)
@pytest.mark.parametrize("kind", ["none", "clusters", "ordered"])
@pytest.mark.parametrize("dtype,d", [("f32", 32), ("f32", 128), ("bf16", 64), ("fp8", 128)])
def test_same_as_the_streamed_form(kind, dtype, d):
    x, scales = _points(kind, d, dtype)
    row = d * {"f32": 4, "bf16": 2, "fp8": 1}[dtype]
    least = int(20e9 / (N * row)) + 1
    for K in (least - 1, least, max(least, 300)):
        _same(x, scales, dtype, K, hands=int(K >= least))


def test_given_seeds_and_exact_draws():
    x, _ = _points("none", 128, "f32")
    K = 30
    forced = np.random.default_rng(2).integers(0, N, size=K).tolist()
    for n in (5, 9, 10, 11, 12, K):
        _same(x, None, "f32", K, hands=1, forced=forced[:n])
    ref = kpp.seed(x, K, 7, opts={"form": kpp.FORM_STREAMED})
    out = kpp.seed(x, K, 7, opts={"exact_draws": 1})
    assert torch.equal(ref[0], out[0]) and torch.equal(ref[1], out[1])


def test_fewer_distinct_points_than_seeds():
    """A degenerate stop before and after the pass that hands over."""
    g = torch.Generator(device=DEV)
    g.manual_seed(1)
    for distinct in (6, 14):
        rows = torch.randn(distinct, 128, generator=g, device=DEV)
        # all but a few points are one row: next to nothing can be skipped for long
        x = rows[0].repeat(N, 1)
        x[5:5 + distinct] = rows
        out = _same(x, None, "f32", 24, hands=1)
        assert int((out[0] == -1).sum()) == 24 - distinct


def test_inside_a_captured_graph():
    x, _ = _points("none", 128, "f32")
    ref = kpp.seed(x, 24, 3)
    with torch.cuda.device(DEV):
        ws = kpp.workspace_for(N, 128, 24, kpp.F32, x.device)
        assert kpp.kpp_describe(N, 128, 24, kpp.F32)[1].launches == 2
    out = tuple(torch.zeros_like(t) for t in ref)
    graph = torch.cuda.CUDAGraph()
    with torch.cuda.graph(graph):
        kpp.seed(x, 24, 3, workspace=ws, out=out, check=False)
    for _ in range(2):
        for t in out:
            t.zero_()
        graph.replay()
        torch.cuda.synchronize()
        for a, b in zip(ref, out):
            assert torch.equal(a, b)


def _ms(x, K, opts):
    with torch.cuda.device(DEV):
        ws = kpp.workspace_for(N, x.shape[1], K, kpp.F32, x.device, opts)
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


def test_no_slower_than_reading_every_row():
    x, _ = _points("none", 64, "f32")
    K = 256
    plain = _ms(x, K, {"form": kpp.FORM_PERSISTENT, "smem_cache": 1 << 30})
    # 17 of 256 passes at up to 1.1 times the plain ones', and 2 % between runs
    assert _ms(x, K, None) <= 1.03 * plain
