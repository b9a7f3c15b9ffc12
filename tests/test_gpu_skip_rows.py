"""The persistent and batched passes that skip rows the new centre cannot bring
nearer (triangle inequality): indices and D^2 bit-identical to the streamed
form, which reads every row, over sizes at the edges of warps, blocks and the
list of rows, both homes of D^2, every stored type, and data at the ends of
the FP32 range; and the bound itself in NumPy FP32."""
import numpy as np
import pytest
import torch

import paper_1908_02136_gb300 as kpp
from paper_1908_02136_gb300 import datagen

DEV = "cuda:0"


def _stored(x, dtype):
    t = torch.from_numpy(x).to(DEV)
    if dtype == "f32":
        return t, None
    if dtype == "bf16":
        return kpp.quantize(t, "bf16"), None
    return kpp.quantize(t, "fp8")


def _both(x, K, dtype="f32", seed=5, opts=None, forced=None, workspace=None):
    q, s = _stored(x, dtype)
    kw = dict(dtype=dtype, row_scales=s, forced=forced, check=False)
    ref = kpp.seed(q, K, seed, opts={"form": kpp.FORM_STREAMED}, **kw)
    out = kpp.seed(q, K, seed, opts={"form": kpp.FORM_PERSISTENT, "smem_cache": -1, **(opts or {})},
                   workspace=workspace, **kw)
    torch.cuda.synchronize()
    return ref, out


def _same(ref, out):
    assert torch.equal(ref[0], out[0])
    assert torch.equal(ref[1].view(torch.int32), out[1].view(torch.int32))
    a, b = float(ref[2][0]), float(out[2][0])
    assert a == b or abs(a - b) <= 1e-13 * abs(a) or (np.isnan(a) and np.isnan(b)) or a == b


# in shared memory (the default block) and in the output array (70 000-row blocks)
@pytest.mark.gpu
@pytest.mark.parametrize("rows", [0, 70_000])
@pytest.mark.parametrize("dtype,d", [("f32", 8), ("f32", 16), ("f32", 32), ("f32", 64), ("f32", 128),
                                     ("bf16", 8), ("bf16", 32), ("bf16", 128), ("fp8", 16),
                                     ("fp8", 64), ("fp8", 128)])
@pytest.mark.parametrize("N", [2047, 4097, 70_001])
def test_same_as_reading_every_row(N, dtype, d, rows):
    x = datagen.gmm(N, d, 24, seed=N + d, outlier_frac=0.05)
    _same(*_both(x, 40, dtype, opts={"min_rows_per_cta": rows}))


@pytest.mark.gpu
@pytest.mark.parametrize("N", [1, 31, 33, 511, 513, 16 * 256 - 1, 16 * 256 + 1])
def test_edges_of_the_list(N):
    x = datagen.gmm(N, 32, 4, seed=N)
    K = min(N, 12)
    _same(*_both(x, K))
    _same(*_both(x, K, opts={"min_rows_per_cta": 70_000}))


@pytest.mark.gpu
@pytest.mark.parametrize("scale", [1e-30, 1e-22, 1e-19, 1.0, 1e17, 3e18, 1e19])
def test_ends_of_the_fp32_range(scale):
    x = (datagen.gmm(9001, 32, 12, seed=3) * np.float32(scale)).astype(np.float32)
    x[7] = 0.0
    x[100:140] = x[99]  # duplicates
    # the seeds are given: where D^2 overflows, a sum is infinite and the two
    # forms' draws, which scan it differently, part
    forced = np.random.default_rng(1).integers(0, len(x), size=20).tolist()
    ref, out = _both(x, 20, forced=forced)
    assert torch.equal(ref[1].view(torch.int32), out[1].view(torch.int32))


@pytest.mark.gpu
def test_infinities_and_nan_are_read():
    x = datagen.gmm(6000, 16, 8, seed=4)
    x[17, 3] = np.inf
    x[4000, 0] = np.nan
    forced = list(range(100, 110)) + [17, 4000] + list(range(200, 210))
    ref, out = _both(x, len(forced), forced=forced)
    assert torch.equal(ref[1].isnan(), out[1].isnan())
    keep = ~ref[1].isnan()
    assert torch.equal(ref[1][keep], out[1][keep])


@pytest.mark.gpu
def test_more_centres_than_have_bounds():
    x = datagen.gmm(30_000, 16, 64, seed=6)
    _same(*_both(x, 2200))
    _same(*_both(x, 2200, opts={"min_rows_per_cta": 70_000}))


@pytest.mark.gpu
def test_workspace_without_labels_reads_every_row():
    x = datagen.gmm(150_000, 16, 32, seed=7)
    opts = {"form": kpp.FORM_PERSISTENT, "smem_cache": -1, "min_rows_per_cta": 70_000}
    st, plan = kpp.kpp_describe(150_000, 16, 40, kpp.F32, opts)
    need = kpp.kpp_workspace_size(150_000, 16, 40, kpp.F32, opts)
    assert st == kpp.OK and need > plan.workspace_bytes
    ws = torch.empty(plan.workspace_bytes, dtype=torch.uint8, device=DEV)
    _same(*_both(x, 40, opts=opts, workspace=ws))


@pytest.mark.gpu
def test_batch_equals_single_seedings():
    xs = [datagen.gmm(N, d, 16, seed=N) for N, d in [(1000, 8), (5001, 32), (40_000, 32), (2500, 128)]]
    Ks = [40, 7, 33, 64]
    ts = [torch.from_numpy(x).to(DEV) for x in xs]
    outs, ws = kpp.seed_batched(ts, Ks, [9] * 4)
    small = torch.empty(ws.numel() - 80_000, dtype=torch.uint8, device=DEV)  # no room for labels
    plain, _ = kpp.seed_batched(ts, Ks, [9] * 4, workspace=small)
    for t, K, p, a, b in zip(ts, Ks, range(4), outs, plain):
        ref = kpp.seed(t, K, 9, p, opts={"form": kpp.FORM_STREAMED})
        for o in (a, b):
            assert torch.equal(ref[0], o[0]) and torch.equal(ref[1], o[1])


def test_bound_never_skips_a_nearer_row():
    """prune_bound in FP32: wherever D^2 <= bound(|c - a|^2), the new FP32
    distance is not below D^2 -- points placed near the bound's surface."""
    rng = np.random.default_rng(0)
    f = np.float32

    def sq(a, b):  # FP32 difference form, sequential over the features
        s = np.zeros(a.shape[0], f)
        for j in range(a.shape[1]):
            t = (a[:, j] - b[:, j]).astype(f)
            s = (s + t * t).astype(f)
        return s

    for d in (1, 2, 16, 128):
        for scale in (1e-18, 1e-3, 1.0, 1e3, 1e18):
            n = 4000
            a = rng.normal(size=(n, d)) * scale
            c = a + rng.normal(size=(n, d)) * scale * 10.0 ** rng.uniform(-4, 2, size=(n, 1))
            # on the segment from a to c, just short of or past its middle
            x = a + (c - a) * (0.5 + rng.normal(size=(n, 1)) * 10.0 ** rng.uniform(-8, -1, size=(n, 1)))
            a, c, x = a.astype(f), c.astype(f), x.astype(f)
            with np.errstate(over="ignore"):
                s2, d2, v = sq(c, a), sq(x, a), sq(x, c)
                bound = np.where(s2 < f(1e37), np.where(s2 < f(1e-30), f(0), s2 * f(0.25 * (1 - 2**-8))),
                                 f(-1))
            skipped = d2 <= bound
            assert not (v[skipped] < d2[skipped]).any()


# any d (the automatic choice; a named form still refuses or streams it): rows
# at every alignment, one chunk to many, the last row ending inside a chunk
@pytest.mark.gpu
@pytest.mark.parametrize("dtype", ["f32", "bf16", "fp8"])
@pytest.mark.parametrize("N,d", [(120_001, 1), (60_001, 3), (40_003, 5), (30_001, 7), (20_011, 12),
                                 (20_001, 15), (20_003, 17), (9_001, 33), (9_003, 50), (5_001, 100),
                                 (5_003, 129), (3_001, 300), (2_500, 784), (601, 4095), (700, 4096)])
def test_any_width_same_as_the_streamed_form(N, d, dtype):
    x = datagen.gmm(N, d, 12, seed=N + d, outlier_frac=0.05)
    q, s = _stored(x, dtype)
    for K in (5, 40):
        ref = kpp.seed(q, K, 3, dtype=dtype, row_scales=s, opts={"form": kpp.FORM_STREAMED})
        for opts in (None, {"min_rows_per_cta": 70_000}):  # D^2 in shared memory / in the output
            _same(ref, kpp.seed(q, K, 3, dtype=dtype, row_scales=s, opts=opts))


@pytest.mark.gpu
@pytest.mark.parametrize("d", [32, 50])
def test_seeding_inside_a_captured_graph(d):
    x = torch.from_numpy(datagen.gmm(60_000, d, 16, seed=d)).to(DEV)
    ref = kpp.seed(x, 24, 3)
    ws = kpp.workspace_for(60_000, d, 24, kpp.F32, x.device)
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
