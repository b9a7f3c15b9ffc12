"""Batches that mix problems whose passes skip rows with problems that read
every row (few seeds, narrow rows, no room for labels): the indices and D^2 of
the single seedings, in every stored type."""
import pytest
import torch

import paper_1908_02136_gb300 as kpp
from paper_1908_02136_gb300 import datagen

pytestmark = pytest.mark.gpu

DEV = "cuda:0"
# (N, d, K): teams and single CTAs, K on both sides of 8, rows on both sides of 16 bytes
SIZES = [(60_000, 64, 4), (30_011, 64, 200), (9_000, 2, 40), (2_500, 4, 7), (45_001, 32, 8),
         (120_001, 128, 5), (1_000, 16, 64), (70_000, 8, 100)]


@pytest.mark.parametrize("dtype", ["f32", "bf16", "fp8"])
@pytest.mark.parametrize("labels", [True, False])
def test_equal_to_single_seedings(dtype, labels):
    xs, scales = [], []
    for N, d, K in SIZES:
        x, s = torch.from_numpy(datagen.gmm(N, d, 16, seed=N)).to(DEV), None
        if dtype == "bf16":
            x = kpp.quantize(x, dtype)
        elif dtype == "fp8":
            x, s = kpp.quantize(x, dtype)
        xs.append(x)
        scales.append(s)
    Ks = [K for _, _, K in SIZES]
    kw = {"dtype": dtype, "row_scales": scales if dtype == "fp8" else None}
    outs, ws = kpp.seed_batched(xs, Ks, [9] * len(Ks), **kw)
    if not labels:
        ws = torch.empty(ws.numel() - 2 * max(N for N, _, _ in SIZES) // 4, dtype=torch.uint8,
                         device=DEV)
        outs, _ = kpp.seed_batched(xs, Ks, [9] * len(Ks), workspace=ws, **kw)
    for p, (x, s, K, out) in enumerate(zip(xs, scales, Ks, outs)):
        ref = kpp.seed(x, K, 9, p, dtype=dtype, row_scales=s, opts={"form": kpp.FORM_STREAMED})
        assert torch.equal(ref[0], out[0]) and torch.equal(ref[1], out[1])
