"""The persistent any-d kernel itself: every case's plan is it, with D^2 in
shared memory or in the output array as named, and its indices and D^2 are the
streamed form's, bit for bit -- rows of odd bytes, one chunk to many, points
that begin on a 32-byte boundary and 16 bytes past one."""
import pytest
import torch

import paper_1908_02136_gb300 as kpp
from paper_1908_02136_gb300 import datagen

pytestmark = pytest.mark.gpu

DEV = "cuda:0"
CODES = {"f32": kpp.F32, "bf16": kpp.BF16, "fp8": kpp.FP8_E4M3}
BYTES = {"f32": 4, "bf16": 2, "fp8": 1}


def _at(t, offset):
    """A copy of t that begins `offset` bytes past a 32-byte boundary, the bytes
    around it set."""
    raw = t.contiguous().view(torch.uint8).reshape(-1)
    buf = torch.full((raw.numel() + 128,), 0x7F, dtype=torch.uint8, device=DEV)
    start = (-buf.data_ptr()) % 32 + 32 + offset
    buf[start:start + raw.numel()] = raw
    out = buf[start:start + raw.numel()].view(t.dtype).reshape(t.shape)
    assert out.data_ptr() % 32 == offset
    return out


@pytest.mark.parametrize("offset", [0, 16])
@pytest.mark.parametrize("dtype,d", [("f32", 10), ("f32", 11), ("f32", 17), ("f32", 33), ("f32", 50),
                                     ("f32", 129), ("f32", 784), ("f32", 4095), ("bf16", 20),
                                     ("bf16", 21), ("bf16", 47), ("bf16", 129), ("bf16", 1001),
                                     ("bf16", 4096), ("fp8", 40), ("fp8", 41), ("fp8", 63),
                                     ("fp8", 81), ("fp8", 130), ("fp8", 255), ("fp8", 2049)])
def test_same_as_the_streamed_form(dtype, d, offset):
    # too many for the small form, and a last group that is not whole
    N = 70_001 if d < 100 else (9_003 if d < 1000 else 2_051)
    x, scales = torch.from_numpy(datagen.gmm(N, d, 12, seed=d, outlier_frac=0.05)).to(DEV), None
    if dtype == "bf16":
        x = kpp.quantize(x, dtype)
    elif dtype == "fp8":
        x, scales = kpp.quantize(x, dtype)
    x = _at(x, offset)
    for K in (16, 40) if d * BYTES[dtype] < 80 else (2, 5, 16, 40):
        ref = kpp.seed(x, K, 3, dtype=dtype, row_scales=scales, opts={"form": kpp.FORM_STREAMED})
        for rows in (0, 70_000):
            opts = {"min_rows_per_cta": rows}
            with torch.cuda.device(DEV):
                st, plan = kpp.kpp_describe(N, d, K, CODES[dtype], opts)
                assert st == kpp.OK
                assert plan.form == kpp.FORM_PERSISTENT and plan.lanes_per_row == 0
                assert plan.d2_in_smem == (rows == 0)
                if rows:  # room for the labels
                    assert (kpp.kpp_workspace_size(N, d, K, CODES[dtype], opts) >=
                            plan.workspace_bytes + 2 * N)
                assert kpp.kpp_skips_rows(N, d, K, CODES[dtype], opts) == (K >= 8)
            out = kpp.seed(x, K, 3, dtype=dtype, row_scales=scales, opts=opts)
            assert torch.equal(ref[0], out[0])
            assert torch.equal(ref[1].view(torch.int32), out[1].view(torch.int32))


# data that nothing can be skipped on, for more passes than have bounds to take
@pytest.mark.parametrize("d,K", [(16, 600), (50, 600), (64, 2100)])
def test_no_clusters_and_many_seeds(d, K):
    x = torch.randn(30_000, d, device=DEV)
    ref = kpp.seed(x, K, 3, opts={"form": kpp.FORM_STREAMED})
    opts = {} if d == 50 else {"form": kpp.FORM_PERSISTENT, "smem_cache": -1}
    for rows in (0, 70_000):
        out = kpp.seed(x, K, 3, opts={"min_rows_per_cta": rows, **opts})
        assert torch.equal(ref[0], out[0])
        assert torch.equal(ref[1].view(torch.int32), out[1].view(torch.int32))
