"""Infinite coordinates and sums beyond the FP32 range in the Lloyd update: the
update over points ordered by label gives the infinities (and NaN) of the
direct update, which a workspace without the point order runs."""
import numpy as np
import pytest
import torch

import paper_1908_02136_gb300 as kpp

pytestmark = pytest.mark.gpu

DEV = "cuda:0"


def _means(x, C, spare):
    N, d = x.shape
    K = C.shape[0]
    ll = kpp.Lloyd(x, K)
    lab = torch.empty(N, dtype=torch.int32, device=DEV)
    out = torch.empty_like(C)
    st = kpp.kpp_lloyd_step(x.data_ptr(), N, d, C.data_ptr(), K, lab.data_ptr(), None,
                            out.data_ptr(), None, None, ll.ws.data_ptr(), ll.ws.numel() - spare,
                            None)
    assert st == kpp.OK and kpp.kpp_read_status(ll.ws.data_ptr(), None) == kpp.OK
    return lab.cpu().numpy(), out.cpu().numpy()


@pytest.mark.parametrize("d", [1, 4, 8, 16, 32, 40, 96, 128])
def test_infinities_as_in_the_direct_update(d):
    N, K = 200_003, 5
    rng = np.random.default_rng(d)
    group = np.arange(N) % K
    x = rng.normal(size=(N, d)).astype(np.float32)
    x[:, 0] += 100 * group
    C = np.zeros((K, d), np.float32)
    C[:, 0] = 100 * np.arange(K)
    x[7, -1] = np.inf
    x[11, d // 2] = -np.inf
    x[13] = np.nan
    x[group == 3, -1] = 2e38  # two of them leave the FP32 range
    if d > 1:
        C[3, -1] = 2e38
    x, C = torch.from_numpy(x).to(DEV), torch.from_numpy(C).to(DEV)
    (la, a), (lb, b) = _means(x, C, 0), _means(x, C, 4 * N)
    assert np.array_equal(la, lb)
    assert np.isinf(b).any()
    assert np.array_equal(np.isnan(a), np.isnan(b))
    assert np.array_equal(np.where(np.isinf(a), a, 0), np.where(np.isinf(b), b, 0))
    ok = np.isfinite(b)
    # the direct update adds a centre's values of one CTA (some 300, below 500) in
    # FP32: each mean is off by at most 300 x 500 x 2^-24 = 9e-3
    np.testing.assert_allclose(a[ok], b[ok], rtol=0, atol=1e-2)
