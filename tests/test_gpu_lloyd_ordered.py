"""The Lloyd update over points ordered by label (kpp_lloyd_step from 200 000
points, or many features or centres): integer coordinates bit-identical to the
oracle's step at the edges of its lanes-per-row variants, with one centre,
empty centres and a partial last batch; on mixtures the same labels, counts
and, within FP32 rounding, D^2 and centres as the direct update (which a
workspace without the point order still runs)."""
import numpy as np
import pytest
import torch

import oracle
import paper_1908_02136_gb300 as kpp
from paper_1908_02136_gb300 import datagen

pytestmark = pytest.mark.gpu

DEV = "cuda:0"


def _step(x, C, spare=0):
    """One step through the C entry point; `spare` bytes of the workspace withheld."""
    N, d = x.shape
    K = C.shape[0]
    ll = kpp.Lloyd(x, K)
    outs = (torch.empty(N, dtype=torch.int32, device=DEV), torch.empty(N, device=DEV),
            torch.empty_like(C), torch.empty(K, dtype=torch.int64, device=DEV),
            torch.empty(1, dtype=torch.float64, device=DEV))
    lab, d2, C2, cnt, phi = outs
    st = kpp.kpp_lloyd_step(x.data_ptr(), N, d, C.data_ptr(), K, lab.data_ptr(), d2.data_ptr(),
                            C2.data_ptr(), cnt.data_ptr(), phi.data_ptr(), ll.ws.data_ptr(),
                            ll.ws.numel() - spare, None)
    assert st == kpp.OK
    assert kpp.kpp_read_status(ll.ws.data_ptr(), None) == kpp.OK
    return [t.cpu().numpy() for t in outs]


@pytest.mark.parametrize("N,d,K", [(200_000, 1, 7), (200_001, 4, 16), (200_003, 5, 33),
                                   (200_031, 8, 1), (200_033, 9, 64), (200_000, 16, 100),
                                   (200_017, 17, 20), (250_007, 32, 5), (200_511, 33, 40),
                                   (160_001, 64, 300), (200_000, 65, 12), (110_001, 96, 50),
                                   (110_000, 97, 9), (110_003, 128, 77), (9_000, 128, 2000)])
def test_integer_points_equal_the_oracle(N, d, K):
    x = datagen.integer_points(N, d, seed=N + d, n_comp=8)
    C = x[np.random.default_rng(d).choice(N, size=K, replace=False)].astype(np.float32)
    if K > 4:
        C[K // 2] = 1000.0  # a centre no point chooses
    lab, d2, C2, cnt, phi = _step(torch.from_numpy(x).to(DEV), torch.from_numpy(C).to(DEV))
    ref = oracle.lloyd_step(x, C.astype(np.float64))
    assert np.array_equal(lab, ref["labels"])
    assert np.array_equal(cnt, ref["counts"])
    assert np.array_equal(d2, ref["d2"].astype(np.float32))
    assert phi[0] == ref["d2"].sum()
    assert np.array_equal(C2, ref["centres"].astype(np.float32))


@pytest.mark.parametrize("N,d,K", [(200_003, 3, 50), (200_003, 40, 256), (300_007, 100, 300)])
def test_ordered_and_direct_updates_agree(N, d, K):
    x = torch.from_numpy(datagen.gmm(N, d, K, seed=N)).to(DEV)
    C = x[:K].clone()
    a, b = _step(x, C), _step(x, C, spare=4 * N)
    assert np.array_equal(a[0], b[0]) and np.array_equal(a[3], b[3])
    # each is a sum of d squares, rounded d + 1 times at most
    np.testing.assert_allclose(a[1], b[1], rtol=2 * (d + 1) * 2.0**-24)
    np.testing.assert_allclose(a[2], b[2], rtol=1e-5, atol=1e-5 * float(x.abs().max()))
    assert a[4][0] == pytest.approx(b[4][0], rel=1e-6)
