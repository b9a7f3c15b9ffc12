"""A kernel's shared-memory limit belongs to the kernel, not to a call: launches
go through while another thread keeps planning calls of the same kernel that
need less."""
import threading

import pytest
import torch

import paper_1908_02136_gb300 as kpp

pytestmark = pytest.mark.gpu

DEV = "cuda:0"


def _while_planning(plan, call, n):
    """Runs `call` n times while another thread repeats `plan`."""
    stop = threading.Event()

    def loop():
        with torch.cuda.device(DEV):
            while not stop.is_set():
                plan()

    t = threading.Thread(target=loop)
    t.start()
    try:
        for i in range(n):
            call()
            if i % 50 == 49:
                torch.cuda.synchronize()
    finally:
        stop.set()
        t.join()
    torch.cuda.synchronize()


def test_batches_of_many_and_few_centres():
    xs = [torch.randn(2500, 16, device=DEV) for _ in range(2)]
    outs, ws = kpp.seed_batched(xs, [2000, 2000], [1, 1])
    one = (kpp.Problem * 1)()
    one[0] = kpp.Problem(xs[0].data_ptr(), None, 2500, 16, 8, 1, 0, outs[0][0].data_ptr(),
                         outs[0][1].data_ptr(), None)
    _while_planning(lambda: kpp.kpp_batch_workspace_size(one, 1, kpp.F32),
                    lambda: kpp.seed_batched(xs, [2000, 2000], [1, 1], workspace=ws, outs=outs,
                                             check=False), 200)


# the small form; the persistent form reading every row, and skipping rows
@pytest.mark.parametrize("N,d,K,less", [(9000, 4, 4, 900), (200_000, 16, 4, 70_000),
                                        (200_000, 16, 40, 70_000)])
def test_seedings_of_large_and_small_sets(N, d, K, less):
    x = torch.randn(N, d, device=DEV)
    ws = kpp.workspace_for(N, d, K, kpp.F32, x.device)
    out = kpp.seed(x, K, 1, workspace=ws)
    _while_planning(lambda: kpp.kpp_workspace_size(less, d, K, kpp.F32),
                    lambda: kpp.seed(x, K, 1, workspace=ws, out=out, check=False), 2000)
