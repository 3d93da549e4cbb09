"""The library's workspace pool: it keeps at most 1/16 of the device's memory
between calls, hands it back on request, and serves several threads with
streams of their own at a time."""

import threading

import pytest
import torch

from paper_1805_10121_gb300 import chase
from tests.test_gpu_rns import DEV, gauss, hermitian

pytestmark = pytest.mark.gpu


@pytest.fixture(scope="module", autouse=True)
def _lib():
    from paper_1805_10121_gb300 import build
    build.build()
    chase.lib()


def test_memory_is_bounded_and_given_back():
    h, v = hermitian(3000, 1, False), gauss(3000, 40, 2, False).clone()
    chase.chase_release_workspace()
    torch.cuda.synchronize()
    before, total = torch.cuda.mem_get_info()
    chase.chase_filter(h, v, [4] * 40, 1.6, -1.5, -0.9)
    torch.cuda.synchronize()
    kept = before - torch.cuda.mem_get_info()[0]
    assert 0 < kept <= total // 16
    chase.chase_release_workspace()
    assert before - torch.cuda.mem_get_info()[0] <= 64 << 20


def test_threads_on_their_own_streams():
    n, b = 700, 30
    hs = [hermitian(n, 10 + i, False) for i in range(4)]
    vs = [gauss(n, b, 20 + i, False).clone() for i in range(4)]
    want = [chase.chase_filter(h, v.clone(), [8] * b, 1.6, -1.5, -0.9) for h, v in zip(hs, vs)]
    got = [[v.clone() for _ in range(3)] for v in vs]
    torch.cuda.synchronize()

    def work(i):
        s = torch.cuda.Stream(DEV)
        for x in got[i]:
            chase.chase_filter(hs[i], x, [8] * b, 1.6, -1.5, -0.9, stream=s.cuda_stream)
        s.synchronize()

    ts = [threading.Thread(target=work, args=(i,)) for i in range(4)]
    for t in ts:
        t.start()
    for t in ts:
        t.join()
    for i in range(4):
        for x in got[i]:
            assert torch.equal(x, want[i])
