"""Resident sweeps of two contexts launched by two threads on two streams, with
more strips than the device holds at once, and beside long kernels of another
stream: every launch ends with the result it has by itself, and no wait gives up."""
import threading

import pytest

from test_gpu_resident_strips import case, dev  # noqa: F401

pytestmark = pytest.mark.gpu
torch = pytest.importorskip("torch")
hp = pytest.importorskip("paper_2109_09363_gb300")


@pytest.mark.parametrize("shape", [(1, 512, 512), (16, 512, 512), (1, 700, 1024)])
def test_two_streams_and_other_kernels(dev, shape):  # noqa: F811
    u0, v0, fl = case(*shape, dev)
    prm = hp.ProjectParams(threshold=0.0, max_iters=100)
    ctx = [hp.Context(*shape) for _ in range(2)]
    streams = [torch.cuda.Stream() for _ in range(2)]
    ref = [u0.clone(), v0.clone()]
    hp.hp_project(ctx[0], *ref, fl, prm)
    torch.cuda.synchronize()
    out = [None, None]

    def work(i):
        with torch.cuda.stream(streams[i]):
            for _ in range(20):
                out[i] = [u0.clone(), v0.clone()]
                hp.hp_project(ctx[i], *out[i], fl, prm, stream=streams[i])

    threads = [threading.Thread(target=work, args=(i,)) for i in range(2)]
    for t in threads:
        t.start()
    for t in threads:
        t.join()
    torch.cuda.synchronize()
    a = torch.randn(4096, 4096, device=dev, dtype=torch.bfloat16)
    torch.cuda.synchronize()
    with torch.cuda.stream(streams[0]):
        for _ in range(200):
            a @ a
    beside = [u0.clone(), v0.clone()]
    hp.hp_project(ctx[1], *beside, fl, prm)
    torch.cuda.synchronize()
    for c in ctx:
        c.check()
    for got in out + [beside]:
        assert torch.equal(got[0], ref[0]) and torch.equal(got[1], ref[1])
