"""Weight gradient on the tensor cores where its pieces and K steps end: images
narrower than a segment, a last K step that is not full, a second segment of
four pixels, heights of four rows; pieces that cross images.

1. Against the FP64 oracle backward, under the bar of the other gradient tests.
2. The gradient of four grids against the mean of the four single gradients:
   the mean over a batch scales every BF16 gradient by an exact 1/4, so both
   are sums of the same terms, cut into pieces differently.  A piece adds at
   most 64 groups of 16 terms one after the other in FP32 here, 64 * 2^-24 =
   4e-6 of the sum of the terms' magnitudes; with a hundredfold cancellation
   4e-4 of the largest entry, bar 1e-3.  A row counted twice or left out is
   worth a few percent."""
import numpy as np
import pytest

import oracle
from oracle import cnn as C
from paper_2109_09363_gb300 import workloads as W
from test_gpu_train import oracle_gradient

pytestmark = pytest.mark.gpu
torch = pytest.importorskip("torch")
hp = pytest.importorskip("paper_2109_09363_gb300")

SIZES = [(4, 32), (12, 36), (8, 132), (4, 260)]


@pytest.fixture(scope="module")
def dev():
    if not torch.cuda.is_available():
        pytest.skip("no CUDA device")
    from paper_2109_09363_gb300 import build
    build.build()
    oracle.build()
    return torch.device("cuda:0")


def inputs(dev, B, ny, nx):
    n = max(ny, nx)
    u, v, fl = W.training_case(B, n, 900 + nx)
    t = lambda a, dt: torch.from_numpy(np.ascontiguousarray(a, dt)).to(dev)  # noqa: E731
    f = t(fl[:, :ny, :nx], np.uint8)
    div = hp.hp_divergence(t(u[:, :ny, :nx + 1], np.float32), t(v[:, :ny + 1, :nx], np.float32), f)
    tgt = np.random.default_rng(nx).standard_normal((B, ny, nx))
    return div, f, t(tgt, np.float32)


def params_of(arch):
    rng = np.random.default_rng(3)
    return [(w, 0.05 * rng.standard_normal(b.shape)) for w, b in C.init_params(17, arch)]


def gradient(params, arch, div, f, tgt):
    B, ny, nx = f.shape
    cnn = hp.CNN(B, ny, nx, params=C.flatten(params), arch=arch)
    g, _ = hp.Trainer(cnn, B, ny, nx).gradient(div, f, tgt, lambda_div=1.0)
    phi, s = hp.hp_cnn_forward(cnn, div, f)
    torch.cuda.synchronize()
    cnn.check()
    return g.cpu().numpy().astype(np.float64), phi, s


@pytest.mark.parametrize("ny,nx", SIZES)
def test_edges_match_oracle_backward(dev, ny, nx):
    params = params_of("monoscale")
    div, f, tgt = inputs(dev, 1, ny, nx)
    flat, phi, s = gradient(params, "monoscale", div, f, tgt)
    args = [x.cpu().numpy() for x in (phi, div, f, tgt)] + [[float(x) for x in s.cpu()], 1.0]
    _, ref = oracle_gradient(params, *args, act_round=C.round_bf16)
    _, ref64 = oracle_gradient(params, *args, act_round=None)
    k = 0
    for (w, b), (w64, b64) in zip(ref, ref64):
        r, r64 = (np.concatenate([a.ravel(), c.ravel()]) for a, c in ((w, b), (w64, b64)))
        bar = max(5e-2 * np.abs(r).max(), 3.0 * np.abs(r - r64).max()) + 1e-9
        assert np.abs(flat[k:k + r.size] - r).max() <= bar, k
        k += r.size


@pytest.mark.parametrize("arch,scale", [("monoscale", 1), ("smallscale", 4)])
@pytest.mark.parametrize("ny,nx", SIZES)
def test_pieces_across_images(dev, arch, scale, ny, nx):
    ny, nx = ny * scale, nx * scale  # the coarsest branch at the size
    params = params_of(arch)
    div, f, tgt = inputs(dev, 4, ny, nx)
    both, _, _ = gradient(params, arch, div, f, tgt)
    mean = sum(gradient(params, arch, *(x[b:b + 1].contiguous() for x in (div, f, tgt)))[0]
               for b in range(4)) / 4
    k = 0
    for w, b in params:
        n = w.size + b.size
        m = mean[k:k + n]
        assert np.abs(both[k:k + n] - m).max() <= 1e-3 * np.abs(m).max(), k
        k += n
