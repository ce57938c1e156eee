"""The supervised loss at the sizes where the number of its partial sums changes
(one for every 2,048 cells of a grid, eight at most), against the oracle's loss of
the GPU's own output: FP64 sums of FP32 residuals, bar 1e-4 as for the gradient
tests; a part left out or counted twice is worth a tenth or more."""
import numpy as np
import pytest

from oracle import cnn as C
from oracle import train as TR
from paper_2109_09363_gb300 import workloads as W
from test_gpu_train import dev  # noqa: F401

pytestmark = pytest.mark.gpu
torch = pytest.importorskip("torch")
hp = pytest.importorskip("paper_2109_09363_gb300")


@pytest.mark.parametrize("B,ny,nx", [(70, 16, 16), (2, 44, 44), (2, 32, 64), (2, 64, 64),
                                     (3, 120, 136), (2, 128, 128), (1, 132, 128)])
def test_loss_matches_oracle(dev, B, ny, nx):  # noqa: F811
    rng = np.random.default_rng(ny)
    u, v, fl = W.training_case(min(B, 4), max(ny, nx), 800 + nx)
    take = lambda a, h, w: np.ascontiguousarray(a[np.arange(B) % len(a), :h, :w])  # noqa: E731
    u, v, fl = take(u, ny, nx + 1), take(v, ny + 1, nx), take(fl, ny, nx)
    fd = torch.from_numpy(fl).to(dev)
    div = hp.hp_divergence(torch.from_numpy(u.astype(np.float32)).to(dev),
                           torch.from_numpy(v.astype(np.float32)).to(dev), fd)
    tgt = torch.from_numpy(rng.standard_normal((B, ny, nx)).astype(np.float32)).to(dev)
    cnn = hp.CNN(B, ny, nx, params=C.flatten(C.init_params(5, "monoscale")), arch="monoscale")
    _, loss = hp.Trainer(cnn, B, ny, nx).gradient(div, fd, tgt, lambda_div=1.0)
    phi, s = hp.hp_cnn_forward(cnn, div, fd)
    phi, s, d, t = (x.cpu().numpy() for x in (phi, s, div, tgt))
    ref = np.mean([TR.loss_and_grad(phi[b], t[b], d[b], fl[b], float(s[b]), 1.0)[0]
                   for b in range(B)])
    assert np.isclose(float(loss.item()), ref, rtol=1e-4)
