"""The hybrid projection on grids wider than 512 cells when it stops within
eight sweeps, that is before the strips have exchanged their copied columns: a
strip reads cells of the guess that its neighbour owns, which must still be the
guess when the neighbour already stores its result.  Against the blocked kernel
(one update, one order: every bit must agree), with many more grids than the
SMs hold at once, so that the CTAs of a group start at different times."""
import pytest

from paper_2109_09363_gb300 import training as T
from test_gpu_resident_strips import case, dev  # noqa: F401

pytestmark = pytest.mark.gpu
torch = pytest.importorskip("torch")
hp = pytest.importorskip("paper_2109_09363_gb300")


@pytest.mark.parametrize("shape", [(1, 304, 1024), (1, 128, 2048), (70, 64, 1040)])
def test_early_stops_match_blocked_kernel(dev, shape):  # noqa: F811
    B = shape[0]
    u, v, fl = case(*shape, dev)
    cnn = hp.CNN(*shape, params=T.init_params(2, "monoscale"), arch="monoscale")
    ctx = [hp.Context(*shape) for _ in range(2)]

    def project(c, kernel, **kw):
        a, b = u.clone(), v.clone()
        o = hp.hp_project_hybrid(c, cnn, a, b, fl, hp.ProjectParams(sweep_kernel=kernel, **kw))
        c.check()
        return dict(o, u=a, v=b)

    hist = hp.hp_project_hybrid(ctx[0], cnn, u.clone(), v.clone(), fl,
                                hp.ProjectParams(0.0, 9, sweep_kernel=2), hist_len=10)["e_hist"]
    e = hist.max(dim=0).values.cpu().tolist()
    for kw in [dict(fixed_iters=n) for n in range(1, 10)] + [
            dict(threshold=0.5 * (e[k - 1] + e[k]), max_iters=300) for k in range(1, 10)]:
        ref = project(ctx[0], 2, **kw)
        if "threshold" in kw:
            assert int(ref["iters"].max()) <= 9
        for _ in range(1 if B > 1 else 20):
            got = project(ctx[1], 0, **kw)
            for k in ref:
                assert torch.equal(ref[k], got[k]), (k, kw)
    assert cnn.check() == 0
