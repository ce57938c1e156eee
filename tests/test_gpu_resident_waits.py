"""Bounded waits of the grid-resident sweeps made to run out (one poll each:
no message between SMs, and no sum of several sweeps, arrives within it): the
kernel returns, hp_ctx_check reports it, the outputs are marked (-1 sweeps, not
converged, NaN in every field), and the next call is right again.
Strips with one and with several columns, grids of one CTA, more grids than
fit at once, a fixed count and a stop with a replay."""
import pytest

from test_gpu_resident_strips import case, dev  # noqa: F401

pytestmark = pytest.mark.gpu
torch = pytest.importorskip("torch")
hp = pytest.importorskip("paper_2109_09363_gb300")

SHAPES = [(1, 512, 512), (40, 300, 256), (200, 64, 128), (2, 300, 600), (12, 200, 1000)]


def project(ctx, u, v, fl, **kw):
    a, b = u.clone(), v.clone()
    o = hp.hp_project(ctx, a, b, fl, hp.ProjectParams(**kw), hist_len=kw.get("max_iters", 0))
    torch.cuda.synchronize()
    return dict(o, u=a, v=b)


@pytest.mark.parametrize("kw", [dict(threshold=2e-3, max_iters=400), dict(fixed_iters=41)])
@pytest.mark.parametrize("shape", SHAPES)
def test_waits_that_run_out_return_and_are_reported(dev, shape, kw):  # noqa: F811
    u, v, fl = case(*shape, dev)
    ctx = hp.Context(*shape)
    ref = project(ctx, u, v, fl, **kw)
    ctx.check()
    # a fixed count of grids of one CTA waits for nothing
    waits = "threshold" in kw or shape != (200, 64, 128)
    ctx.set_wait_limit(1)
    for _ in range(3):
        void = project(ctx, u, v, fl, **kw)
        if waits:
            assert (void["iters"] == -1).all() and (void["converged"] == 0).all()
            for k in set(ref) - {"iters", "converged"}:
                assert torch.isnan(void[k]).all(), k
            with pytest.raises(hp.HprojError, match="status 7"):
                ctx.check()
    ctx.set_wait_limit(0)
    got = project(ctx, u, v, fl, **kw)
    ctx.check()
    for k in ref:
        assert torch.equal(torch.nan_to_num(ref[k]), torch.nan_to_num(got[k])), k
    # outputs that carry no counts: the sweeps by themselves
    div = torch.randn(shape, generator=torch.Generator().manual_seed(3)).to(dev)
    phi = torch.zeros(shape, device=dev)
    ctx.set_wait_limit(1)
    if shape != (200, 64, 128):
        assert torch.isnan(hp.hp_jacobi_sweeps(ctx, phi, div, fl, 41)).all()
