"""GPU: mixed-radix rows in narrow and wide thread groups.  A batch that fills
the chip runs narrow groups where a single map runs wide ones; every map comes
out the same bit for bit."""
import math

import numpy as np
import pytest

from workloads import synth

torch = pytest.importorskip("torch")
pytestmark = pytest.mark.gpu

if not torch.cuda.is_available():  # pragma: no cover
    pytest.skip("needs a CUDA GPU", allow_module_level=True)

import paper_1109_0286_gb300 as cg  # noqa: E402


def case(ny, nx):
    P = synth.spectrum_cmb_like(ny, nx, 2 * math.pi / max(ny, nx))
    obs = synth.mask_band_discs(ny, nx, max(1, ny // 10), 8, 2.0, 5.0, 3)
    return P, obs, np.random.default_rng(3).standard_normal((ny, nx))


@pytest.mark.parametrize("precond", [True, False])
@pytest.mark.parametrize("ny,nx,mode,batch", [(50, 900, "fp32", 80), (49, 900, "fp32", 80),
                                              (280, 504, "fp32", 16), (60, 700, "fp64", 24),
                                              (45, 1050, "mixed", 96)])
def test_batches_equal_single_maps(ny, nx, mode, batch, precond):
    P, obs, d = case(ny, nx)
    dg = torch.from_numpy(d).to(torch.float32 if mode == "fp32" else torch.float64).cuda()
    seeds = list(range(11, 11 + batch))
    many = cg.Plan(P, obs, mode=mode, batch=batch, precond=precond, max_iter=25)
    x, st = many.realize(dg, seeds, 1e-6, check=False)
    one = cg.Plan(P, obs, mode=mode, precond=precond, max_iter=25)
    for i in (0, 1, batch // 2, batch - 1):
        y, s1 = one.realize(dg, seeds[i:i + 1], 1e-6, check=False)
        assert torch.equal(x[i], y[0]), i
        assert [st[i][k] for k in ("iters", "rel_resid")] == [s1[0][k] for k in ("iters", "rel_resid")]
    r, sr = many.relax(dg, 3)
    q, sq = one.relax(dg, 3)
    assert torch.equal(r[batch - 1], q[0]) and sr[batch - 1]["rel_resid"] == sq[0]["rel_resid"]
    if mode != "mixed":
        return
    plans = [cg.Plan(P, obs, mode=mode, precond=precond, max_iter=25) for _ in range(batch)]
    xs, _ = cg.realize_batch(plans, [dg] * batch, seeds, 1e-6, check=False)
    assert all(torch.equal(xs[i][0], x[i]) for i in range(batch))


@pytest.mark.parametrize("mode,batch", [("fp32", 80), ("fp64", 40)])
def test_rows_per_cta(mode, batch):
    """Every height that narrow groups admit, in a batch and alone."""
    P, obs, d = case(50, 900)
    dg = torch.from_numpy(d).to(torch.float32 if mode == "fp32" else torch.float64).cuda()
    ref = None
    for rows in (2, 4, 8) + ((16,) if mode == "fp32" else ()):
        for b in (batch, 1):
            plan = cg.Plan(P, obs, mode=mode, batch=b, rows_per_cta=rows, max_iter=10)
            x = plan.realize(dg, list(range(1, b + 1)), 1e-6, check=False)[0][0].clone()
            plan.close()
            ref = x if ref is None else ref
            assert torch.equal(x, ref), (rows, b)
