"""CTA shapes of the mixed-radix passes: a grid whose few transforms get wider
thread groups still takes every shape that fits the narrower ones (cut to the
groups that one CTA holds), from the options and from a tuning cache, and
refuses what those refused."""
import numpy as np
import pytest

torch = pytest.importorskip("torch")
pytestmark = pytest.mark.gpu

if not torch.cuda.is_available():  # pragma: no cover
    pytest.skip("needs a CUDA GPU", allow_module_level=True)

import paper_1109_0286_gb300 as cg  # noqa: E402
from workloads import synth  # noqa: E402

# relative difference of two solutions of the same system, each to the tolerance:
# cond * tol, cond ~ 1e3 for this spectrum without its red end
TOL = {"fp64": 1e-12, "mixed": 1e-11, "fp32": 1e-6}
BOUND = {"fp64": 1e-9, "mixed": 1e-8, "fp32": 1e-3}


@pytest.mark.parametrize("mode", ["fp32", "mixed", "fp64"])
@pytest.mark.parametrize("ny,nx,groups", [(375, 1050, 5), (280, 504, 3)])
def test_shapes_of_narrow_groups(ny, nx, groups, mode, tmp_path):
    rng = np.random.default_rng(3)
    P = synth.spectrum_lorentz_beam(ny, nx, sb=0.8, noise_frac=1e-2)
    obs = np.ones((ny, nx), np.uint8)
    obs[ny // 2 - 5:ny // 2 + 5] = 0
    obs.ravel()[rng.integers(0, ny * nx, 300)] = 0
    m = obs == 0
    dt = torch.float32 if mode == "fp32" else torch.float64
    d = torch.from_numpy(rng.standard_normal((ny, nx))).to(dt).cuda()

    def ml(cache=None, **opts):
        plan = cg.Plan(P, obs, mode=mode, **opts)
        if cache:
            plan.autotune(str(cache))
        x, st = plan.ml(d, TOL[mode])
        assert st[0]["status"] == 0
        plan.close()
        return x.reshape(ny, nx).double().cpu().numpy()[m]

    ref = ml()
    v = 1 if mode == "fp64" else 2
    prec = 1 if mode == "fp64" else 0
    for rows, ffts in ((v, v), (4 * v, 4 * v), (v, 2 * v), (4, groups * v)):
        x = ml(rows_per_cta=rows, ffts_per_cta=ffts)
        assert np.linalg.norm(x - ref) <= BOUND[mode] * np.linalg.norm(ref), (rows, ffts)
    cache = tmp_path / "shape.txt"
    cache.write_text(f"g {prec} {ny} {nx} 1 {4 * v} {4 * v} 0 0\n")
    x = ml(cache)
    assert np.linalg.norm(x - ref) <= BOUND[mode] * np.linalg.norm(ref)
    for opts in ({"rows_per_cta": 64 * v}, {"ffts_per_cta": 64 * v}, {"rows_per_cta": 3 * v}):
        with pytest.raises(Exception):
            cg.Plan(P, obs, mode=mode, **opts)
