"""GPU: masks of scattered pixels -- device memory of a plan and the fills."""
import numpy as np
import pytest

from workloads import synth

torch = pytest.importorskip("torch")
pytestmark = pytest.mark.gpu

if not torch.cuda.is_available():  # pragma: no cover
    pytest.skip("needs a CUDA GPU", allow_module_level=True)

import paper_1109_0286_gb300 as cg  # noqa: E402
from test_gpu_vectors import BOUND, dense_ml  # noqa: E402


@pytest.mark.parametrize("mode,elem", [("fp32", 4), ("fp64", 8), ("mixed", 12)])
def test_plan_memory_follows_the_masked_pixels(mode, elem):
    """Six vectors per precision (FP32 and double-float in mixed mode) of at
    most two values per masked pixel, over a plan with one masked pixel."""
    n = 2048
    P = np.ones((n, n // 2 + 1))
    obs = np.ones((n, n), np.uint8)

    def used(o):
        torch.cuda.synchronize()
        free = torch.cuda.mem_get_info()[0]
        plan = cg.Plan(P, o, mode=mode)
        b = free - torch.cuda.mem_get_info()[0]
        plan.close()
        return b

    obs[5, 7] = 0
    used(obs)
    base = used(obs)
    obs.ravel()[np.random.default_rng(1).choice(n * n, n * n // 20, replace=False)] = 0
    masked = int((obs == 0).sum())
    assert used(obs) - base <= 6 * 2 * masked * elem + 12 * 2 ** 21   # and 2 MB granules


@pytest.mark.parametrize("mode", ["fp64", "mixed", "fp32"])
@pytest.mark.parametrize("precond", [True, False])
@pytest.mark.parametrize("ny,nx", [(16, 64), (45, 70)])
def test_scattered_masks(ny, nx, precond, mode):
    """Every place of a word alone, every second pixel, and a fifth at random."""
    n = ny * nx
    P = synth.spectrum_lorentz_beam(ny, nx, sb=0.8, noise_frac=1e-2)
    d = np.random.default_rng(ny).standard_normal((ny, nx))
    dt = torch.float32 if mode == "fp32" else torch.float64
    tol = {"fp64": 1e-13, "mixed": 1e-11, "fp32": 1e-6}[mode]
    rng = np.random.default_rng(7)
    for masked in (np.arange(0, n, 33), np.arange(0, n, 2), np.arange(1, n, 2),
                   rng.choice(n, n // 5, replace=False)):
        obs = np.ones(n, np.uint8)
        obs[masked] = 0
        obs = obs.reshape(ny, nx)
        plan = cg.Plan(P, obs, mode=mode, precond=precond)
        for _ in range(2):   # the second call starts from used vectors
            x = plan.ml(torch.from_numpy(d).to(dt).cuda(), tol)[0][0].double().cpu().numpy()
        ref = dense_ml(P, obs, d.astype(np.float32).astype(np.float64) if mode == "fp32" else d)
        m = obs == 0
        assert np.linalg.norm(x[m] - ref[m]) <= BOUND[mode] * np.linalg.norm(ref[m])
        plan.close()
