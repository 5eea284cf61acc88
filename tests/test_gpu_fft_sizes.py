"""GPU: every power-of-two transform length (each number of elements per
thread and leading radix of the register FFTs), and the CTA shapes that the
options may ask for."""
import math

import numpy as np
import pytest

from workloads import synth

torch = pytest.importorskip("torch")
pytestmark = pytest.mark.gpu

if not torch.cuda.is_available():  # pragma: no cover
    pytest.skip("needs a CUDA GPU", allow_module_level=True)

import paper_1109_0286_gb300 as cg  # noqa: E402

# bounds of the operator parity tests
BOUND = {"fp64": 1e-12, "mixed": 1e-11, "fp32": 2e-6}


def grid(ny, nx):
    P = synth.spectrum_cmb_like(ny, nx, 2 * math.pi / max(ny, nx))
    obs = synth.mask_band_discs(ny, nx, max(1, ny // 8), 3, 1.5, 3.0, ny + nx)
    x = np.random.default_rng(ny * nx).standard_normal((ny, nx))
    return P, obs, x


@pytest.mark.parametrize("mode", ["fp64", "mixed", "fp32"])
@pytest.mark.parametrize("log", range(5, 14))
def test_every_transform_length(log, mode):
    dt = torch.float32 if mode == "fp32" else torch.float64
    for ny, nx in ((16, 1 << log), (1 << (log if log > 5 else 4), 32), (1 << log, 64)):
        P, obs, x = grid(ny, nx)
        plan = cg.Plan(P, obs, mode=mode)
        got = plan.apply(0, torch.from_numpy(x).to(dt).cuda()).double().cpu().numpy()
        ref = np.fft.irfft2(np.fft.rfft2(x) / P, s=(ny, nx))
        assert np.linalg.norm(got - ref) <= BOUND[mode] * np.linalg.norm(ref), (ny, nx)
        plan.close()


@pytest.mark.parametrize("mode,ny,nx,rows,ffts", [
    ("fp32", 64, 64, 64, 32), ("fp32", 256, 512, 32, 32), ("fp32", 64, 4096, 8, 64),
    ("fp64", 64, 64, 64, 32), ("fp64", 128, 1024, 16, 32), ("fp64", 64, 4096, 4, 64),
    ("mixed", 256, 256, 64, 16)])
def test_large_cta_shapes_are_cut_to_what_fits(mode, ny, nx, rows, ffts):
    """Shapes within the limits at 16 elements per thread stay accepted; the
    results are the default schedule's up to the rounding of the sums."""
    P, obs, x = grid(ny, nx)
    dt = torch.float32 if mode == "fp32" else torch.float64
    d = torch.from_numpy(x).to(dt).cuda()
    tol, bound = (1e-6, 1e-5) if mode == "fp32" else (1e-10, 1e-8)
    ref = cg.Plan(P, obs, mode=mode).ml(d, tol)[0]
    got = cg.Plan(P, obs, mode=mode, rows_per_cta=rows, ffts_per_cta=ffts).ml(d, tol)[0]
    assert (got - ref).norm() <= bound * ref.norm()


@pytest.mark.parametrize("mode,rows", [("fp32", 16), ("fp64", 8), ("mixed", 16)])
def test_cta_shapes_beyond_the_limit_stay_refused(mode, rows):
    P, obs, _ = grid(64, 4096)
    with pytest.raises(cg.FillError):
        cg.Plan(P, obs, mode=mode, rows_per_cta=rows)
