"""GPU: CG sums beyond the FP32 range in whole solves, and CTA heights that
differ in effect."""
import math

import numpy as np
import pytest

import oracle as O
from workloads import synth

torch = pytest.importorskip("torch")
pytestmark = pytest.mark.gpu

if not torch.cuda.is_available():  # pragma: no cover
    pytest.skip("needs a CUDA GPU", allow_module_level=True)

import paper_1109_0286_gb300 as cg  # noqa: E402

FLT_MAX = float(np.finfo(np.float32).max)


@pytest.mark.parametrize("precond", [True, False])
@pytest.mark.parametrize("mode", ["fp32", "mixed"])
# values that one thread adds; segments below and above a warp, and mixed radix
@pytest.mark.parametrize("ny,nx,values", [(64, 64, 8), (64, 1024, 32), (45, 70, 8), (24, 900, 24)])
def test_sums_beyond_the_fp32_range(ny, nx, values, mode, precond):
    """||b||^2 above the largest FP32 number while no thread's share comes near it
    (half the pixels masked, a spectrum within a factor 6 of flat, so that the
    other sums are within a factor 50 of it).  The ML fill is linear in the data
    and a power of two scales it without rounding, so only the sums' last bits
    may differ: fills to 1e-6 agree to 1e-5."""
    s = synth.spectrum_lorentz_beam(ny, nx, noise_frac=0.0)
    P = 0.2 + s / s.max()
    rng = np.random.default_rng(3)
    obs = (rng.random((ny, nx)) < 0.5).astype(np.uint8)
    d = rng.standard_normal((ny, nx))
    M = obs == 0
    b = O.apply_power(np.where(M, 0.0, d), O.hermitian_full(P, nx), -1.0)[M]
    total = float(np.sum(b * b))
    k = int(math.ceil(0.5 * math.log2(1.5 * FLT_MAX / total)))
    assert total * 4.0 ** k > 1.4 * FLT_MAX
    assert float(np.max(b * b)) * 4.0 ** k * values < FLT_MAX / 8
    dt = torch.float32 if mode == "fp32" else torch.float64
    d = torch.from_numpy(d).to(dt).cuda()
    plan = cg.Plan(P, obs, mode=mode, precond=precond)
    ref, _ = plan.ml(d, 1e-6)
    x, st = plan.ml(d * 2.0 ** k, 1e-6)
    assert st[0]["status"] == 0
    y = x.double() * 2.0 ** -k
    assert (y - ref.double()).norm() <= 1e-5 * ref.double().norm()


@pytest.mark.parametrize("ny,nx,threads", [(64, 256, 32), (32, 128, 16), (64, 512, 64)])
def test_fp64_heights_from_four_rows_up(ny, nx, threads):
    """FP64 heights of 4, 8 and more rows (threads per row times rows within the
    512 of a CTA, so none is cut): the same fills bit for bit."""
    P = synth.spectrum_cmb_like(ny, nx, 2 * math.pi / max(ny, nx))
    obs = synth.mask_band_discs(ny, nx, max(1, ny // 8), 4, 2.0, 5.0, 3)
    dg = torch.from_numpy(np.random.default_rng(3).standard_normal((ny, nx))).cuda()
    heights = [r for r in (4, 8, 16, 32) if r * threads <= 512]
    assert len(heights) >= 2
    xs = [cg.Plan(P, obs, mode="fp64", rows_per_cta=r).realize(dg, [9], 1e-8)[0] for r in heights]
    assert all(torch.equal(x, xs[0]) for x in xs[1:])
