"""GPU: the grid reductions of the CG scalars (inner products and norms)."""
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


def case(ny, nx, seed=3):
    P = synth.spectrum_cmb_like(ny, nx, 2 * math.pi / max(ny, nx))
    obs = synth.mask_band_discs(ny, nx, max(1, ny // 8), 4, 2.0, 5.0, seed)
    d = np.random.default_rng(seed).standard_normal((ny, nx))
    return P, obs, d


@pytest.mark.parametrize("ny,nx", [(64, 64), (32, 1024), (256, 128), (16, 4096)])
@pytest.mark.parametrize("mode", ["fp32", "fp64", "mixed"])
def test_sums_do_not_depend_on_the_cta_height(ny, nx, mode):
    """Partial sums cover four rows whatever the CTA height, so the solves are
    the same bit for bit (segments below, at and above one warp)."""
    P, obs, d = case(ny, nx)
    dt = torch.float32 if mode == "fp32" else torch.float64
    dg = torch.from_numpy(d).to(dt).cuda()
    ref = None
    for rows in (4, 8, 16):
        if rows * (nx // 32) > (512 if mode == "fp64" else 1024):
            continue
        plan = cg.Plan(P, obs, mode=mode, rows_per_cta=rows)
        x, st = plan.realize(dg, [9], 1e-6)
        ref = x.clone() if ref is None else ref
        assert torch.equal(x, ref), (rows, st)
        plan.close()


@pytest.mark.parametrize("ny,nx", [(64, 64), (64, 1024), (45, 70)])
def test_sums_beyond_the_fp32_range(ny, nx):
    """||b||^2 near and above the largest FP32 number: the partials of a warp
    or a CTA leave the FP32 range although no product does.  The ML fill is
    linear in the data and a power of two scales it without rounding, so only
    the rounding of the sums (2^-44) may differ."""
    P, obs, d = case(ny, nx)
    M = obs == 0
    b = O.apply_power(np.where(M, 0.0, d), O.hermitian_full(P, nx), -1.0)[M]
    total = float(np.sum(b * b))
    plan = cg.Plan(P, obs, mode="fp32")
    ref, _ = plan.ml(torch.from_numpy(d).float().cuda(), 1e-5)
    for target in (1e35, 1e38, 2e39):
        k = int(math.floor(0.5 * math.log2(target / total)))
        if float(np.max(b * b)) * 4.0 ** k * 64 > 1e38:
            continue   # a thread's own products would overflow
        x, st = plan.ml(torch.from_numpy(d * 2.0 ** k).float().cuda(), 1e-5)
        y = x.double() * 2.0 ** -k
        assert st[0]["status"] == 0
        assert (y - ref.double()).norm() <= 1e-5 * ref.double().norm()
