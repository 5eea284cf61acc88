"""GPU: draws and operator applications read and write the caller's maps in
place; the kernel Laplace solver runs its annuli together."""
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
from paper_1109_0286_gb300 import laplace  # noqa: E402

DT = {"fp64": torch.float64, "mixed": torch.float64, "fp32": torch.float32}


@pytest.mark.parametrize("ny,nx", [(64, 128), (45, 70)])
@pytest.mark.parametrize("mode", ["fp64", "fp32"])
def test_maps_off_pair_alignment(ny, nx, mode):
    """Maps at an odd element offset take the copying path; same results."""
    P = synth.spectrum_cmb_like(ny, nx, 2 * math.pi / max(ny, nx))
    obs = synth.mask_band_discs(ny, nx, ny // 8, 3, 1.5, 4.0, 1)
    plan = cg.Plan(P, obs, mode=mode, batch=2)
    x = torch.from_numpy(np.random.default_rng(0).standard_normal((ny, nx))).to(DT[mode]).cuda()
    buf = torch.empty(2 * ny * nx + 1, dtype=DT[mode], device="cuda")
    off = buf[1:1 + ny * nx].view(ny, nx)
    off.copy_(x)
    for which in range(4):
        assert torch.equal(plan.apply(which, x), plan.apply(which, off))
    out = buf[1:].view(2, ny, nx)
    assert torch.equal(plan.draw([3, 4]), plan.draw([3, 4], out=out))


@pytest.mark.parametrize("ny,nx", [(128, 256), (90, 140)])
@pytest.mark.parametrize("mode,bound", [("fp64", 1e-11), ("mixed", 1e-10), ("fp32", 2e-5)])
def test_laplace_annuli_grow(ny, nx, mode, bound):
    """One annulus, then more on the same plan, two maps at once: against the
    oracle's sweeps (bounds of the solver's parity tests)."""
    obs = np.ones((ny, nx), np.uint8)
    obs[ny // 3:ny // 3 + ny // 4] = 0
    obs[5:9, 20:30] = 0
    d = np.random.default_rng(2).standard_normal((2, ny, nx))
    plan = cg.Plan(np.ones((ny, nx // 2 + 1)), obs, mode=mode, batch=2)
    dg = torch.from_numpy(d).to(DT[mode]).cuda()
    for nk in (1, 4):
        radii = laplace.ms_radii(nk)
        plan.set_annuli([r[0] for r in radii], [r[1] for r in radii])
        cls = laplace.ms_classes(torch.from_numpy(obs).cuda(), radii)
        x, _ = plan.laplace_ms(dg, 6, cls)
        for i in range(2):
            ref = O.laplace_ms(obs, d[i], radii, 6)
            got = x[i].double().cpu().numpy()
            assert np.linalg.norm(got - ref) <= bound * np.linalg.norm(ref), (nk, i)
