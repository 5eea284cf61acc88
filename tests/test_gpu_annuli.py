"""GPU: memory of the kernel Laplace solver's tables and spectra, and its
kernels taken in turns where their spectra do not fit at once."""
import numpy as np
import pytest

torch = pytest.importorskip("torch")
pytestmark = pytest.mark.gpu

if not torch.cuda.is_available():  # pragma: no cover
    pytest.skip("needs a CUDA GPU", allow_module_level=True)

import paper_1109_0286_gb300 as cg  # noqa: E402
from paper_1109_0286_gb300 import laplace  # noqa: E402

ELEM = {"fp32": 4, "fp64": 8, "mixed": 8}   # bytes of a value of the solver's precision


def make(n, mode, batch=1):
    obs = np.ones((n, n), np.uint8)
    obs[n // 3:n // 3 + n // 4] = 0
    return obs, cg.Plan(np.ones((n, n // 2 + 1)), obs, mode=mode, batch=batch)


def set_annuli(plan, nk):
    radii = laplace.ms_radii(nk)
    plan.set_annuli([r[0] for r in radii], [r[1] for r in radii])
    return radii


@pytest.mark.parametrize("mode", ["fp32", "fp64", "mixed"])
def test_only_the_present_set_is_held(mode):
    """However the number of annuli grew, a plan holds one table and one complex
    spectrum per annulus in the solver's precision (and the allocator's 2 MB
    granules)."""
    n, free = 1024, lambda: torch.cuda.mem_get_info()[0]   # noqa: E731
    _, plan = make(n, mode)
    torch.cuda.synchronize()
    before = free()
    for nk in (2, 5, 9, 4):
        set_annuli(plan, nk)
    assert before - free() <= 9 * 3 * n * (n // 2 + 1) * ELEM[mode] + 4 * 2 ** 21
    plan.close()


@pytest.mark.parametrize("mode", ["fp32", "mixed"])
def test_kernels_in_turns(mode):
    """A batch whose spectra exceed 1 GB for all annuli takes them in turns;
    every map as in a plan of its own, whose annuli run together."""
    n, nk = 2048, 9
    batch = 4 if mode == "mixed" else 8
    one = batch * 2 * n * (n // 2 + 1) * ELEM[mode]
    assert nk * one > 2 ** 30 >= nk * one // batch
    obs, many = make(n, mode, batch)
    _, single = make(n, mode)
    for p in (many, single):
        radii = set_annuli(p, nk)
    cls = laplace.ms_classes(torch.from_numpy(obs).cuda(), radii)
    assert len(torch.unique(cls[torch.from_numpy(obs).cuda() == 0])) == nk
    dt = torch.float32 if mode == "fp32" else torch.float64
    d = torch.from_numpy(np.random.default_rng(2).standard_normal((batch, n, n))).to(dt).cuda()
    x, _ = many.laplace_ms(d, 3, cls)
    for i in range(batch):
        assert torch.equal(x[i], single.laplace_ms(d[i], 3, cls)[0][0]), i
