"""GPU: the CG vectors' storage (32 values per mask word with a masked pixel)
at the edges of words, rows and the map."""
import numpy as np
import pytest

from workloads import synth

torch = pytest.importorskip("torch")
pytestmark = pytest.mark.gpu

if not torch.cuda.is_available():  # pragma: no cover
    pytest.skip("needs a CUDA GPU", allow_module_level=True)

import paper_1109_0286_gb300 as cg  # noqa: E402

BOUND = {"fp64": 1e-10, "mixed": 1e-8, "fp32": 1e-4}   # of the converged fills


def dense_ml(P, obs, d):
    """-(Q_MM)^-1 Q_MU d_U with the columns of Q from numpy's FFT."""
    ny, nx = obs.shape
    apply = lambda v: np.fft.irfft2(np.fft.rfft2(v) / P, s=(ny, nx))   # noqa: E731
    m = np.flatnonzero(obs.ravel() == 0)
    Q = np.zeros((m.size, m.size))
    for j, i in enumerate(m):
        e = np.zeros(ny * nx)
        e[i] = 1.0
        Q[:, j] = apply(e.reshape(ny, nx)).ravel()[m]
    b = -apply(np.where(obs == 0, 0.0, d)).ravel()[m]
    x = d.copy().ravel()
    x[m] = np.linalg.solve(Q, b)
    return x.reshape(ny, nx)


@pytest.mark.parametrize("mode", ["fp64", "mixed", "fp32"])
@pytest.mark.parametrize("precond", [True, False])
@pytest.mark.parametrize("ny,nx", [(16, 32), (32, 256), (45, 70)])
def test_masks_at_word_edges(ny, nx, precond, mode):
    n = ny * nx
    P = synth.spectrum_lorentz_beam(ny, nx, sb=0.8, noise_frac=1e-2)
    d = np.random.default_rng(ny).standard_normal((ny, nx))
    dt = torch.float32 if mode == "fp32" else torch.float64
    tol = {"fp64": 1e-13, "mixed": 1e-11, "fp32": 1e-6}[mode]
    for masked in ([0], [n - 1], [31, 32], [30, 33, 63], [nx - 1, nx], list(range(32, 64)),
                   list(range(0, n, 65)), [1, n // 2, n - 2]):
        obs = np.ones(n, np.uint8)
        obs[masked] = 0
        obs = obs.reshape(ny, nx)
        plan = cg.Plan(P, obs, mode=mode, precond=precond)
        assert plan.masked_count == len(masked)
        for _ in range(2):   # the second call starts from used vectors
            x = plan.ml(torch.from_numpy(d).to(dt).cuda(), tol)[0][0].double().cpu().numpy()
        ref = dense_ml(P, obs, d.astype(np.float32).astype(np.float64) if mode == "fp32" else d)
        m = obs == 0
        assert np.linalg.norm(x[m] - ref[m]) <= BOUND[mode] * np.linalg.norm(ref[m]), masked
        plan.close()
