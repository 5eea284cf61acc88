"""GPU: the limits of the CG loops -- max_iter when every iteration asks for a
residual update, and how far a host-driven loop runs past convergence."""
import numpy as np
import pytest

from workloads import synth

torch = pytest.importorskip("torch")
pytestmark = pytest.mark.gpu

if not torch.cuda.is_available():  # pragma: no cover
    pytest.skip("needs a CUDA GPU", allow_module_level=True)

import paper_1109_0286_gb300 as cg  # noqa: E402

OK, ENOTCONV = 0, 3


def flat_case(ny, nx):
    """A spectrum within a factor 6 of flat: every CG iteration lowers the
    residual to less than half, so update_delta = 0.9 asks for an update each."""
    s = synth.spectrum_lorentz_beam(ny, nx, noise_frac=0.0)
    P = 0.2 + s / s.max()
    obs = synth.mask_band_discs(ny, nx, ny // 8, 4, 2.0, 5.0, 3)
    return P, obs, np.random.default_rng(3).standard_normal((ny, nx))


@pytest.mark.parametrize("max_iter", [1, 3, 4, 6])
@pytest.mark.parametrize("precond", [True, False])
@pytest.mark.parametrize("ny,nx", [(64, 64), (45, 70)])
def test_updates_every_iteration_stop_at_max_iter(ny, nx, precond, max_iter):
    P, obs, d = flat_case(ny, nx)
    dg = torch.from_numpy(d).cuda()
    full = cg.Plan(P, obs, precond=precond, update_delta=0.9)
    _, st = full.ml(dg, 1e-12)
    need = st[0]["iters"]
    assert st[0]["status"] == OK and need > 7 and st[0]["refine_steps"] >= need - 1
    for host in (False, True):
        plan = cg.Plan(P, obs, precond=precond, update_delta=0.9, max_iter=max_iter,
                       host_loops=host)
        _, st = plan.ml(dg, 1e-12, check=False)
        assert (st[0]["iters"], st[0]["status"]) == (max_iter, ENOTCONV), host
    plans = [cg.Plan(P, obs, precond=precond, update_delta=0.9, max_iter=max_iter)
             for _ in range(2)]
    _, st = cg.realize_batch(plans, [dg, dg], [1, 2], 1e-12, check=False)
    assert [(s["iters"], s["status"]) for s in st] == [(max_iter, ENOTCONV)] * 2
    # converged by the last iteration that is allowed
    plan = cg.Plan(P, obs, precond=precond, update_delta=0.9, max_iter=need)
    _, st = plan.ml(dg, 1e-12)
    assert (st[0]["iters"], st[0]["status"]) == (need, OK)


@pytest.mark.parametrize("precond", [True, False])
@pytest.mark.parametrize("iters", [1, 8, 33])
def test_host_loop_checks_every_8_iterations(precond, iters):
    """Kernels of a host-driven solve of `iters` iterations: those of the graph
    form, up to 8 iterations more, and one check per 8 iterations."""
    _, obs, d = flat_case(64, 64)
    P = synth.spectrum_cmb_like(64, 64, 2 * np.pi / 64)   # some 50 iterations to 1e-6
    dg = torch.from_numpy(d).float().cuda()
    n = []
    for host in (False, True):
        plan = cg.Plan(P, obs, mode="fp32", precond=precond, max_iter=iters, host_loops=host)
        _, st = plan.ml(dg, 0.0, check=False)
        assert (st[0]["iters"], st[0]["status"]) == (iters, ENOTCONV)
        n.append(st[0]["launches"])
    passes = 8 if precond else 4
    assert n[1] - n[0] <= 8 * passes + iters // 8 + 1
