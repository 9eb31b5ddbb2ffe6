"""FP64 GMRES at the edges of its pipelined steps: cycles that end on the
restart length, on the iteration cap and on convergence, one to five
right-hand sides, against the oracle's LU solution."""
import numpy as np
import pytest
import torch

import mtf_inputs as mi
from oracle.mtf import MTFSystem
from tests.oracle_helpers import skeleton_of

pytestmark = pytest.mark.gpu


@pytest.fixture(scope="module")
def api():
    if not torch.cuda.is_available():
        pytest.skip("needs a CUDA device")
    from paper_2502_10907_gb300.build import build
    build()
    from paper_2502_10907_gb300 import api as A
    return A


@pytest.fixture(scope="module")
def problem():
    cfg = mi.config_split_sphere(rings=2, k0=1.0)
    sk = skeleton_of(cfg["mesh"])
    ref = MTFSystem(sk, cfg["k0"], cfg["eps_r"], cfg["mu_r"])
    return cfg, ref


@pytest.mark.parametrize("nrhs, restart, precond", [(1, 25, 1), (2, 1000, 0), (5, 30, 1), (3, 1000, 1)])
def test_converged_solves_match_lu(api, problem, nrhs, restart, precond):
    """Relative residual 1e-11 times the condition of this small system (below 1e3): 1e-8."""
    cfg, ref = problem
    dirs, pols = mi.plane_wave_batch(3)
    dirs, pols = dirs[:nrhs], pols[:nrhs]
    s = api.System(api.Mesh.from_inputs(cfg["mesh"]), cfg["k0"], cfg["eps_r"], cfg["mu_r"], tol=1e-11, restart=restart,
                   max_iter=4000, precond=precond)
    x, st = s.solve(dirs, pols)
    xr = ref.solve_lu(ref.rhs(dirs, pols)).T
    assert st.converged == 1 and st.rel_residual <= 1e-11
    assert np.linalg.norm(x.cpu().numpy() - xr) < 1e-8 * np.linalg.norm(xr)
    # the same handle again: nothing of the step queued past convergence stays behind
    x2, st2 = s.solve(dirs, pols)
    assert st2.converged == 1
    assert np.linalg.norm(x2.cpu().numpy() - xr) < 1e-8 * np.linalg.norm(xr)


@pytest.mark.parametrize("restart, max_iter", [(1, 3), (4, 10), (50, 7)])
def test_iteration_cap(api, problem, restart, max_iter):
    cfg, _ = problem
    s = api.System(api.Mesh.from_inputs(cfg["mesh"]), cfg["k0"], cfg["eps_r"], cfg["mu_r"], tol=1e-12, restart=restart,
                   max_iter=max_iter)
    x, st = s.solve(cfg["dirs"], cfg["pols"], raise_on_noconv=False)
    assert st.converged == 0 and st.iterations == max_iter
    b = s.rhs(cfg["dirs"], cfg["pols"])
    r = torch.linalg.vector_norm(b - s.matvec(x), dim=1) / torch.linalg.vector_norm(b, dim=1)
    assert abs(float(r.max()) - st.rel_residual) < 1e-10 and float(r.max()) <= 1.0
