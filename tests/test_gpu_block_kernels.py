"""Block FGMRES at the widths where its per-step kernels change: register
tiers of 4, 8, 12 and 16 columns, runs of 4 basis vectors or single ones in
the tiled copies, wide blocks, FMA projections, deflated directions."""
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
    cfg = mi.config_cube2(n=2, k0=3.0, n_dirs=9)
    return cfg, MTFSystem(skeleton_of(cfg["mesh"]), cfg["k0"], cfg["eps_r"], cfg["mu_r"])


@pytest.mark.parametrize("nrhs, opts", [(4, {}), (5, {}), (7, {}), (8, {}), (11, {}), (12, {}), (13, {}), (16, {}), (17, {}),
                                        (6, dict(mv_tensor=0)), (16, dict(mv_tensor=0)), (16, dict(gs_dots_half=0))])
def test_block_solves_match_lu(api, problem, nrhs, opts):
    """Mixed path at tol 1e-8 against LU: the stated 1e-5."""
    cfg, ref = problem
    dirs, pols = cfg["dirs"][:nrhs], cfg["pols"][:nrhs]
    s = api.System(api.Mesh.from_inputs(cfg["mesh"]), cfg["k0"], cfg["eps_r"], cfg["mu_r"], precision=1, precond=1,
                   osrc_np=16, tol=1e-8, restart=300, max_iter=2000, **opts)
    x, st = s.solve(dirs, pols)
    xr = ref.solve_lu(ref.rhs(dirs, pols)).T
    err = np.linalg.norm(x.cpu().numpy() - xr, axis=1) / np.linalg.norm(xr, axis=1)
    assert st.converged == 1 and err.max() < 1e-5


def test_dependent_right_hand_sides(api, problem):
    """Repeated and scaled columns are deflated from the block; every column still meets its tolerance."""
    cfg, ref = problem
    s = api.System(api.Mesh.from_inputs(cfg["mesh"]), cfg["k0"], cfg["eps_r"], cfg["mu_r"], precision=1, precond=1,
                   osrc_np=16, tol=1e-8, restart=300, max_iter=2000)
    b = s.rhs(cfg["dirs"][:6], cfg["pols"][:6])
    b = torch.cat([b, b[:2], 0.5 * b[2:3] + b[3:4]])  # 9 columns of rank 6
    x, st = s.solve_rhs(b)
    xr = ref.solve_lu(b.cpu().numpy().T).T
    err = np.linalg.norm(x.cpu().numpy() - xr, axis=1) / np.linalg.norm(xr, axis=1)
    assert st.converged == 1 and err.max() < 1e-5
