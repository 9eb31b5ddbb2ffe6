"""FP64 matvec at the edges of its tiling, against the oracle: passes of 4
right-hand sides, columns in tiles of 128, ragged rows per CTA."""
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


# blocks of 30, 12 to 36, 99 and 120 / 480 dofs; mu_r != 1 (rho != sqrt(eps))
@pytest.mark.parametrize("mesh, nrhs", [("ico0", 1), ("cubes", 2), ("uv", 3), ("uv", 4), ("ico1", 5), ("ico2", 1), ("ico2", 7)])
@pytest.mark.parametrize("opts", [{}, dict(precision=1, residual_df=0)])
def test_matvec_over_tiles(api, mesh, nrhs, opts):
    """Row sums of up to 960 FP64 products: 1e-13 of the stored blocks' product, norm-wise."""
    m = {"ico0": lambda: mi.icosphere(0), "ico1": lambda: mi.icosphere(1), "ico2": lambda: mi.icosphere(2),
         "uv": lambda: mi.uv_sphere(5, 7), "cubes": lambda: mi.cube_partition((2, 1, 1), 1)}[mesh]()
    eps = np.concatenate([[1.0], np.linspace(1.5, 2.5, m.n_domains - 1)])
    mu = np.concatenate([[1.0], np.linspace(1.3, 0.7, m.n_domains - 1)])
    sk = skeleton_of(m)
    ref = MTFSystem(sk, 1.3, eps, mu, assemble=False)
    s = api.System(api.Mesh.from_inputs(m), 1.3, eps, mu, **opts)
    for i in range(m.n_domains):
        T, K = (t.cpu().numpy() for t in s.block(i))
        ref.T.append(T)
        ref.K.append(K)
    rng = np.random.default_rng(nrhs)
    x = rng.standard_normal((nrhs, sk.n_total)) + 1j * rng.standard_normal((nrhs, sk.n_total))
    y = s.matvec(torch.from_numpy(x).cuda()).cpu().numpy()
    yr = ref.matvec(x.T).T
    assert np.linalg.norm(y - yr) < 1e-13 * np.linalg.norm(yr)


@pytest.mark.parametrize("mesh, nrhs", [("ico0", 1), ("cubes", 2), ("uv", 3), ("uv", 4), ("ico2", 7)])
@pytest.mark.parametrize("pairs", [0, 1])
def test_double_float_matvec_over_tiles(api, mesh, nrhs, pairs):
    """The same with FP32 entries (pairs 0) or FP32 pairs of the FP64 entries
    (pairs 1) and double-float sums: products and sums to about 2^-46, up to
    960 of them, 1e-12 of the blocks' product norm-wise."""
    m = {"ico0": lambda: mi.icosphere(0), "ico2": lambda: mi.icosphere(2), "uv": lambda: mi.uv_sphere(5, 7),
         "cubes": lambda: mi.cube_partition((2, 1, 1), 1)}[mesh]()
    eps = np.concatenate([[1.0], np.linspace(1.5, 2.5, m.n_domains - 1)])
    mu = np.concatenate([[1.0], np.linspace(1.3, 0.7, m.n_domains - 1)])
    sk = skeleton_of(m)
    ref = MTFSystem(sk, 1.3, eps, mu, assemble=False)
    mesh_ = api.Mesh.from_inputs(m)
    s = api.System(mesh_, 1.3, eps, mu, precision=1, residual_fp64=pairs)
    blocks = api.System(mesh_, 1.3, eps, mu) if pairs else s
    for i in range(m.n_domains):
        T, K = (t.cpu().numpy() for t in blocks.block(i))
        ref.T.append(T)
        ref.K.append(K)
    rng = np.random.default_rng(nrhs)
    x = rng.standard_normal((nrhs, sk.n_total)) + 1j * rng.standard_normal((nrhs, sk.n_total))
    y = s.matvec(torch.from_numpy(x).cuda()).cpu().numpy()
    yr = ref.matvec(x.T).T
    assert np.linalg.norm(y - yr) < 1e-12 * np.linalg.norm(yr)
