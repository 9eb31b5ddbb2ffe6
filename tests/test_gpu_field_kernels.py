"""Far- and near-field kernels at the edges of their tiling, against the
oracle: right-hand-side passes of 32, groups of 8 points, chunks of 32
triangles."""
import numpy as np
import pytest
import torch

import mtf_inputs as mi
from oracle.mtf import MTFSystem
from oracle.nearfield import representation
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


@pytest.mark.parametrize("mesh, k0, nrhs, npts", [("ico0", 0.7, 1, 1), ("split2", 2.0, 3, 8), ("uv", 6.0, 5, 9),
                                                  ("cubes", 3.0, 17, 30), ("split2", 12.0, 33, 5), ("ico1", 1.0, 64, 17)])
def test_fields_over_tiles(api, mesh, k0, nrhs, npts):
    """Sums of a few thousand FP64 products per value: 1e-12 norm-wise."""
    m = {"ico0": lambda: mi.icosphere(0), "ico1": lambda: mi.icosphere(1), "split2": lambda: mi.split_sphere(2),
         "uv": lambda: mi.uv_sphere(5, 7), "cubes": lambda: mi.cube_partition((2, 2, 1), 2)}[mesh]()
    eps = np.concatenate([[1.0], np.linspace(1.5, 2.5, m.n_domains - 1)])
    mu = np.concatenate([[1.0], np.linspace(1.2, 0.8, m.n_domains - 1)])
    ref = MTFSystem(skeleton_of(m), k0, eps, mu, assemble=False)
    s = api.System(api.Mesh.from_inputs(m), k0, eps, mu)
    rng = np.random.default_rng(npts)
    x = rng.standard_normal((nrhs, s.mesh.n_total)) + 1j * rng.standard_normal((nrhs, s.mesh.n_total))
    xt = torch.from_numpy(x).cuda()
    d = rng.standard_normal((npts, 3))
    d /= np.linalg.norm(d, axis=1, keepdims=True)
    d[0] = [0.0, 0.0, 1.0]
    f = s.farfield(xt, d).cpu().numpy()
    fr = ref.farfield(x.T, d).transpose(2, 0, 1)
    assert np.linalg.norm(f - fr) < 1e-12 * np.linalg.norm(fr)
    # points of every subdomain in mixed order, one triangle diameter and more away
    pts = 3.0 * d
    dom = rng.integers(0, m.n_domains, npts)
    u = s.nearfield(xt, pts, dom).cpu().numpy()
    ur = representation(ref, x.T, pts, dom).transpose(2, 0, 1)
    assert np.linalg.norm(u - ur) < 1e-12 * np.linalg.norm(ur)
