"""Near field close to the skeleton, on both sides of it, and inside small
subdomains, against the oracle's sums over the same rule."""
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


# triangles 0.3 to 1.2 across: phases of every series length and beyond it; distances of 0.05 to 1 diameters
@pytest.mark.parametrize("mesh, k0", [("ico1", 0.3), ("ico1", 6.0), ("split2", 2.0), ("cubes", 1.5), ("cubes", 20.0),
                                      ("uv", 9.0)])
@pytest.mark.parametrize("distance", [0.05, 0.3, 1.0])
def test_close_points(api, mesh, k0, distance):
    """A point at distance r of a rule's point: coordinates rounded at 2^-53
    of the mesh's size give 2^-53 / r in r and three times that in 1 / r^3, and
    the moments about a vertex cancel to r of a triangle's size: about 1e-13 of
    the largest contribution at the closest points here, 1e-12 norm-wise."""
    m = {"ico1": lambda: mi.icosphere(1), "split2": lambda: mi.split_sphere(2), "uv": lambda: mi.uv_sphere(5, 7),
         "cubes": lambda: mi.cube_partition((2, 2, 2), 2)}[mesh]()
    eps = np.concatenate([[1.0], np.linspace(1.5, 2.5, m.n_domains - 1)])
    mu = np.concatenate([[1.0], np.linspace(1.2, 0.8, m.n_domains - 1)])
    ref = MTFSystem(skeleton_of(m), k0, eps, mu, assemble=False)
    s = api.System(api.Mesh.from_inputs(m), k0, eps, mu)
    rng = np.random.default_rng(7)
    x = rng.standard_normal((3, s.mesh.n_total)) + 1j * rng.standard_normal((3, s.mesh.n_total))
    t = rng.permutation(len(m.triangles))[:24]
    v = np.asarray(m.vertices)[np.asarray(m.triangles)[t]]
    n = np.cross(v[:, 1] - v[:, 0], v[:, 2] - v[:, 0])
    n /= np.linalg.norm(n, axis=1, keepdims=True)
    diam = np.linalg.norm(v - np.roll(v, 1, axis=1), axis=2).max(axis=1)
    w = rng.dirichlet([1.0, 1.0, 1.0], len(t))
    base = np.einsum("tv,tvc->tc", w, v)
    lab = np.asarray(m.labels)[t]
    pts = np.concatenate([base - distance * diam[:, None] * n, base + distance * diam[:, None] * n])
    dom = np.concatenate([lab[:, 0], lab[:, 1]]).astype(np.int32)
    u = s.nearfield(torch.from_numpy(x).cuda(), pts, dom).cpu().numpy()
    ur = representation(ref, x.T, pts, dom).transpose(2, 0, 1)
    assert np.linalg.norm(u - ur) < 1e-12 * np.linalg.norm(ur)
    # and point by point, on the scale of the field there
    err = np.linalg.norm(u - ur, axis=2).max(axis=0)
    assert (err < 1e-11 * np.linalg.norm(ur, axis=2).max(axis=0)).all(), err.max()


@pytest.mark.parametrize("npts, nrhs", [(1, 2), (1, 33), (3, 40), (37, 1), (40, 19), (120, 2), (300, 1), (700, 2), (700, 70)])
def test_points_per_work_item(api, npts, nrhs):
    """4 or 8 points per work item and passes of 4 to 32 right-hand sides, by the
    size of the call: sums of a few
    thousand FP64 products per value, 1e-12 norm-wise."""
    m = mi.split_sphere(2)
    eps = np.array([1.0, 2.0, 3.0])
    ref = MTFSystem(skeleton_of(m), 1.5, eps, np.ones(3), assemble=False)
    s = api.System(api.Mesh.from_inputs(m), 1.5, eps, np.ones(3))
    rng = np.random.default_rng(npts)
    x = rng.standard_normal((nrhs, s.mesh.n_total)) + 1j * rng.standard_normal((nrhs, s.mesh.n_total))
    xt = torch.from_numpy(x).cuda()
    d = rng.standard_normal((npts, 3))
    d /= np.linalg.norm(d, axis=1, keepdims=True)
    f = s.farfield(xt, d).cpu().numpy()
    fr = ref.farfield(x.T, d).transpose(2, 0, 1)
    assert np.linalg.norm(f - fr) < 1e-12 * np.linalg.norm(fr)
    dom = rng.integers(0, 3, npts).astype(np.int32)
    u = s.nearfield(xt, 2.0 * d, dom).cpu().numpy()
    ur = representation(ref, x.T, 2.0 * d, dom).transpose(2, 0, 1)
    assert np.linalg.norm(u - ur) < 1e-12 * np.linalg.norm(ur)
