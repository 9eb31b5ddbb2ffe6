"""Assembly kernels at the edges of their dispatch rules, against the oracle's
blocks (FP64 systems)."""
import numpy as np
import pytest
import torch

import mtf_inputs as mi
from oracle.operators import assemble_block
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


def rel(a, b):
    return np.linalg.norm(a - b) / np.linalg.norm(b)


# k h of the adjacent pairs (triangle pairs up to 1.2 across) runs through every length of the radial power series and
# into the point-by-point sums beyond it; n_ss through odd, even, smallest and largest rules
@pytest.mark.parametrize("k0, n_ss", [(0.1, 1), (0.2, 4), (0.4, 3), (0.7, 5), (1.1, 4), (1.6, 2), (3.0, 4), (9.0, 6),
                                      (1.0, 12)])
def test_singular_pairs_over_kappa_and_rule_size(api, k0, n_ss):
    """Sums of at most 12^4 products per pair in FP64: within 1e-12 of the oracle norm-wise (2^-53 times a few hundred
    for the sums and the cancellation of the 3 x 3 combinations)."""
    m = mi.split_sphere(2) if n_ss < 12 else mi.icosphere(0)
    eps = np.concatenate([[1.0], np.linspace(1.5, 2.5, m.n_domains - 1)])
    sk = skeleton_of(m)
    s = api.System(api.Mesh.from_inputs(m), k0, eps, np.ones(m.n_domains), n_ss=n_ss)
    for i in range(m.n_domains):
        T, K = (t.cpu().numpy() for t in s.block(i))
        Tr, Kr = assemble_block(sk, i, k0 * np.sqrt(eps[i]), n_ss=n_ss)
        assert rel(T, Tr) < 1e-12 and rel(K, Kr) < 1e-12, (i, rel(T, Tr), rel(K, Kr))


# tiles of 16 triangles: blocks of 8, 20, 24, 32 and 80 triangles (fewer than a tile, ragged, whole tiles) and every
# length of the phase series, up to pairs that fall back to sincos (k times the radii above 2)
@pytest.mark.parametrize("mesh, k0", [("cube1", 0.3), ("ico0", 0.5), ("ico0", 4.0), ("split2", 0.9), ("ico1", 2.0),
                                      ("ico1", 6.0), ("uv", 1.3)])
@pytest.mark.parametrize("precision", [0, 1])
def test_regular_pairs_over_tiles_and_phases(api, mesh, k0, precision):
    """FP64: 1e-12 as above.  Mixed: FP32 products of about 60 rounded operations per evaluation, summed over the
    pairs of an entry: 64 x 2^-24 = 4e-6 norm-wise."""
    m = {"cube1": lambda: mi.cube_partition((1, 1, 2), 1), "ico0": lambda: mi.icosphere(0), "ico1": lambda: mi.icosphere(1),
         "split2": lambda: mi.split_sphere(2), "uv": lambda: mi.uv_sphere(5, 7)}[mesh]()
    eps = np.concatenate([[1.0], np.linspace(1.5, 2.5, m.n_domains - 1)])
    sk = skeleton_of(m)
    s = api.System(api.Mesh.from_inputs(m), k0, eps, np.ones(m.n_domains), precision=precision)
    tol = 4e-6 if precision else 1e-12
    for i in range(m.n_domains):
        T, K = (t.cpu().numpy() for t in s.block(i))
        Tr, Kr = assemble_block(sk, i, k0 * np.sqrt(eps[i]))
        assert rel(T, Tr) < tol and rel(K, Kr) < tol, (i, rel(T, Tr), rel(K, Kr))
        assert np.array_equal(T, T.T) and np.array_equal(K, K.T)
