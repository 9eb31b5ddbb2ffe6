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
