"""Mixed-precision blocks of structured meshes, where the rounding of a factor
is the same for every triangle and adds up, against the FP64 blocks."""
import numpy as np
import pytest
import torch

import mtf_inputs as mi

pytestmark = pytest.mark.gpu


@pytest.fixture(scope="module")
def api():
    if not torch.cuda.is_available():
        pytest.skip("needs a CUDA device")
    from paper_2502_10907_gb300.build import build
    build()
    from paper_2502_10907_gb300 import api as A
    return A


@pytest.mark.parametrize("n", [2, 4, 5])
def test_structured_blocks(api, n):
    """Entries are sums of a few FP32 contributions of either sign, stored in
    FP32 (2^-25 on average each): 2^-23 norm-wise for K, twice that for T,
    whose div-div parts cancel further.  Two RWG factors rounded alike in every
    row and column would add up to 2^-23 by themselves."""
    m = mi.cube_partition((2, 2, 2), n)
    eps = np.concatenate([[1.0], np.linspace(1.5, 3.9, m.n_domains - 1)])
    mesh = api.Mesh.from_inputs(m)
    exact = api.System(mesh, 3.0, eps, np.ones(m.n_domains))
    mixed = api.System(mesh, 3.0, eps, np.ones(m.n_domains), precision=1)
    rel = lambda a, b: float(torch.linalg.vector_norm(a - b) / torch.linalg.vector_norm(b))
    for i in range(m.n_domains):
        (T, K), (t, k) = exact.block(i), mixed.block(i)
        assert rel(k, K) < 2.0 ** -23 and rel(t, T) < 2.0 ** -22, (i, rel(k, K), rel(t, T))
