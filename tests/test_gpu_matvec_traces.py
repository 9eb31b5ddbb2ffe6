"""Matvecs with one trace empty: T exceeds K by about 1 / (k h), so a norm over
both traces hides what a product loses of K.  The D and the N rows are each
compared with the stored blocks' products in FP64."""
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


MESHES = {"ico2": lambda: mi.icosphere(2), "cubes": lambda: mi.cube_partition((2, 1, 1), 3), "uv": lambda: mi.uv_sphere(5, 7)}


def materials(m, contrast):
    """eps_r, mu_r of one wavenumber with rho = 1, contrast, 1 / contrast, ..."""
    rho = np.array([1.0] + [contrast if i % 2 else 1.0 / contrast for i in range(1, m.n_domains)])
    index = np.array([1.0] + [1.6] * (m.n_domains - 1))
    return index * rho, index / rho


def dense_part(sk, blocks, rho, x):
    """2 A x: M x without the exchange."""
    y = np.zeros_like(x)
    for i, (T, K) in enumerate(blocks):
        d, n = sk.block_slices(i)
        y[:, d] = 2 * (x[:, d] @ K.T + x[:, n] @ T.T / rho[i])
        y[:, n] = 2 * (x[:, n] @ K.T - x[:, d] @ T.T * rho[i])
    return y


def errors(api, m, k0, contrast, nrhs, apply, dtype, **opts):
    """For one trace empty, then the other, and every block and slot: the
    error of the rows against FP64, their dense part and exchange part, and
    (|K| + |T|) (|u_D| + |w|) as the rows' products add it up, w = u_N / rho."""
    epsr, mur = materials(m, contrast)
    sk = skeleton_of(m)
    mesh = api.Mesh.from_inputs(m)
    s = api.System(mesh, k0, epsr, mur, **opts)
    blocks = [tuple(t.cpu().numpy() for t in s.block(i)) for i in range(m.n_domains)]
    ref = MTFSystem(sk, k0, epsr, mur, assemble=False)
    ref.T, ref.K = [b[0] for b in blocks], [b[1] for b in blocks]
    rho = np.sqrt(epsr / mur)
    rng = np.random.default_rng(nrhs)
    for empty in (0, 1):
        x = (rng.standard_normal((nrhs, sk.n_total)) + 1j * rng.standard_normal((nrhs, sk.n_total))).astype(dtype)
        for i in range(m.n_domains):
            x[:, sk.block_slices(i)[empty]] = 0
        y = apply(s)(torch.from_numpy(x).cuda()).cpu().numpy().astype(np.complex128)
        xd = x.astype(np.complex128)
        yr = ref.matvec(xd.T).T
        dense = dense_part(sk, blocks, rho, xd)
        for i, (T, K) in enumerate(blocks):
            d, n = sk.block_slices(i)
            sums = 2 * (np.abs(xd[:, d]) + np.abs(xd[:, n]) / rho[i]) @ (np.abs(K) + np.abs(T)).T
            for slot, sl in enumerate((d, n)):
                nrm = np.linalg.norm
                yield ((i, slot, empty), nrm(y[:, sl] - yr[:, sl]), nrm(dense[:, sl]), nrm(yr[:, sl] - dense[:, sl]),
                       nrm(sums) * (rho[i] if slot else 1.0))


# every width of the tensor-core kernel (32, 64, 128 columns) and the FMA stream (4)
@pytest.mark.parametrize("mesh, nrhs", [("ico2", 5), ("cubes", 8), ("uv", 9), ("ico2", 16), ("cubes", 32), ("uv", 4)])
@pytest.mark.parametrize("k0, contrast", [(0.05, 1.0), (0.3, 0.1), (0.3, 10.0), (1.3, 1.0)])
def test_matvec_f32_keeps_both_traces(api, mesh, nrhs, k0, contrast):
    """Operands of 22 significant bits (rounding, dropped lo x lo: 3 x 2^-22)
    and FP32 sums of up to 2 x 480 products: 8 x 2^-22 of the dense part,
    2^-22 of the exchange part's FP32 sums."""
    for where, err, dense, exchange, _ in errors(api, MESHES[mesh](), k0, contrast, nrhs, lambda s: s.matvec_f32,
                                                 np.complex64, precision=1):
        assert err < 2.0 ** -22 * (8 * dense + exchange), (where, err / dense)


@pytest.mark.parametrize("mesh, nrhs", [("ico2", 1), ("cubes", 2), ("uv", 5)])
@pytest.mark.parametrize("k0, contrast", [(0.05, 1.0), (0.3, 0.1), (0.3, 10.0), (1.3, 1.0)])
@pytest.mark.parametrize("opts, unit", [({}, 2.0 ** -53), (dict(precision=1), 2.0 ** -46),
                                        (dict(precision=1, residual_df=0), 2.0 ** -53)])
def test_matvec_within_the_stated_bound(api, mesh, nrhs, k0, contrast, opts, unit):
    """mtf_matvec's rows, each trace by itself, to the bound of mtf.h: its unit
    times (|K| + |T|) (|u_D| + |w|) summed over the row, with 16 for the
    roundings of up to 2 x 480 products per row in chains of at most 60."""
    for where, err, _, exchange, sums in errors(api, MESHES[mesh](), k0, contrast, nrhs, lambda s: s.matvec,
                                                np.complex128, **opts):
        assert err < unit * 16 * sums + 2.0 ** -51 * exchange, (where, err / sums)
