"""FP64 systems without the optional copy of their blocks: the matvec rotates
the blocks as it reads them, with the same results to the bit."""
import ctypes
import os
import subprocess

import numpy as np
import pytest
import torch

import mtf_inputs as mi

pytestmark = pytest.mark.gpu
ROOT = os.path.dirname(os.path.dirname(os.path.abspath(__file__)))


@pytest.fixture(scope="module")
def api():
    if not torch.cuda.is_available():
        pytest.skip("needs a CUDA device")
    from paper_2502_10907_gb300.build import build
    build()
    from paper_2502_10907_gb300 import api as A
    return A


@pytest.fixture(scope="module")
def drop(tmp_path_factory):
    so = str(tmp_path_factory.mktemp("drop") / "drop_rotated.so")
    cuda = os.path.dirname(os.path.dirname(os.path.realpath("/usr/local/cuda/bin/nvcc")))
    subprocess.run(["g++", "-O2", "-std=c++17", "-shared", "-fPIC", "-I", os.path.join(cuda, "include"),
                    "-I", os.path.join(ROOT, "paper_2502_10907_gb300", "csrc"),
                    os.path.join(ROOT, "tests", "host_src", "drop_rotated.cpp"), "-o", so], check=True)
    lib = ctypes.CDLL(so)
    lib.drop_rotated.argtypes = [ctypes.c_void_p]
    return lib.drop_rotated


@pytest.mark.parametrize("mesh, nrhs", [("ico0", 1), ("cubes", 2), ("uv", 3), ("uv", 4), ("ico2", 7)])
def test_matvec_without_copy(api, drop, mesh, nrhs):
    m = {"ico0": lambda: mi.icosphere(0), "ico2": lambda: mi.icosphere(2), "uv": lambda: mi.uv_sphere(5, 7),
         "cubes": lambda: mi.cube_partition((2, 1, 1), 1)}[mesh]()
    eps = np.concatenate([[1.0], np.linspace(1.5, 2.5, m.n_domains - 1)])
    mu = np.concatenate([[1.0], np.linspace(1.3, 0.7, m.n_domains - 1)])
    s = api.System(api.Mesh.from_inputs(m), 1.3, eps, mu)
    x = torch.randn((nrhs, s.mesh.n_total), dtype=torch.complex128, device="cuda")
    y = s.matvec(x)
    assert drop(s.handle) == 1
    assert torch.equal(s.matvec(x), y)
    s.reassemble(1.3, eps, mu)  # stays without: other sums of the same entries (the assembly's atomics)
    assert torch.linalg.vector_norm(s.matvec(x) - y) < 1e-13 * torch.linalg.vector_norm(y)
    assert drop(s.handle) == 0
