"""The kernels' own FP32 operations (reciprocal, quotient and root by Newton steps, the closure built on
them) against CUDA's IEEE operators, bit for bit over all mantissas: tests/cuda/checks.cu, compiled here with
the library's flags."""
import ctypes as C
import importlib.util
import os
import subprocess

import pytest
import torch

pytestmark = pytest.mark.gpu
ROOT = os.path.dirname(os.path.dirname(os.path.abspath(__file__)))


def build_checks(path):
    """Compile tests/cuda/checks.cu into the folder ``path`` and load it."""
    spec = importlib.util.spec_from_file_location("_hlbm_build", os.path.join(ROOT, "paper_2207_11567_gb300", "build.py"))
    b = importlib.util.module_from_spec(spec)
    spec.loader.exec_module(b)
    so = os.path.join(str(path), "libchecks.so")
    subprocess.run([b.nvcc(), *b.FLAGS, "-I", b.CSRC, "-shared", os.path.join(ROOT, "tests", "cuda", "checks.cu"),
                    "-o", so], check=True)
    return C.CDLL(so)


@pytest.fixture(scope="module")
def checks(tmp_path_factory):
    lib = build_checks(tmp_path_factory.mktemp("checks"))
    for f in ("check_tau", "check_rcp", "check_sqrt", "check_div"):
        getattr(lib, f).restype = C.c_longlong
    lib.check_tau.argtypes = [C.c_float, C.c_float, C.c_int]
    return lib


@pytest.mark.parametrize("tau0, k, e", [(0.5, 0.736, -20), (0.5, 64.0, 10), (0.9, 0.25, -45)])
def test_relaxation_time(checks, tau0, k, e):
    assert checks.check_tau(tau0, k, e) == 0


@pytest.mark.parametrize("e", [-126, -67, -1, 63, 124])
def test_reciprocal(checks, e):
    """Exponents e and e + 1: 2^-126 .. 2^126."""
    assert checks.check_rcp(e) == 0


@pytest.mark.parametrize("e", [-67, -2, 1, 64, 126])
def test_square_root(checks, e):
    assert checks.check_sqrt(e) == 0


def test_quotient(checks):
    """2^24 random pairs; a numerator below 2^-100 may be off by one unit in the last place."""
    assert checks.check_div(-100, 106, 0) == 0
    assert checks.check_div(-105, -100, 1) == 0


def test_sensor_at_zero_temperature(checks):
    """No reaction at T = 0 or without a finite exponent: F_loc = 1 (F = 8 here, reached when hot)."""
    T = torch.tensor([0.0, 1e-30, 100.0, 2000.0], dtype=torch.float32, device="cuda")
    out = torch.full_like(T, -1.0)
    assert checks.sensor(C.c_void_p(T.data_ptr()), T.numel(), C.c_void_p(out.data_ptr())) == 0
    assert out.tolist()[:3] == [1.0, 1.0, 1.0]
    assert out[3].item() == 8.0
