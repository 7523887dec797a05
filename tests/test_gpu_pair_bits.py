"""The thermal D3Q27 stream-collide of two cells per thread carries out the operations of the one-cell kernel
in their order and roundings (reacting flows turn a changed rounding into differences of another size): the same
bits on the same state, for even rows (pairs loaded as one) and odd ones (pairs that straddle two rows, a last
cell without a partner), with walls, inlet, outlet, solids and sealed or periodic faces."""
import ctypes as C

import numpy as np
import pytest
import torch

import workloads as W
from tests.test_gpu_arith import build_checks

pytestmark = pytest.mark.gpu
CODE = {"periodic": 0, "wall": 1, "inlet": 2, "outlet": 3}


@pytest.fixture(scope="module")
def checks(tmp_path_factory):
    return build_checks(tmp_path_factory.mktemp("checks"))


def _ptr(t):
    return C.c_void_p(t.data_ptr())


@pytest.mark.parametrize("storage", ["f32", "f16"])
@pytest.mark.parametrize("faces", ["open", "sealed", "periodic"])
@pytest.mark.parametrize("n", [(38, 20, 14), (37, 21, 15), (37, 20, 15), (3, 9, 8), (131, 8, 9)])
def test_same_bits_as_one_cell_per_thread(checks, n, faces, storage):
    from paper_2207_11567_gb300 import from_workload
    if min(n) < 8:
        wl = W.generate.box(3, n, storage=storage, seed=1)
    else:
        wl = W.generate.swirl_3d(*n, storage=storage, seed=5)
        if faces == "sealed":
            wl.cfg["bc"]["x"] = ("wall", "wall")
    if faces == "periodic":
        wl.cfg["bc"] = {a: ("periodic", "periodic") for a in "xyz"}
    s = from_workload(wl)
    words = s.links()
    s.close()
    bc = (C.c_int * 6)(*[CODE[f] for a in "xyz" for f in wl.cfg["bc"][a]])
    dims = (C.c_int * 3)(*n)
    N = wl.N
    gen = torch.Generator("cuda").manual_seed(7)
    rnd = lambda *sh: torch.randn(*sh, generator=gen, device="cuda")
    g = (0.02 * rnd(27, N)).to(torch.float16 if storage == "f16" else torch.float32)
    rho = 0.2 + torch.rand(N, generator=gen, device="cuda")
    lam, T = 1e-3 * rnd(N), 300.0 + 1700.0 * torch.rand(N, generator=gen, device="cuda")
    u, inlet = 0.02 * rnd(3, N), 0.03 * rnd(3, n[1] * n[2])
    links = torch.from_numpy(words.view(np.int32)).cuda()
    fluid = links < 0  # bit 31
    for omega_b, smag_k, P_ref in ((1.0, 0.736, 0.0), (0.8, 0.736, 0.03), (1.0, 0.0, 0.03), (0.8, 0.0, 0.0)):
        got = []
        for two in (0, 1):
            out, uo, ph = torch.zeros_like(g), torch.zeros_like(u), torch.zeros(N, device="cuda")
            assert checks.stream_collide(two, int(storage == "f16"), dims, bc, _ptr(g), _ptr(links), _ptr(rho), _ptr(lam),
                                         _ptr(T), _ptr(inlet), _ptr(u), C.c_float(-2e-5), C.c_float(omega_b), C.c_float(smag_k), C.c_float(P_ref), _ptr(out),
                                         _ptr(uo), _ptr(ph)) == 0
            got.append((out, uo, ph))
        assert torch.isfinite(got[0][0][:, fluid]).all() and got[0][0][:, fluid].abs().max() > 0
        for a, b in zip(*got):
            assert torch.equal(a, b), (omega_b, smag_k, P_ref, int((a != b).sum()))
