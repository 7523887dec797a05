"""Reactive 3-D grids whose rows are not a multiple of 4 cells: the general FD update over the whole grid
(constant and variable heat capacities) and the stream-collide with pairs that straddle rows, against the FP64
oracle. The mixture has every species everywhere and is too cold to burn out in a step, so that no cell sits
at the rate law's switch max(Y, 0), where a rounding is amplified (FP32 storage floors: 1e-7 to 6e-6 over 10
steps, several seeds). Bound per field: max(1e-5, 3 x the FP32 storage floor), FP16 storage 2e-3 in relative L2
of u; pressure and mass 1e-6."""
import numpy as np
import pytest

import workloads as W
from tests.parity import compare, gpu_run, oracle_run, rel_l2, storage_floor
from workloads.configs import variable_cp

pytestmark = pytest.mark.gpu
STEPS = 10


def _burner(n, storage="f32", sealed=False, vcp=False):
    wl = W.generate.swirl_3d(*n, reactive=True, storage=storage, seed=21, dt=2e-6, T_hot=1300.0)
    wl.Y = 0.8 * wl.Y + 0.2 * wl.Y.mean(axis=1, keepdims=True)
    if sealed:
        wl.cfg["bc"]["x"] = ("wall", "wall")
        r = np.arange(wl.N)
        wl.u[0] = 0.02 * np.sin(np.pi * (r % n[0] + 0.5) / n[0]) * np.sin(np.pi * (r // n[0] % n[1] + 0.5) / n[1])
        wl.u[:, wl.mask != 0] = 0.0
    if vcp:
        variable_cp(wl.cfg)
    return wl


def _check(wl):
    o, st = oracle_run(wl, STEPS)
    gpu = gpu_run(wl, STEPS)
    assert np.array_equal(gpu["stencil_words"].astype(np.int64), o.stencil_words_packed().numpy())
    assert abs(gpu["scalars"]["P_th"] - st["P_th"]) <= 1e-6 * st["P_th"]
    assert abs(gpu["scalars"]["M"] - st["M"]) <= 1e-6 * abs(st["M"])
    if wl.cfg["storage"] == "f16":
        assert compare(wl, gpu, st, metric=rel_l2)["u"] <= 2e-3
        return
    errs, floor = compare(wl, gpu, st), storage_floor(wl, STEPS, st)
    bad = {k: (v, floor[k]) for k, v in errs.items() if not v <= max(1e-5, 3.0 * floor[k])}
    assert not bad, f"errors above max(1e-5, 3 x floor): {bad}"


@pytest.mark.parametrize("vcp", [False, True])
@pytest.mark.parametrize("n", [(37, 21, 15), (38, 20, 13)])
def test_burner(n, vcp):
    _check(_burner(n, vcp=vcp))


def test_variable_cp_in_tiles_of_four():
    _check(_burner((36, 20, 13), vcp=True))


@pytest.mark.parametrize("n", [(37, 21, 15), (38, 20, 13)])
def test_burner_f16(n):
    _check(_burner(n, storage="f16"))


def test_solid_column_beside_an_odd_row():
    """A sealed grid of odd rows (elements loaded one by one) and the same with a solid column behind each
    row (pairs loaded as one): the same bits in every fluid cell."""
    n = (37, 21, 15)
    odd = _burner(n, sealed=True)
    even = _burner((38, 21, 15), sealed=True)
    pad = lambda a: np.concatenate([a.reshape(*a.shape[:-1], 15, 21, 37)] + [a.reshape(*a.shape[:-1], 15, 21, 37)[..., -1:]], -1)
    for k in ("T", "Y", "u", "P_h"):
        setattr(even, k, np.ascontiguousarray(pad(getattr(odd, k)).reshape(*getattr(odd, k).shape[:-1], -1)))
    mask = pad(odd.mask)
    mask[..., -1] = 1
    even.mask = np.ascontiguousarray(mask.reshape(-1))
    even.u[:, even.mask != 0] = 0.0
    a, b = gpu_run(odd, STEPS), gpu_run(even, STEPS)
    assert a["scalars"]["P_th"] == b["scalars"]["P_th"] and a["scalars"]["M"] == b["scalars"]["M"]
    fluid = np.asarray(odd.mask) == 0
    for k in ("T", "Y", "u", "P_h", "rho", "lam", "g"):
        x = a[k][..., fluid]
        y = b[k].reshape(*b[k].shape[:-1], 15, 21, 38)[..., :37].reshape(*b[k].shape[:-1], -1)[..., fluid]
        assert np.array_equal(x, y), k
