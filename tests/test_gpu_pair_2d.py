"""The two-cells-per-thread stream-collide of large 2-D FP32 grids (100,000 cells and more; smaller ones run one
cell per thread) against the FP64 oracle: rows of even and of odd length, the latter with an odd cell count,
a periodic box, and a reacting chamber with walls, inlet, outlet and obstacles. Bounds as in test_gpu_pair.py."""
import pytest

import workloads as W
from tests.parity import compare, gpu_run, oracle_run, rel_l2, storage_floor

pytestmark = pytest.mark.gpu
STEPS = 6


def _check(wl):
    assert wl.N >= 100000
    _, st = oracle_run(wl, STEPS)
    gpu = gpu_run(wl, STEPS)
    if wl.cfg["storage"] == "f16":
        assert compare(wl, gpu, st, metric=rel_l2)["u"] <= 2e-3
        return
    errs, floor = compare(wl, gpu, st), storage_floor(wl, STEPS, st)
    bad = {k: (v, floor[k]) for k, v in errs.items() if not v <= max(1e-5, 3.0 * floor[k])}
    assert not bad, f"errors above max(1e-5, 3 x floor): {bad}"


@pytest.mark.parametrize("storage", ["f32", "f16"])
@pytest.mark.parametrize("n", [(400, 256), (401, 251)])
def test_periodic_box(n, storage):
    wl = W.generate.box(2, n, storage=storage, tau=0.7, seed=3, pert=2e-3, U=0.03)
    wl.cfg["smag_cs"] = 0.1
    _check(wl)


@pytest.mark.parametrize("storage", ["f32", "f16"])
@pytest.mark.parametrize("n", [(400, 256), (401, 251)])
def test_chamber(n, storage):
    _check(W.generate.chamber_2d(*n, dt=5e-7, seed=5, inlet=True, storage=storage, u_init=0.01))
