"""The two-cells-per-thread stream-collide (FP32 arithmetic, default rates) at its edges, against the
FP64 oracle: rows of one pair or less, odd row lengths and odd cell counts (no 64-bit access, the last
cell without a partner, pairs that straddle two rows), periodic wrap within a pair, and walls, inlet
and outlet met by either cell of a pair. FP32 per field within max(1e-5, 3 x the FP32 storage floor),
FP16 storage within a relative L2 of 2e-3 on the velocity, as in the other parity tests."""
import pytest

import workloads as W
from tests.parity import compare, gpu_run, oracle_run, rel_l2, storage_floor

pytestmark = pytest.mark.gpu
STEPS = 20


def _check(wl):
    _, st = oracle_run(wl, STEPS)
    gpu = gpu_run(wl, STEPS)
    if wl.cfg["storage"] == "f16":
        assert compare(wl, gpu, st, metric=rel_l2)["u"] <= 2e-3
        return
    errs, floor = compare(wl, gpu, st), storage_floor(wl, STEPS, st)
    bad = {k: (v, floor[k]) for k, v in errs.items() if not v <= max(1e-5, 3.0 * floor[k])}
    assert not bad, f"errors above max(1e-5, 3 x floor): {bad}"


@pytest.mark.parametrize("storage", ["f32", "f16"])
@pytest.mark.parametrize("n", [(2, 3), (3, 3), (5, 4), (130, 3), (3, 3, 3), (2, 4, 5), (6, 5, 4), (66, 3, 3)])
def test_periodic_box(n, storage):
    wl = W.generate.box(len(n), n, storage=storage, tau=0.7, seed=3, pert=2e-3, U=0.03)
    wl.cfg["smag_cs"] = 0.1
    _check(wl)


@pytest.mark.parametrize("storage", ["f32", "f16"])
@pytest.mark.parametrize("n", [(28, 18, 16), (27, 17, 15), (27, 18, 16)])
def test_walls_inlet_outlet_isothermal(n, storage):
    _check(W.generate.swirl_3d(*n, storage=storage, seed=9))


@pytest.mark.parametrize("n", [(50, 22), (49, 21)])
def test_chamber_2d(n):
    _check(W.generate.chamber_2d(*n, dt=5e-7, seed=5, inlet=True))
