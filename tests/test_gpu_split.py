"""The one-warp-per-field FD update of small 2-D FP64 grids against the FP64 oracle: cell counts that are
not multiples of a warp, a single row, obstacles with inlet and outlet, the flame sensor, and a sealed
domain whose thermodynamic pressure comes from the update's partial sums. Bound: relative L-infinity
1e-10 per field, as for the other FP64 parity tests."""
import pytest

import workloads as W
from tests.parity import compare, gpu_run, oracle_run

pytestmark = pytest.mark.gpu
STEPS = 20


def _check(wl):
    _, st = oracle_run(wl, STEPS)
    gpu = gpu_run(wl, STEPS)
    bad = {k: v for k, v in compare(wl, gpu, st).items() if not v <= 1e-10}
    assert not bad, f"errors above 1e-10: {bad}"
    if wl.cfg["closed_domain"]:
        assert abs(gpu["scalars"]["P_th"] - st["P_th"]) <= 1e-10 * st["P_th"]
        assert abs(gpu["scalars"]["M"] - st["M"]) <= 1e-10 * abs(st["M"])


@pytest.mark.parametrize("n", [(64, 1), (33, 3), (63, 8)])
def test_planar_flame(n):
    _check(W.generate.flame_2d(nx=n[0], ny=n[1], seed=5))


@pytest.mark.parametrize("sensor", [False, True])
@pytest.mark.parametrize("ends", ["inlet", "sealed"])
def test_chamber(ends, sensor):
    wl = W.generate.chamber_2d(nx=47, ny=29, dt=5e-7, storage="f64", seed=3, inlet=ends == "inlet")
    if ends == "sealed":
        wl.cfg["bc"]["x"] = ("wall", "wall")
    wl.cfg["closed_domain"] = True
    wl.cfg["flame_sensor"] = sensor
    _check(wl)
