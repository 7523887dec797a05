"""The tiled FD update (3-D FP32) launches only tiles that hold fluid and skips rows of cells without a
fluid face: the reactive burner with whole tiles of 32 x 8 cells and single rows inside live tiles made
solid, at the high and the low side of the fluid, against the FP64 oracle. Bound per field as for the other
tiles at edges: max(1e-5, 3 x the FP32 storage floor); thermodynamic pressure 1e-12, mass 1e-6."""
import numpy as np
import pytest

import workloads as W
from tests.parity import compare, gpu_run, oracle_run, storage_floor

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("slab", ["y_high", "z_low"])
def test_solid_tiles_and_rows_f32(slab):
    wl = W.generate.swirl_3d(36, 20, 13, reactive=True, seed=21, dt=2e-6)
    mask = np.asarray(wl.mask).reshape(13, 20, 36)
    if slab == "y_high":
        mask[:, 15:, :32] = 1  # tiles from y = 16 on, and the row y = 15 of the tiles below them
    else:
        mask[:4, :, :32] = 1
        mask[4, 0:2, :32] = 1
    o, st = oracle_run(wl, 20)
    gpu = gpu_run(wl, 20)
    assert np.array_equal(gpu["stencil_words"].astype(np.int64), o.stencil_words_packed().numpy())
    errs, floor = compare(wl, gpu, st), storage_floor(wl, 20, st)
    bad = {k: (v, floor[k]) for k, v in errs.items() if not v <= max(1e-5, 3.0 * floor[k])}
    assert not bad, f"errors above max(1e-5, 3 x floor): {bad}"
    assert abs(gpu["scalars"]["P_th"] - st["P_th"]) <= 1e-12 * st["P_th"]
    assert abs(gpu["scalars"]["M"] - st["M"]) <= 1e-6 * abs(st["M"])
