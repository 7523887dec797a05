"""The stream-collide of the cells with interpolated wall links runs in the first blocks of the launch over
the other cells. A sealed burner, whose thermodynamic pressure changes every step: graphs over step pairs,
direct launches in one call, and single direct steps with a synchronisation after each give the same bits."""
import numpy as np
import pytest

import workloads as W

pytestmark = pytest.mark.gpu
STEPS = 12


def _run(wl, how):
    from paper_2207_11567_gb300 import from_workload
    s = from_workload(wl)
    s.use_graphs(how == "graphs")
    p = []
    if how == "single":
        for _ in range(STEPS):
            s.step(1)
            s.synchronize()
            p.append(s.scalars()["P_th"])
    else:
        s.step(STEPS)
    out = s.fields()
    out["P_th"] = np.array(s.scalars()["P_th"])
    s.close()
    return out, p


@pytest.mark.parametrize("storage", ["f32", "f16", "f64"])
@pytest.mark.parametrize("n", [(40, 20, 20), (37, 21, 18)])
def test_sealed_burner_same_bits(n, storage):
    wl = W.generate.swirl_3d(*n, reactive=True, curved=True, storage=storage, seed=4, dt=2e-6)
    wl.cfg["bc"]["x"] = ("wall", "wall")
    one, p = _run(wl, "single")
    assert len(set(p)) == STEPS  # the pressure moved in every step
    for how in ("graphs", "direct", "graphs"):
        got, _ = _run(wl, how)
        for k in one:
            assert np.array_equal(got[k], one[k]), (how, k)


@pytest.mark.parametrize("storage", ["f32", "f16"])
def test_isothermal_same_bits(storage):
    wl = W.generate.swirl_3d(40, 20, 20, curved=True, storage=storage, seed=4)
    one, _ = _run(wl, "single")
    for how in ("graphs", "direct"):
        got, _ = _run(wl, how)
        for k in one:
            assert np.array_equal(got[k], one[k]), (how, k)


def test_grid_without_planes_to_spare():
    """65,535 cells along z, the most that a grid of blocks has: a duct that is periodic in z gives each of
    its planes the bits of a shallow one."""
    def run(nz):
        wl = W.generate.duct_3d(nx=3, ny=4, nz=nz, q=0.35, storage="f64")
        out, _ = _run(wl, "graphs")
        return [out["g"].reshape(27, nz, 12), out["u"].reshape(3, nz, 12), out["P_h"].reshape(1, nz, 12)]
    for deep, flat in zip(run(65535), run(4)):
        assert np.isfinite(flat).all() and np.abs(flat).max() > 0
        assert (deep == flat[:, :1]).all()


def test_curved_walls_f16():
    """FP16 storage against the FP64 oracle: relative L2 of u, as in the other FP16 tests."""
    from oracle.step import Oracle
    from tests.parity import compare, gpu_run, rel_l2
    wl = W.generate.swirl_3d(40, 20, 20, curved=True, storage="f16", seed=4)
    c, d, q = wl.info["wall_links"]
    q = np.asarray(q, dtype=np.float32).astype(np.float64)
    wl.info["wall_links"] = (c, d, q)
    dense = np.zeros((27, wl.N))
    dense[d, c] = q
    o = Oracle(wl.cfg, wl.mask, wl.inlet_u, qwall=dense)
    st = o.run(o.round_state(o.init_state(T=wl.T, Y=wl.Y, u=wl.u, P_h=wl.P_h, g_pert=wl.g_pert)), 20)
    assert compare(wl, gpu_run(wl, 20), st, metric=rel_l2)["u"] <= 2e-3
