"""The grid-barrier form of the persistent update (k_persist_c) in the FP32 and
16-bit storages.  Instances of up to 8192 non-solid cells run on chip there, so
the shapes here hold more: one wave of threads that keep their cells (8193 to
65,536 cells, what AUTO gives it), and more than the resident threads (blocks
that stride over the items).  The states equal two launches per update bit for
bit in every storage, for both equilibria, the third-order regularisation and
every wall model, with INLET and OUTLET planes and batches, stepped and in the
steady loop; and after a barrier gave up, this kernel updates the context again."""
import numpy as np
import pytest

from paper_1711_03254_gb300 import workloads as W
from .test_gpu_persistent import _geometry, _run, _same, lbm  # noqa: F401

pytestmark = pytest.mark.gpu

KEPT, STRIDED = (28, 24, 20), (64, 40, 40)  # about 12,000 and 92,000 non-solid cells
CFGS = [dict(), dict(eq_order=1, wall_model=0), dict(reg_order=3, wall_model=3), dict(eq_order=1, wall_model=1),
        dict(eq_order=1, reg_order=3)]


def _params(B):
    return [dict(tau=(0.7 + 0.1 * k, 1.4), G=-1.4, rho_s=0.2 - 0.1 * k, g=(1e-4, 0, 2e-5), rho_in=(0.2, 0.8),
                 u_in=(0.02, 0, 0)) for k in range(B)]


@pytest.mark.parametrize("precision", ["fp32", "fp16s", "bf16s"])
@pytest.mark.parametrize("shape,B", [(KEPT, 1), (KEPT, 3), (STRIDED, 1)])
@pytest.mark.parametrize("cfg", CFGS, ids=str)
@pytest.mark.parametrize("inlet_outlet", [False, True])
def test_grid_barrier_update_equals_two_launches(lbm, precision, shape, B, cfg, inlet_outlet):  # noqa: F811
    geo = [_geometry(shape, 0.1, 11 + k, inlet_outlet) for k in range(B)]
    assert min(int((g[0] != 1).sum()) for g in geo) > 8192
    a = _run(lbm, "compact", shape, _params(B), geo, [3, 2], precision, **cfg)
    b = _run(lbm, "persistent", shape, _params(B), geo, [3, 2], precision, **cfg)
    assert _same(a, b)


@pytest.mark.parametrize("precision", ["fp32", "fp16s", "bf16s"])
def test_steady_loop_equals_two_launches(lbm, precision):  # noqa: F811
    t, r1, r2, u = W.droplet(24, 24, 24, 6.0)
    out = []
    for kernel in ("compact", "persistent"):
        sim = lbm.Sim(24, 24, 24, [dict(tau=(1.0, 0.8), G=-2.0), dict(tau=(0.9, 1.1), G=-1.9)], precision=precision,
                      kernel=kernel)
        sim.set_geometry(np.repeat(t[None], 2, 0))
        assert not lbm.lbm_resolved_onchip(sim.ctx, 7)
        sim.set_fields(*(np.repeat(f[None], 2, 0) for f in (r1, r2, u)))
        done, res = lbm.lbm_run_to_steady(sim.ctx, 7, 1e-12, 35, 2)
        out.append((done, res.copy(), sim.get_fields(), sim.get_f()))
        sim.close()
    (da, ra, fa, ga), (db, rb, fb, gb) = out
    assert da == db and np.array_equal(ra, rb) and _same((fa, ga), (fb, gb))


@pytest.mark.parametrize("precision", ["fp32", "fp16s"])
def test_update_after_a_barrier_gave_up(lbm, precision):  # noqa: F811
    geo = [_geometry(KEPT, 0.1, 9)]
    nx, ny, nz = KEPT
    sim = lbm.Sim(nx, ny, nz, _params(1), precision=precision, kernel="persistent")
    sim.set_geometry(geo[0][0][None])
    assert not lbm.lbm_resolved_onchip(sim.ctx, 3)
    fields = [geo[0][k][None] for k in (1, 2, 3)]
    sim.set_fields(*fields)
    lbm.lbm_set_barrier_test(sim.ctx, 20_000_000, 1)
    sim.step(3)
    with pytest.raises(lbm.LbmError) as e:
        sim.get_fields()
    assert e.value.status == 5 and "barrier" in str(e.value)
    lbm.lbm_set_barrier_test(sim.ctx, 4_000_000_000, 0)
    sim.set_fields(*fields)
    sim.step(5)
    a = sim.get_fields(), sim.get_f()
    sim.close()
    assert _same(a, _run(lbm, "compact", KEPT, _params(1), geo, [5], precision))
