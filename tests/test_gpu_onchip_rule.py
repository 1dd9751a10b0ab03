"""AUTO's choice between the on-chip update (an instance per thread-block
cluster) and two launches per update for batches of small instances: on chip
where it measured faster by more than a tenth, two launches where they did.  A
GPC holds only one cluster of 11 to 16 blocks, so instances of 5121 to 8192 cells
leave SMs idle when they come in many waves of clusters."""
import numpy as np
import pytest

pytestmark = pytest.mark.gpu

# shape, instances, storage, updates, time on chip / time of two launches (GB300)
ONCHIP = [((16, 16, 16), 1, "fp32", 8, 0.4), ((4, 128, 4), 16, "fp32", 100, 0.3), ((128, 32, 1), 104, "fp32", 400, 0.6),
          ((8, 8, 8), 256, "fp16s", 8, 0.5), ((16, 16, 16), 104, "fp16s", 8, 0.84), ((16, 16, 16), 256, "fp32", 8, 0.78),
          ((17, 17, 16), 104, "bf16s", 200, 0.82), ((20, 20, 20), 7, "fp16s", 8, 0.46), ((18, 18, 18), 16, "fp32", 8, 0.73),
          ((4, 4, 504), 104, "fp32", 200, 0.57), ((4, 4, 2), 1024, "fp16s", 200, 0.25)]
TWO_LAUNCHES = [((18, 18, 16), 104, "fp16s", 200, 1.3), ((18, 18, 18), 256, "fp16s", 200, 1.21),
                ((19, 19, 19), 256, "bf16s", 200, 1.26), ((20, 20, 20), 256, "fp16s", 8, 1.32),
                ((18, 18, 16), 256, "fp32", 8, 1.30), ((19, 19, 19), 256, "fp32", 8, 1.27),
                ((15, 15, 15), 1024, "fp16s", 8, 1.29)]


@pytest.fixture(scope="module")
def lbm():
    from paper_1711_03254_gb300 import build
    build.build()
    from paper_1711_03254_gb300 import lbm as mod
    return mod


@pytest.mark.parametrize("case", ONCHIP + TWO_LAUNCHES, ids=str)
def test_auto_takes_the_faster_update(lbm, case):
    (nx, ny, nz), batch, precision, n, _ = case
    sim = lbm.Sim(nx, ny, nz, [dict(tau=(1.0, 1.0), G=-1.8)] * batch, precision=precision)
    sim.set_geometry(np.zeros((batch, nz, ny, nx), np.uint8))
    assert lbm.lbm_resolved_kernel(sim.ctx, n) == ("persistent" if case in ONCHIP else "compact")
    sim.close()


def test_library_says_whether_instances_stay_on_chip(lbm):
    """lbm_resolved_onchip follows the kernel that runs: storage, instance size, number of
    updates, wall slip, and the failure test of the grid-wide barriers."""
    def ctx(shape, precision="fp32", kernel="auto", **params):
        nx, ny, nz = shape
        sim = lbm.Sim(nx, ny, nz, [dict(tau=(1.0, 1.0), G=-1.8, **params)], precision=precision, kernel=kernel)
        assert not lbm.lbm_resolved_onchip(sim.ctx, 10)  # no geometry yet
        sim.set_geometry(np.zeros((1, nz, ny, nx), np.uint8))
        return sim
    sim = ctx((20, 20, 20))
    assert lbm.lbm_resolved_onchip(sim.ctx, 8) and not lbm.lbm_resolved_onchip(sim.ctx, 7)
    lbm.lbm_set_barrier_test(sim.ctx, 4_000_000_000, 1)
    assert not lbm.lbm_resolved_onchip(sim.ctx, 8)
    lbm.lbm_set_barrier_test(sim.ctx, 4_000_000_000, 0)
    sim.set_params([dict(tau=(1.0, 1.0), slip=0.5)])
    assert not lbm.lbm_resolved_onchip(sim.ctx, 8)
    sim.close()
    for shape, precision, kernel, want in (((32, 16, 16), "fp16s", "persistent", True),
                                           ((31, 17, 16), "bf16s", "persistent", False),  # 8432 cells
                                           ((16, 16, 16), "fp64", "persistent", False),
                                           ((16, 16, 16), "fp32", "compact", False)):
        sim = ctx(shape, precision, kernel)
        assert lbm.lbm_resolved_onchip(sim.ctx, 2) == want, (shape, precision, kernel)
        sim.close()
