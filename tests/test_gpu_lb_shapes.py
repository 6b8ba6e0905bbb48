"""The stream-collide kernel on box widths that leave rows with padding, on
boxes smaller than one group or than the grid, and on several boxes of
different sizes in one context: against the FP64 oracle (FP32 storage, the
32^3 parity bar of relative L2 1e-5 on u) and bit for bit against other
launch shapes and against each box alone (every storage)."""
import numpy as np
import pytest

from paper_2503_20605_gb300 import iblb
from paper_2503_20605_gb300 import inputs as I
from gpu_util import oracle_sim, rel_l2, stream

pytestmark = pytest.mark.gpu

W = np.array([1 / 3] + [1 / 18] * 6 + [1 / 36] * 12)
BOXES = [(8, 8, 8), (9, 11, 10), (17, 8, 13), (31, 29, 20), (50, 21, 12), (85, 13, 9), (8, 90, 8), (257, 9, 8)]


def _ctx(boxes, storage, walls=1):
    lats = [iblb.lattice_desc(*b, tau_out=0.8, storage=storage, walls=walls, body_force=(1e-5, -2e-5, 5e-6))
            for b in boxes]
    c = iblb.iblb_batch_create(lats, [iblb.physics_desc() for _ in boxes], stream())
    for k in range(len(boxes)):
        cells = iblb.iblb_info(c, k)["cells"]
        iblb.iblb_set_populations(c, k, I.perturbed_populations(cells, W, 11 + k, 1e-2))
    return c


@pytest.mark.parametrize("box", BOXES)
@pytest.mark.parametrize("walls", [0, 1])
def test_widths_against_oracle(box, walls):
    c = _ctx([box], "f32", walls)
    s = oracle_sim(*box, tau=0.8, walls=walls, body_force=(1e-5, -2e-5, 5e-6))
    try:
        s.set_populations(I.perturbed_populations(iblb.iblb_info(c)["cells"], W, 11, 1e-2))
        iblb.iblb_step(c, 20)
        rho, u = iblb.iblb_get_macros(c, 0)
    finally:
        iblb.iblb_destroy(c)
    s.step(20)
    rho_o, u_o = s.macros()
    assert rel_l2(u, u_o) < 1e-5 and rel_l2(rho, rho_o) < 1e-6


@pytest.mark.parametrize("storage", ["f32", "f16", "bf16"])
def test_batch_and_launch_shapes_give_the_same_bits(storage):
    def run(boxes, *options):
        c = _ctx(boxes, storage)
        try:
            for o, v in options:
                iblb.iblb_set_option(c, o, v)
            iblb.iblb_step(c, 7)
            iblb.iblb_sync(c)
            return [iblb.iblb_get_populations(c, k) for k in range(len(boxes))]
        finally:
            iblb.iblb_destroy(c)
    together = run(BOXES)
    for k, b in enumerate(BOXES):
        c = _ctx([b], storage)
        try:
            # the same inputs as in the batch
            iblb.iblb_set_populations(c, 0, I.perturbed_populations(iblb.iblb_info(c)["cells"], W, 11 + k, 1e-2))
            iblb.iblb_step(c, 7)
            np.testing.assert_array_equal(iblb.iblb_get_populations(c, 0), together[k])
        finally:
            iblb.iblb_destroy(c)
    for options in ([(iblb.IBLB_OPT_LB_GROUP_CELLS, 40)], [(iblb.IBLB_OPT_LB_GROUP_CELLS, 900)],
                    [(iblb.IBLB_OPT_LB_STAGES, 2)], [(iblb.IBLB_OPT_LB_ROW_MULT, 3)]):
        for a, b in zip(run(BOXES, *options), together):
            np.testing.assert_array_equal(a, b)
