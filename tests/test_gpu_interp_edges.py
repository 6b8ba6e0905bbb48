"""The interpolation's support rows where they wrap, leave the fluid or span
the whole box: one step of a free membrane carried by a uniform stream moves
every node by exactly that velocity where its support lies in the fluid
(the kernel's partition of unity, FP32 arithmetic on weights that sum to one
within a few ulp: 1e-6 relative), in boxes down to 8 cells a side; and one
step against the oracle at walls and across the periodic seams."""
import numpy as np
import pytest

from paper_2503_20605_gb300 import iblb
from paper_2503_20605_gb300 import inputs as I
from gpu_util import gpu_ctx, pair

pytestmark = pytest.mark.gpu

W = np.array([1 / 3] + [1 / 18] * 6 + [1 / 36] * 12)
C = np.array([(0, 0, 0), (1, 0, 0), (-1, 0, 0), (0, 1, 0), (0, -1, 0), (0, 0, 1), (0, 0, -1), (1, 1, 0), (-1, -1, 0),
              (1, -1, 0), (-1, 1, 0), (0, 1, 1), (0, -1, -1), (0, 1, -1), (0, -1, 1), (1, 0, 1), (-1, 0, -1),
              (1, 0, -1), (-1, 0, 1)], float)


@pytest.mark.parametrize("box", [(8, 8, 8), (9, 10, 11), (13, 8, 21)])
@pytest.mark.parametrize("level", [0, 2])
def test_uniform_stream_moves_every_node_alike(box, level):
    U = np.array([0.03, -0.02, 0.011])
    cu = C @ U
    f = W * (1 + 3 * cu + 4.5 * cu ** 2 - 1.5 * U @ U)
    xyz, tri = I.icosphere(level, 2.1, (0.4, box[1] - 0.3, 0.2))      # across the seams of every axis
    c = gpu_ctx(*box, tau=0.8, walls=0, mesh=(xyz, tri))
    try:
        iblb.iblb_set_populations(c, 0, np.repeat(f, box[0] * box[1] * box[2]))
        iblb.iblb_step(c, 1)
        iblb.iblb_sync(c)
        moved = iblb.iblb_get_nodes(c, 0) - xyz
    finally:
        iblb.iblb_destroy(c)
    assert np.abs(moved - U).max() < 1e-6 * np.abs(U).max()


def test_step_at_the_wall_and_across_seams():
    xyz, tri = I.icosphere(2, 3.0, (0.7, 15.6, 0.5 + 3.0 + 0.6))
    xyz = I.jitter_nodes(xyz, 3, 0.05)
    g, s = pair(nx=17, ny=16, nz=14, tau=0.9, sigma=0.02, theta=80.0, xi=1.5, mesh=(xyz, tri))
    try:
        f = I.perturbed_populations(iblb.iblb_info(g)["cells"], W, 5, 1e-2)
        iblb.iblb_set_populations(g, 0, f)
        s.set_populations(f)
        iblb.iblb_step(g, 3)
        iblb.iblb_sync(g)
        q = iblb.iblb_get_nodes(g, 0)
    finally:
        iblb.iblb_destroy(g)
    s.step(3)
    # FP32 velocities of order 0.01 over three steps
    assert np.abs(q - s.nodes()).max() < 3e-7
