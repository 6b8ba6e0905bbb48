"""The force kernel's kernel supports and tile lists where positions and tiles
are not the ordinary ones: boxes whose sides end on a partial tile of 1, 2 or
3 cells (supports over three tiles an axis), membranes across every periodic
seam, at negative coordinates and beyond the box, nodes exactly on lattice
points and half-way, nodes within a few thousandths of a cell of the wall
plane without the near-wall guard.  Forces and force density against the
oracle with the bars of the parity tests."""
import numpy as np
import pytest

import oracle.oracle as O
from paper_2503_20605_gb300 import iblb
from paper_2503_20605_gb300 import inputs as I
from gpu_util import pair, rel_l2, stream

pytestmark = pytest.mark.gpu


def _check(xyz, tri, bar=1e-5, **kw):
    g, s = pair(mesh=(xyz, tri), tau=0.9, sigma=0.02, **kw)
    try:
        iblb.iblb_compute_forces(g)
        phi = iblb.iblb_get_node_forces(g, 0)
        F = iblb.iblb_get_force_density(g, 0)
    finally:
        iblb.iblb_destroy(g)
    want = O.membrane_forces(s.p, xyz, tri)[0]
    assert rel_l2(phi, want) < bar
    assert rel_l2(F, O.spread(s.p, xyz, want)) < bar


@pytest.mark.parametrize("box", [(16, 16, 16), (17, 18, 19), (9, 10, 11), (13, 14, 15)])
@pytest.mark.parametrize("shift", [(0.0, 0.0, 0.0), (-3.7, 20.3, 0.0), (31.25, -16.5, 0.0)])
def test_partial_tiles_and_seams(box, shift):
    xyz, tri = I.icosphere(2, 3.0, (1.3, box[1] - 1.2, box[2] / 2))
    _check(I.jitter_nodes(xyz, 3, 0.1) + np.array(shift), tri, nx=box[0], ny=box[1], nz=box[2], walls=0)


def test_seams_in_z():
    xyz, tri = I.icosphere(3, 5.0, (8.0, 8.0, 0.4))
    _check(xyz, tri, nx=17, ny=16, nz=15, walls=0)
    _check(xyz + np.array([0.0, 0.0, -15.0]), tri, nx=17, ny=16, nz=15, walls=0)


def test_nodes_on_lattice_points_and_midpoints():
    xyz, tri = I.icosphere(1, 6.0, (12.0, 12.0, 10.0))       # edges of 3 cells: snapping leaves no face degenerate
    xyz[::4] = np.round(xyz[::4])
    xyz[1::4] = np.round(xyz[1::4] * 2.0) / 2.0
    _check(xyz, tri, nx=24, ny=24, nz=22, theta=70.0, xi=2.0)


@pytest.mark.parametrize("gap", [3e-3, 0.01, 0.3])
def test_heights_near_the_wall_without_a_guard(gap):
    xyz, tri = I.icosphere(2, 3.0, (8.0, 8.0, 0.5 + 3.0 + gap))
    xyz[:, 2] = np.maximum(xyz[:, 2], 0.5 + gap)
    _check(xyz, tri, nx=16, ny=16, nz=16, theta=120.0, xi=1.5, h_min_frac=0.0)


@pytest.mark.parametrize("n", [3, 4, 5])
def test_block_order_of_large_batches(n):
    """From 16 blocks an SM on (four L5 meshes on 152 SMs) the force kernel's
    blocks take their pieces in another order, the grid rounded up to whole
    pieces: every droplet as alone, bit for bit."""
    box = 64
    meshes = [I.icosphere(5, 20.0 + 0.5 * k, (32.2, 31.7, 31.5 + 0.1 * k)) for k in range(n)]

    def run(ms):
        c = iblb.iblb_batch_create([iblb.lattice_desc(box, box, box, tau_out=0.9) for _ in ms],
                                   [iblb.physics_desc(sigma=0.01, theta_eq_deg=80.0, xi=2.0) for _ in ms], stream())
        try:
            for k, m in enumerate(ms):
                iblb.iblb_set_membrane(c, k, *m)
            iblb.iblb_step(c, 2)
            return [(iblb.iblb_get_nodes(c, k), iblb.iblb_get_node_forces(c, k)) for k in range(len(ms))]
        finally:
            iblb.iblb_destroy(c)

    together = run(meshes)
    for m, (xyz, phi) in zip(meshes, together):
        alone = run([m])[0]
        np.testing.assert_array_equal(xyz, alone[0])
        np.testing.assert_array_equal(phi, alone[1])
