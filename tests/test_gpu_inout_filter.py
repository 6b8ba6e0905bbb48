"""The in/out flags where their FP32 decisions must hand over to FP64: meshes
with vertices, edges and faces exactly on lattice columns and layers, faces
far larger and far smaller than a cell, jittered and rotated spheres across
the periodic seams, widths around a 32-bit word and a 128-column row; bit for
bit against the oracle, again after the droplet has moved (words that were
set must be cleared), and in a batch with a droplet of one viscosity."""
import numpy as np
import pytest

import oracle.oracle as O
from paper_2503_20605_gb300 import iblb
from paper_2503_20605_gb300 import inputs as I
from gpu_util import gpu_ctx, oracle_sim, stream

pytestmark = pytest.mark.gpu

OCT = np.array([(1, 0, 0), (-1, 0, 0), (0, 1, 0), (0, -1, 0), (0, 0, 1), (0, 0, -1)], float)
OCT_TRI = np.array([(0, 2, 4), (2, 1, 4), (1, 3, 4), (3, 0, 4), (2, 0, 5), (1, 2, 5), (3, 1, 5), (0, 3, 5)], np.int32)


def _rotated(level, R, c, seed, jitter=0.0):
    xyz, tri = I.icosphere(level, R)
    q, _ = np.linalg.qr(np.random.default_rng(seed).normal(size=(3, 3)))
    if np.linalg.det(q) < 0:
        q[:, 0] = -q[:, 0]
    return I.jitter_nodes(xyz @ q.T, seed, jitter) + np.asarray(c), tri


def _flags(box, xyz, tri, walls=1):
    g = gpu_ctx(*box, tau=0.8, lam=4.0, walls=walls, mesh=(xyz, tri))
    s = oracle_sim(*box, tau=0.8, lam=4.0, walls=walls)
    try:
        iblb.iblb_compute_forces(g)
        a = iblb.iblb_get_inside(g, 0)
        moved = xyz + np.array([7.0, -3.25, 1.5])
        iblb.iblb_set_nodes(g, 0, moved)
        iblb.iblb_compute_forces(g)
        b = iblb.iblb_get_inside(g, 0)
    finally:
        iblb.iblb_destroy(g)
    assert a.any()
    np.testing.assert_array_equal(a, O.inside(s.p, xyz, tri).ravel())
    np.testing.assert_array_equal(b, O.inside(s.p, moved, tri).ravel())


@pytest.mark.parametrize("scale", [5.0, 10.0, 0.75 * 12])
@pytest.mark.parametrize("shift", [(0, 0, 0), (0.5, 0, 0), (0.25, 0.5, 0.125)])
def test_octahedron_on_lattice_planes(scale, shift):
    _flags((33, 32, 34), OCT * scale + np.array([16.0, 15.0, 13.0]) + shift, OCT_TRI)


@pytest.mark.parametrize("box,walls", [((31, 30, 40), 1), ((32, 33, 36), 1), ((129, 40, 38), 1), ((40, 64, 36), 0)])
@pytest.mark.parametrize("level,jitter", [(1, 0.0), (3, 0.2), (4, 0.01)])
def test_rotated_spheres(box, walls, level, jitter):
    for seed in range(3):
        xyz, tri = _rotated(level, 9.0, (box[0] - 4.3, 3.0 + seed, 15.5), seed, jitter)
        _flags(box, xyz, tri, walls)


def test_nodes_on_columns_and_layers():
    xyz, tri = _rotated(3, 8.0, (16.0, 16.0, 14.0), 2)
    xyz[::3] = np.round(xyz[::3])                 # a third of the nodes on lattice points
    _flags((32, 32, 32), xyz, tri)


def test_batch_with_one_viscosity_beside_two():
    boxes = [(40, 24, 30), (31, 33, 28), (24, 24, 30)]
    lam = [3.0, 1.0, 0.4]
    c = iblb.iblb_batch_create([iblb.lattice_desc(*b, tau_out=0.9, lam=v) for b, v in zip(boxes, lam)],
                               [iblb.physics_desc(sigma=0.01, theta_eq_deg=90.0, xi=2.0) for _ in boxes], stream())
    try:
        meshes = [_rotated(3, 7.0, (b[0] / 2 + 0.3, b[1] / 2, 10.2), k) for k, b in enumerate(boxes)]
        for k, m in enumerate(meshes):
            iblb.iblb_set_membrane(c, k, *m)
        iblb.iblb_compute_forces(c)
        for k, b in enumerate(boxes):
            got = iblb.iblb_get_inside(c, k)
            s = oracle_sim(*b, tau=0.9, lam=lam[k])
            want = O.inside(s.p, *meshes[k]).ravel() if lam[k] != 1.0 else np.zeros_like(got)
            np.testing.assert_array_equal(got, want)
    finally:
        iblb.iblb_destroy(c)


@pytest.mark.parametrize("level,R,box,n", [(1, 6.0, 24, 1), (3, 8.0, 28, 2), (6, 34.0, 80, 4)])
def test_crossings_from_the_spread_and_from_their_own_kernel(level, R, box, n):
    """One kernel per stage lets the spread's blocks take the faces (from far
    fewer faces than threads to several passes over them); with the fused
    membrane kernels they have a launch of their own."""
    meshes = [_rotated(level, R, (box / 2 + 0.3, box / 2, box / 2 - 0.2), k) for k in range(n)]
    got = []
    for fused in (0, 1):
        c = iblb.iblb_batch_create([iblb.lattice_desc(box, box, box, tau_out=0.9, lam=2.0) for _ in meshes],
                                   [iblb.physics_desc(sigma=0.01, theta_eq_deg=90.0, xi=2.0) for _ in meshes],
                                   stream())
        try:
            iblb.iblb_set_option(c, iblb.IBLB_OPT_FUSED_IB, fused)
            for k, m in enumerate(meshes):
                iblb.iblb_set_membrane(c, k, *m)
            iblb.iblb_step(c, 3)
            got.append([(iblb.iblb_get_inside(c, k), iblb.iblb_get_nodes(c, k)) for k in range(n)])
        finally:
            iblb.iblb_destroy(c)
    for (ia, na), (ib, nb) in zip(*got):
        assert ia.any()
        np.testing.assert_array_equal(ia, ib)
        np.testing.assert_array_equal(na, nb)
