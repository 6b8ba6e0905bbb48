"""Observables and snapshots over several droplets and at the ends of the
kernels' ranges: every droplet of a batch gives the same bits through
iblb_observe_all, iblb_observe and alone, for meshes from 12 nodes to several
hundred chunks; the mesh part matches the oracle (FP64, sums of up to 1e5
terms in another order: 1e-12 relative); rho and U of a snapshot match numpy
on the stored populations, on both sides of the FP16 kernel's integer range."""
import numpy as np
import pytest

import oracle.oracle as O
from paper_2503_20605_gb300 import iblb
from paper_2503_20605_gb300 import inputs as I
from gpu_util import gpu_ctx, stream

pytestmark = pytest.mark.gpu

C = np.array([(0, 0, 0), (1, 0, 0), (-1, 0, 0), (0, 1, 0), (0, -1, 0), (0, 0, 1), (0, 0, -1), (1, 1, 0), (-1, -1, 0),
              (1, -1, 0), (-1, 1, 0), (0, 1, 1), (0, -1, -1), (0, 1, -1), (0, -1, 1), (1, 0, 1), (-1, 0, -1),
              (1, 0, -1), (-1, 0, 1)], float)
MESHES = [((24, 20, 26), 0, 5.0), ((33, 30, 28), 2, 7.0), ((40, 41, 34), 3, 9.0), ((70, 66, 60), 5, 20.0)]


def test_every_droplet_alike_in_any_call():
    lats = [iblb.lattice_desc(*b, tau_out=0.9, storage="f16") for b, _, _ in MESHES]
    phys = [iblb.physics_desc(sigma=0.01, theta_eq_deg=60.0, xi=2.0, volume_correction=k % 2)
            for k in range(len(MESHES))]
    meshes = [I.icosphere(lv, R, (b[0] / 2 + 0.2, b[1] / 2, 2.5 + R)) for b, lv, R in MESHES]
    c = iblb.iblb_batch_create(lats, phys, stream())
    try:
        for k, m in enumerate(meshes):
            iblb.iblb_set_membrane(c, k, *m)
        iblb.iblb_step(c, 5)
        every = iblb.iblb_observe_all(c, 0.3, 0.2)
        each = [iblb.iblb_observe(c, k, 0.3, 0.2) for k in range(len(MESHES))]
        nodes = [iblb.iblb_get_nodes(c, k) for k in range(len(MESHES))]
    finally:
        iblb.iblb_destroy(c)
    assert every == each
    for k, m in enumerate(meshes):
        a = iblb.iblb_create(lats[k], phys[k], stream())
        try:
            iblb.iblb_set_membrane(a, 0, *m)
            iblb.iblb_step(a, 5)
            assert iblb.iblb_observe(a, 0, 0.3, 0.2) == every[k]
            np.testing.assert_array_equal(iblb.iblb_get_nodes(a, 0), nodes[k])
        finally:
            iblb.iblb_destroy(a)
        R0 = (3.0 * O.mesh_volume(*m) / (4.0 * np.pi)) ** (1.0 / 3.0)
        want = O.mesh_observe(nodes[k], m[1], R0, zcut_frac=0.3, eps_flat=0.2)
        for key in ("volume", "area", "zmin", "zmax", "rc_cut", "n_cut", "chi_flat"):
            assert every[k][key] == pytest.approx(want[key], rel=1e-12), key


@pytest.mark.parametrize("storage", ["f32", "f16", "bf16"])
@pytest.mark.parametrize("amp", [1e-3, 0.9, 60.0])
@pytest.mark.parametrize("box", [(8, 9, 10), (129, 8, 9)])
def test_snapshot_matches_stored_populations(storage, amp, box):
    c = gpu_ctx(*box, tau=0.9, storage=storage, body_force=(1e-4, -2e-4, 3e-4))
    try:
        cells = iblb.iblb_info(c)["cells"]
        f = 1.0 + amp * np.random.default_rng(4).uniform(0.2, 1.0, (19, cells))
        iblb.iblb_set_populations(c, 0, f)
        f = iblb.iblb_get_populations(c, 0).reshape(19, cells)
        rho, u = iblb.iblb_get_macros(c, 0)
    finally:
        iblb.iblb_destroy(c)
    F = np.array([1e-4, -2e-4, 3e-4]).astype(np.float32).astype(float)
    want = (C.T @ f - 0.5 * F[:, None]) / f.sum(0)
    # FP64 sums of 19 terms of size up to 61: a few units of 61 * 2^-52
    assert np.abs(rho / f.sum(0) - 1.0).max() < 1e-14
    assert np.abs(u.reshape(3, cells) - want).max() < 1e-13
