"""Boxes whose rows are the longest that the stream-collide kernel takes (two
stages of one row in a block's shared memory: 1316 cells in FP32, 2320 in 16
bits), alone, several in a context, and with two viscosities.  What a droplet
does there in a few steps, which it reaches no further than that many cells, is
bit for bit what it does in a short box, and longer rows are refused with an
error as ever."""
import numpy as np
import pytest

from paper_2503_20605_gb300 import iblb
from paper_2503_20605_gb300 import inputs as I
from gpu_util import stream

pytestmark = pytest.mark.gpu

NY, NZ, STEPS, SHORT = 17, 16, 6, 48
MESH = I.icosphere(2, 4.0, (22.3, 8.2, 6.6))        # reaches x = 22.3 +- (4 + 2 + STEPS) at most


def run(nx, storage, lam, several):
    lat = iblb.lattice_desc(nx, NY, NZ, tau_out=0.8, lam=lam, storage=storage)
    phys = iblb.physics_desc(sigma=0.02, theta_eq_deg=70.0, xi=2.0)
    lats, physs = [lat], [phys]
    if several:
        lats.append(iblb.lattice_desc(9, 8, 8, tau_out=0.9, storage=storage))
        physs.append(iblb.physics_desc())
    c = iblb.iblb_batch_create(lats, physs, stream())
    try:
        iblb.iblb_set_membrane(c, 0, *MESH)
        iblb.iblb_step(c, STEPS)
        iblb.iblb_sync(c)
        f = iblb.iblb_get_populations(c, 0).reshape(19, NZ - 2, NY, nx)
        return f, np.asarray(iblb.iblb_get_inside(c, 0)).reshape(NZ - 2, NY, nx), iblb.iblb_get_nodes(c, 0)
    finally:
        iblb.iblb_destroy(c)


@pytest.mark.parametrize("several", [False, True])
@pytest.mark.parametrize("lam", [1.0, 5.0])
@pytest.mark.parametrize("storage,nx", [("f32", 1309), ("f32", 1313), ("f32", 1316), ("f16", 2305), ("f16", 2313),
                                        ("f16", 2320), ("bf16", 2320)])
def test_longest_rows_give_the_short_boxes_bits(storage, nx, lam, several):
    f, inside, q = run(nx, storage, lam, several)
    f0, inside0, q0 = run(SHORT, storage, lam, False)
    np.testing.assert_array_equal(q, q0)
    np.testing.assert_array_equal(f[..., :SHORT - 8], f0[..., :SHORT - 8])
    np.testing.assert_array_equal(inside[..., :SHORT - 8], inside0[..., :SHORT - 8])
    assert inside.any() == (lam != 1.0)
    assert np.all(f[..., SHORT:] == f[:, :, :, -1:])              # at rest


@pytest.mark.parametrize("storage,nx", [("f32", 1317), ("f16", 2321), ("bf16", 8188)])
def test_longer_rows_are_refused(storage, nx):
    with pytest.raises(iblb.IblbError) as e:
        run(nx, storage, 1.0, False)
    assert e.value.code == iblb.IBLB_E_CUDA
    run(SHORT, storage, 1.0, False)
