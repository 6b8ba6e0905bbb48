"""iblb_observe_all over more droplets than a grid has blocks in y (65 535):
each droplet's values are those that iblb_observe gives, on both sides of the
limit, with membranes and without."""
import numpy as np
import pytest

from paper_2503_20605_gb300 import iblb
from paper_2503_20605_gb300 import inputs as I
from gpu_util import stream

pytestmark = pytest.mark.gpu

N = 65539
BOX = (8, 8, 8)
W = np.array([1 / 3] + [1 / 18] * 6 + [1 / 36] * 12)


@pytest.mark.parametrize("meshes", [(), (3, 65534, 65535, N - 1)])
def test_every_droplet_of_many(meshes):
    lat, phys = iblb.lattice_desc(*BOX, tau_out=0.9, storage="f16"), iblb.physics_desc(sigma=0.01)
    c = iblb.iblb_batch_create([lat] * N, [phys] * N, stream())
    try:
        cells = iblb.iblb_info(c, 0)["cells"]
        odd = (0, 7, 65534, 65535, 65536, N - 1)
        for k in odd:
            iblb.iblb_set_populations(c, k, I.perturbed_populations(cells, W, 3 + k, 1e-2))
        for k in meshes:
            iblb.iblb_set_membrane(c, k, *I.icosphere(0, 2.0, (4.1, 3.9, 3.5)))
        every = iblb.iblb_observe_all(c, 0.3, 0.2)
        assert len(every) == N
        for k in {*odd, *meshes, 1, 40000}:
            assert iblb.iblb_observe(c, k, 0.3, 0.2) == every[k], k
        for k in range(N):
            if k not in odd:
                assert every[k]["mass"] == cells, k
            assert (every[k]["volume"] > 0.0) == (k in meshes), k
            assert every[k]["status"] == 0, k
        assert len({every[k]["mass"] for k in odd}) == len(odd)
    finally:
        iblb.iblb_destroy(c)
