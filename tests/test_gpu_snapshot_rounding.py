"""A snapshot's velocities are quotients rounded once.  With FP16 storage the
offsets are multiples of 2^-24 and their sums exact, so rho and U have one
correctly rounded FP64 value each, which numpy's division gives too: every bit
is the same."""
import numpy as np
import pytest

from paper_2503_20605_gb300 import iblb
from gpu_util import gpu_ctx

pytestmark = pytest.mark.gpu

W = np.array([1 / 3] + [1 / 18] * 6 + [1 / 36] * 12)
C = np.array([(0, 0, 0), (1, 0, 0), (-1, 0, 0), (0, 1, 0), (0, -1, 0), (0, 0, 1), (0, 0, -1), (1, 1, 0), (-1, -1, 0),
              (1, -1, 0), (-1, 1, 0), (0, 1, 1), (0, -1, -1), (0, 1, -1), (0, -1, 1), (1, 0, 1), (-1, 0, -1),
              (1, 0, -1), (-1, 0, 1)], float)


@pytest.mark.parametrize("amp", [1e-3, 0.3])
@pytest.mark.parametrize("box", [(8, 9, 10), (129, 20, 12)])
def test_velocities_are_rounded_once(box, amp):
    force = (1e-4, -2e-4, 3e-4)
    c = gpu_ctx(*box, tau=0.9, storage="f16", body_force=force)
    try:
        cells = iblb.iblb_info(c)["cells"]
        o = (amp * np.random.default_rng(9).uniform(-1.0, 1.0, (19, cells))).astype(np.float16).astype(float)
        iblb.iblb_set_populations(c, 0, W[:, None] + o)
        back = iblb.iblb_get_populations(c, 0).reshape(19, cells)
        o = (back - W[:, None]).astype(np.float16).astype(float)           # the offsets as stored
        rho, u = iblb.iblb_get_macros(c, 0)
    finally:
        iblb.iblb_destroy(c)
    F = np.array(force).astype(np.float32).astype(float)
    want_rho = 1.0 + o.sum(0)
    want_u = (C.T @ o - 0.5 * F[:, None]) / want_rho
    np.testing.assert_array_equal(np.asarray(rho), want_rho)
    np.testing.assert_array_equal(np.asarray(u).reshape(3, cells), want_u)


def test_blown_up_cells_divide_as_ever():
    """FP32 storage: density 0, infinite, not a number, huge and tiny, and
    momentum 0, tiny, huge: the quotients of numpy's division, cell by cell."""
    rest = [0.0, -1.0, np.inf, -np.inf, np.nan, 3e38, -3e38, 1e-30, -1.0 + 2.0 ** -24, 0.25]
    mom = [0.0, 1e-38, 1e-45, -1e-45, 3e37, 1e-3, np.inf]
    c = gpu_ctx(len(rest) * len(mom), 8, 8, storage="f32")
    try:
        nx = len(rest) * len(mom)
        f = np.repeat(W, 8 * 6 * nx).reshape(19, 48, nx)
        o = np.zeros((19, nx), np.float32)
        o[0], o[1] = np.repeat(np.array(rest, np.float32), len(mom)), np.tile(np.array(mom, np.float32), len(rest))
        f = f + o.astype(float)[:, None, :]
        iblb.iblb_set_populations(c, 0, f.ravel())
        back = iblb.iblb_get_populations(c, 0).reshape(19, 48, nx)
        rho, u = iblb.iblb_get_macros(c, 0)
    finally:
        iblb.iblb_destroy(c)
    o = (back - W[:, None, None]).astype(np.float32).astype(float)
    rho, u = np.asarray(rho).reshape(48, nx), np.asarray(u).reshape(3, 48, nx)
    with np.errstate(all="ignore"):
        for e, m in enumerate((o[1] - o[2], o[3] - o[4], o[5] - o[6])):
            np.testing.assert_array_equal(u[e], m / rho)
