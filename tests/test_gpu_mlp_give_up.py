"""A network whose wait has given up takes no further step: training reports
IBLB_E_TIMEOUT and leaves parameters and moments as they were, and the next
call works on (the wait is recorded by the self-test, as no wait of these
kernels can be made to run out)."""
import numpy as np
import pytest

from paper_2503_20605_gb300 import iblb
from paper_2503_20605_gb300 import inputs as I
from gpu_util import stream

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("batch", [1, 128, 300])     # one cluster, three clusters and two staged chunks
def test_no_step_after_a_wait_gave_up(batch):
    x = I.warmstart_cases(2 * batch, 5)
    y = 1.0 + 0.1 * np.random.default_rng(5).normal(size=(2 * batch, 64))
    m, other = (iblb.iblb_mlp_create(I.mlp_init(4), batch, stream()) for _ in range(2))
    try:
        before = iblb.iblb_mlp_get_params(m)
        for call in (lambda: iblb.iblb_mlp_train(m, x, y, 3, batch, 1e-3, 1), lambda: iblb.iblb_mlp_grad(m, x[:batch], y[:batch]),
                     lambda: iblb.iblb_mlp_predict(m, x)):
            iblb.iblb_selftest_mlp_give_up(m)
            with pytest.raises(iblb.IblbError) as e:
                call()
            assert e.value.code == iblb.IBLB_E_TIMEOUT
            np.testing.assert_array_equal(iblb.iblb_mlp_get_params(m), before)
        # the moments too: the gradient is that of an untouched network, and so is the first step's direction
        g, loss = iblb.iblb_mlp_grad(m, x[:batch], y[:batch])
        g2, loss2 = iblb.iblb_mlp_grad(other, x[:batch], y[:batch])
        np.testing.assert_array_equal(g, g2)
        assert loss == loss2
        iblb.iblb_mlp_train(m, x, y, 1, batch, 1e-3, 1)
        moved = iblb.iblb_mlp_get_params(m)
        assert np.all(np.isfinite(moved)) and np.any(moved != before)
    finally:
        iblb.iblb_mlp_destroy(m)
        iblb.iblb_mlp_destroy(other)
