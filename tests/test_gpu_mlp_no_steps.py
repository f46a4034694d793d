"""Training for no steps leaves the network as it is and reports the last loss
(0 before any)."""
import numpy as np
import pytest

from paper_2407_11349_gb300.hawkes import MLP

pytestmark = pytest.mark.gpu


def test_no_steps():
    rng = np.random.default_rng(1)
    net = MLP(0, seed=1)
    try:
        net.set_data(rng.normal(size=(200, 6)), rng.normal(size=(200, 7)))
        assert net.train(0, batch=64, lr=1e-3, seed=1) == 0.0
        last = net.train(3, batch=64, lr=1e-3, seed=1)
        p = net.get_params()
        assert last > 0.0
        assert net.train(0, batch=64, lr=1e-3, seed=1) == last
        assert np.array_equal(net.get_params(), p)
    finally:
        net.close()
