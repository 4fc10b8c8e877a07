"""Calls of very many steps, with the results of shorter calls."""
import numpy as np
import pytest

from paper_1204_6734_gb300 import flb, inputs

pytestmark = pytest.mark.gpu


def params(Lx, Ly, seed=3):
    return inputs.LatticeParams(Lx, Ly, 1.0, 0.1, 0.02, 1e-4, inputs.omega_groups(1.2, 0.9, 1.0), "local", "fp32",
                                seed=seed)


def test_batch_past_a_million_steps():
    n = 2 ** 20 + 5
    ps = [params(9, 9, r) for r in range(3)]
    with flb.Batch(ps) as b:
        b.step(n)
        kinds, launches = b.launches()
        assert kinds == {"resident"} and 1 < launches < n // 1000
        b.sync()
        assert b.t == n
        with flb.Lattice(ps[2]) as lat:
            np.testing.assert_array_equal(b.populations(2), lat.step(n).populations())
