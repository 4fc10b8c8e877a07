"""Wide lattices of some hundred rows: cut across x, every pass of a block would hold
lanes on an edge and wait there, so they take one launch per step; low ones (few
rows to a block) are cut, and agree with it bit for bit."""
import numpy as np
import pytest

from paper_1204_6734_gb300 import flb, inputs

pytestmark = pytest.mark.gpu


def params(Lx, Ly, basis="local"):
    return inputs.LatticeParams(Lx, Ly, 1.0, 0.1, 0.02, 1e-4, inputs.omega_groups(1.2, 0.9, 1.0), basis, "fp32", seed=8)


@pytest.mark.parametrize("Lx,Ly", [(5000, 100), (3000, 150), (2500, 200), (2879, 166), (1648, 176), (1147, 319)])
@pytest.mark.parametrize("every", [0, 1])
def test_not_cut_across_x(Lx, Ly, every):
    with flb.Lattice(params(Lx, Ly)) as lat:
        lat.set_sampling(0, every)
        assert lat.step(8).launches() == ({"step"}, 8)


@pytest.mark.parametrize("Lx,Ly", [(4000, 20), (8000, 10), (30000, 9), (2000, 60), (4001, 50)])
def test_low_ones_are(Lx, Ly):
    p = params(Lx, Ly)
    out = []
    for kernel in (None, "pipelined"):
        with flb.Lattice(p, kernel=kernel) as lat:
            lat.set_sampling(0, 1)
            assert lat.step(8).launches() == (({"cut"}, 1) if kernel is None else ({"step"}, 8))
            out.append((lat.populations(), lat.raw_sums()))
    np.testing.assert_array_equal(out[0][0], out[1][0])
    assert out[0][1][2] == out[1][1][2]
