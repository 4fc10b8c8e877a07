"""flb_error_location on lattices that make many steps per launch: the earliest step
with an invalid node and the lowest such node in it, whichever block came to its own
first."""
import numpy as np
import pytest

from paper_1204_6734_gb300 import flb, inputs

pytestmark = pytest.mark.gpu


def params(Lx, Ly, precision="fp32"):
    return inputs.LatticeParams(Lx, Ly, 1.0, 0.0, 0.0, 1e-4, inputs.omega_groups(1.1, 0.8, 1.0), "local", precision, seed=5)


def spoiled(p, nodes):
    f = np.ones((9, p.Ly, p.Lx)) * np.array([4 / 9] + [1 / 9] * 4 + [1 / 36] * 4)[:, None, None]
    for n in nodes:
        y, x = divmod(n, p.Lx)
        f[:, y, x] = 0.0
        f[1, y, x] = 1.0   # u = (1, 0): no basis
    return f


@pytest.mark.parametrize("Lx,Ly", [(21, 21), (64, 64), (300, 130), (20, 601), (900, 900)])
def test_lowest_node_of_the_first_step(Lx, Ly):
    p = params(Lx, Ly)
    g = np.random.Generator(np.random.PCG64(1))
    for first in (0, 3 * Lx + 5, p.nodes // 2 + 1):
        bad = np.unique(np.append(g.integers(first, p.nodes, 200), first))
        with flb.Lattice(p) as lat:
            lat.set_populations(spoiled(p, bad))
            assert lat.step(6).launches()[0] <= {"resident", "cut"}
            with pytest.raises(flb.FlbError) as e:
                lat.sync()
            assert e.value.code == flb.ERR_INVALID_VELOCITY
            assert flb.flb_error_location(lat.h) == (first, 0)


def test_step_of_the_first_error_and_later_launches():
    """The step of a launch that started at t = 17, kept by the launches after it; and after
    a reset the next error counts."""
    p = params(300, 130)
    with flb.Lattice(p) as lat:
        lat.step(17)
        f = lat.populations()
        bad = spoiled(p, [11111, 222])
        f[:, 37, 11] = bad[:, 37, 11]
        lat.set_populations(f)
        lat.step(8)
        lat.step(8)
        with pytest.raises(flb.FlbError):
            lat.sync()
        assert flb.flb_error_location(lat.h) == (37 * 300 + 11, 17)
        lat.set_populations(spoiled(p, [222]))
        lat.step(5)
        with pytest.raises(flb.FlbError):
            lat.sync()
        assert flb.flb_error_location(lat.h) == (222, 33)
