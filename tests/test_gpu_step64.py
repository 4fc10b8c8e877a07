"""The FP64 step at the edges of its launch shapes (one node; a last warp that
is not full; sums in a warp of their own, up to two blocks of 32 nodes per SM,
and in the colliding warp above that) against the oracle, with the tolerances
of test_gpu_parity.py: populations 1e-12 of the largest, sums by the same
relative bound on their summands."""
import numpy as np
import pytest

import oracle
from paper_1204_6734_gb300 import flb, inputs

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("Lx,Ly", [(1, 1), (31, 1), (33, 1), (8, 8), (97, 100), (98, 101)])
@pytest.mark.parametrize("basis", ["standard", "local", "lut"])
def test_step64_equals_oracle(Lx, Ly, basis):
    p = inputs.LatticeParams(Lx, Ly, 1.0, 0.1, -0.05, 1e-4, inputs.omega_groups(1.2, 0.8, 1.0), basis, "fp64", seed=3)
    with flb.Lattice(p) as lat:
        lat.set_sampling(1, 2)
        lat.step(4)
        lat.step(3)
        f = lat.populations()
        S1, S2, n = lat.raw_sums()
    ref = oracle.Run(p, warmup=1, every=2).step(7)
    scale = np.abs(ref.f).max()
    assert np.abs(f - ref.f).max() <= 1e-12 * scale
    assert n == ref.nsamp
    dev = np.sqrt(np.diag(ref.S2) / n)          # spread of the deviations
    assert np.all(np.abs(S2 - ref.S2) <= 2e-12 * scale * n * dev.max())
    assert np.all(np.abs(S1 - ref.S1) <= 1e-12 * scale * n)


@pytest.mark.parametrize("Lx,Ly", [(33, 7), (120, 110)])
def test_sums_do_not_depend_on_the_calls(Lx, Ly):
    p = inputs.LatticeParams(Lx, Ly, 1.0, 0.1, 0.0, 1e-4, inputs.omega_groups(1.2, 0.8, 1.0), "local", "fp64", seed=4)
    out = []
    for cuts in ([9], [1] * 9, [4, 5]):
        with flb.Lattice(p) as lat:
            lat.set_sampling(2, 3)
            for k in cuts:
                lat.step(k)
            out.append(lat.raw_sums())
    for S1, S2, n in out[1:]:
        np.testing.assert_array_equal(S1, out[0][0])
        np.testing.assert_array_equal(S2, out[0][1])
        assert n == out[0][2]
