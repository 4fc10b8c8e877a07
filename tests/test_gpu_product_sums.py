"""Correlation sums with FP32 products (batches in the 128x4 and 64x8 shapes, the FP16
store) against FP64 sums of the very states they sampled, so that nothing but the
rounding of the sums themselves is left.

Products of FP32 numbers are added up in FP32, rounded to nearest, in chains of
at most K = 260 (a lane's share of a warp's 1024 nodes, and two more sums), then in
FP64. A chain's partial sums grow to its total, so a chain is off by about
sqrt(K / 3) 2^-24 / sqrt(3) of it, without bias, and the sum of M chains by that over
sqrt(M). With K / M below 1 / 200 in each case here, four of these are
4 / 3 sqrt(1 / 200) 2^-24 < 2^-27; the bound is twice that, of sqrt(S2_ii S2_jj). (Sums
that cut off instead of rounding are 2^-24 too small and more.)"""
import numpy as np
import pytest

import oracle
from paper_1204_6734_gb300 import flb, inputs

pytestmark = pytest.mark.gpu

BOUND = 2.0 ** -26


def params(Lx, Ly, r=0, precision="fp32", basis="local", kT=1e-4):
    return inputs.LatticeParams(Lx, Ly, 1.0, 0.1, 0.02, kT, inputs.omega_groups(1.2, 0.9, 1.0), basis, precision,
                                seed=30 + r, replica=r)


def check(S1, S2, n, states, p):
    # the kernels subtract c = f^0(rho0, u0) as FP32 numbers
    c = oracle.init_equilibrium(p)[:, :1, 0].astype(np.float32).astype(np.float64)
    R1, R2, m = np.zeros(9), np.zeros((9, 9)), 0
    for f in states:
        d = f.reshape(9, -1) - c
        R1 += d.sum(1)
        R2 += d @ d.T
        m += d.shape[1]
    assert n == m
    q = np.sqrt(np.diag(R2))
    assert np.abs((S2 - R2) / np.outer(q, q)).max() <= BOUND
    assert np.abs((S1 - R1) / (q * np.sqrt(n))).max() <= BOUND


@pytest.mark.parametrize("shapes,kinds", [([(21, 21)] * 24, {"resident"}), ([(9, 7)] * 200, {"resident"}),
                                          ([(64, 64)] * 8, {"cut"}), ([(300, 48)] * 2, {"cut"})])
@pytest.mark.parametrize("tile", ["128x4", "64x8"])
@pytest.mark.parametrize("kT", [1e-4, 1e-3])
def test_batches(shapes, kinds, tile, kT):
    ps = [params(Lx, Ly, r, kT=kT) for r, (Lx, Ly) in enumerate(shapes)]
    n = 40
    with flb.Batch(ps, tile=tile) as b, flb.Batch(ps, tile=tile, kernel="pipelined") as w:
        b.set_sampling(0, 1)
        b.step(n)
        assert b.launches()[0] == kinds
        sums = [b.raw_sums(r) for r in range(len(ps))]
        states = []
        for _ in range(n):
            states += [w.populations(r) for r in range(len(ps))]
            w.step(1)
    check(sum(s[0] for s in sums), sum(s[1] for s in sums), sum(s[2] for s in sums), states, ps[0])


@pytest.mark.parametrize("Lx,Ly,n,kinds", [(21, 21, 500, {"resident"}), (300, 130, 30, {"cut"}), (257, 129, 30, {"cut"}),
                                           (900, 900, 4, {"step"}), (2000, 700, 2, {"step"})])
@pytest.mark.parametrize("basis", ["local", "standard", "lut"])
def test_fp16_store(Lx, Ly, n, kinds, basis):
    p = params(Lx, Ly, precision="fp16dev", basis=basis)
    with flb.Lattice(p) as lat, flb.Lattice(p) as w:
        w.step(3)
        lat.step(3)
        lat.set_sampling(3, 1)
        assert lat.step(n).launches()[0] == kinds
        S1, S2, m = lat.raw_sums()

        def states():
            for _ in range(n):
                yield w.populations()
                w.step(1)
        check(S1, S2, m, states(), p)


@pytest.mark.parametrize("shapes,kinds", [([(21, 21)] * 3, {"resident"}), ([(30, 30)] * 700, {"resident"}),
                                          ([(64, 64)] * 8, {"cut"}), ([(300, 130)], {"cut"})])
def test_partials_of_the_warps_meet_in_fp64(shapes, kinds):
    """Deviations k 2^-25, 2^15 <= k < 2^16, from populations that are powers of two: the
    sum of the 256 nodes that a warp takes at most here is exact in FP32, that of all
    warps is not, so S1 is exact only if the warps' partials are added in FP64 (or as
    it would)."""
    ps = [inputs.LatticeParams(Lx, Ly, 36 / 64, 0.0, 0.0, 1e-4, inputs.omega_groups(1.2, 0.9, 1.0), "local", "fp32",
                               seed=r, replica=r) for r, (Lx, Ly) in enumerate(shapes)]
    c = np.array([16] + [4] * 4 + [1] * 4)[:, None] / 64   # f^0 of rho = 36 / 64 at rest
    g = np.random.Generator(np.random.PCG64(4))
    with flb.Batch(ps) as b:
        want = {}
        for r in (0, len(ps) - 1):
            p = ps[r]
            d = g.integers(2 ** 15, 2 ** 16, (9, p.nodes)) * 2.0 ** -25
            b.set_populations(r, (c + d).reshape(9, p.Ly, p.Lx))
            want[r] = d.sum(1)
        b.set_sampling(0, 1000)
        b.step(4)
        assert b.launches()[0] == kinds
        for r, s in want.items():
            S1, _, n = b.raw_sums(r)
            assert n == ps[r].nodes
            np.testing.assert_array_equal(S1, s)
