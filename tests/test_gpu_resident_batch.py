"""Batches whose replicas stay in shared memory for all steps of a call (small
replicas whole, larger ones cut into rows of blocks) against single lattices
stepped one launch at a time: bit-identical populations, and sums within the
bounds of tests/tolerances.py (shapes with tensor-core sums) or the FP32
summation term alone, 2^-13 sqrt(S2_ii S2_jj) (shapes that form FP32 products:
2^-14 per side for partials of at most 1024 products)."""
import numpy as np
import pytest

from paper_1204_6734_gb300 import flb, inputs

from tolerances import assert_sums_close

pytestmark = pytest.mark.gpu


def replica(Lx, Ly, r, basis="local", ux0=0.1, kT=1e-4):
    return inputs.LatticeParams(Lx, Ly, 1.0, ux0, 0.02, kT, inputs.omega_groups(1.2, 0.9, 1.0), basis, "fp32",
                                seed=40 + r, replica=r)


def alone(p, n, warmup, every, fp32_products=False):
    with flb.Lattice(p, kernel="pipelined", pipeline_sampling=1 if fp32_products else None) as lat:
        lat.set_sampling(warmup, every)
        lat.step(n)
        return lat.populations(), lat.raw_sums()


# whole replicas, more of them than CTAs at once or fewer; cut ones; both kinds
SETS = {
    "many_small": [(21, 21)] * 700,
    "uneven_small": [(1, 1), (3, 5), (64, 64), (21, 21), (9, 30), (40, 37)] * 9,
    "few_cut": [(300, 130), (64, 64), (21, 21), (500, 7), (33, 400)],
    "one_cut": [(512, 300)],
}


@pytest.mark.parametrize("name", sorted(SETS))
@pytest.mark.parametrize("tile", ["128x4", "mixed"])
@pytest.mark.parametrize("basis", ["local", "standard", "lut"])
def test_replicas_equal_lattices_alone(name, tile, basis):
    ps = [replica(Lx, Ly, r, basis) for r, (Lx, Ly) in enumerate(SETS[name])]
    with flb.Batch(ps, tile=tile) as b:
        b.set_sampling(1, 2)
        b.step(9)
        b.step(4)
        b.sync()
        for r in list(range(min(len(ps), 7))) + [len(ps) - 1]:
            f, (R1, R2, m) = alone(ps[r], 13, 1, 2, tile == "128x4")
            np.testing.assert_array_equal(b.populations(r), f)
            S1, S2, n = b.raw_sums(r)
            assert n == m
            if tile == "128x4":
                d = np.sqrt(np.diag(R2))
                assert np.all(np.abs(S2 - R2) <= 2.0 ** -13 * np.outer(d, d))
                assert np.all(np.abs(S1 - R1) <= 2.0 ** -13 * np.sqrt(n) * d)
            else:
                assert_sums_close(S1, S2, R1, R2, n, 0.0, 0.0, 0.0)


def test_replicas_join_end_and_leave_between_launches():
    A, B, C = replica(64, 64, 0), replica(300, 100, 1), replica(21, 21, 2)
    pool = sum(flb.flb_batch_replica_bytes(p) for p in (A, B, C))
    with flb.Batch.open("local", 3, pool) as b:
        ka = b.add(A, 14)              # stops at its 14th step, inside a launch
        kb = b.add(B)
        b.set_sampling(0, 1)
        b.step(9)
        kc = b.add(C)
        b.set_sampling(0, 1, slot=kc)
        b.step(10)
        assert b.replica_time(ka) == 14 and b.replica_time(kb) == 19 and b.replica_time(kc) == 10
        fa, sa = b.populations(ka), b.raw_sums(ka)
        b.remove(ka)
        b.step(2)                      # one launch per step
        b.step(6)
        got = [(fa, sa), (b.populations(kb), b.raw_sums(kb)), (b.populations(kc), b.raw_sums(kc))]
    for (f, s), (p, n) in zip(got, ((A, 14), (B, 27), (C, 18))):
        g, (R1, R2, m) = alone(p, n, 0, 1, True)
        np.testing.assert_array_equal(f, g)
        assert s[2] == m
        d = np.sqrt(np.diag(R2))
        assert np.all(np.abs(s[1] - R2) <= 2.0 ** -13 * np.outer(d, d))


def test_replicas_that_forbid_staging_sample_in_single_steps():
    ps = [replica(21, 21, 0, kT=0.0), replica(30, 20, 1)]
    with flb.Batch(ps) as b:
        b.set_sampling(0, 1)
        b.step(7)
        for r, p in enumerate(ps):
            f, (R1, R2, m) = alone(p, 7, 0, 1, True)
            np.testing.assert_array_equal(b.populations(r), f)
            assert b.raw_sums(r)[2] == m
