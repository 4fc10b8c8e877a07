"""Batches of few replicas, cut into rows of blocks that exchange their edges
through mailboxes: that such a batch is cut at all (as finely as the mailboxes
have room for), and replicas that join, end and leave between its launches.
Populations bit-identical to lattices stepped alone; sums within 2^-13
sqrt(S2_ii S2_jj), FP32 partials of at most 1024 products (2^-14) on either side."""
import numpy as np
import pytest

from paper_1204_6734_gb300 import flb, inputs

from tolerances import assert_sums_close

pytestmark = pytest.mark.gpu


def replica(Lx, Ly, r=0, basis="local"):
    return inputs.LatticeParams(Lx, Ly, 1.0, 0.1, 0.02, 1e-4, inputs.omega_groups(1.2, 0.9, 1.0), basis, "fp32",
                                seed=80 + r, replica=r)


def alone(p, n, warmup=0, every=1, fp32_products=True):
    with flb.Lattice(p, kernel="pipelined", pipeline_sampling=1 if fp32_products else None) as lat:
        lat.set_sampling(warmup, every)
        lat.step(n)
        return lat.populations(), lat.raw_sums()


def check(got, sums, p, n, every=1):
    f, (R1, R2, m) = alone(p, n, every=every)
    np.testing.assert_array_equal(got, f)
    assert sums[2] == m
    d = np.sqrt(np.diag(R2))
    assert np.all(np.abs(sums[1] - R2) <= 2.0 ** -13 * np.outer(d, d))
    assert np.all(np.abs(sums[0] - R1) <= 2.0 ** -13 * np.sqrt(m) * d)


@pytest.mark.parametrize("shapes", [[(256, 256)], [(300, 130)], [(400, 300)] * 2, [(64, 64)] * 8, [(1000, 9), (40, 700)],
                                    [(512, 300)]])
@pytest.mark.parametrize("tile", ["128x4", "mixed"])
def test_few_replicas_are_cut(shapes, tile):
    ps = [replica(Lx, Ly, r) for r, (Lx, Ly) in enumerate(shapes)]
    with flb.Batch(ps, tile=tile) as b:
        b.set_sampling(0, 2)
        for n in (9, 4):
            assert b.step(n).launches() == ({"cut"}, 1)
        for r, p in enumerate(ps):
            if tile == "128x4":
                check(b.populations(r), b.raw_sums(r), p, 13, 2)
            else:
                f, (R1, R2, m) = alone(p, 13, 0, 2, False)
                np.testing.assert_array_equal(b.populations(r), f)
                S1, S2, n = b.raw_sums(r)
                assert n == m
                assert_sums_close(S1, S2, R1, R2, n, 0.0, 0.0, 0.0)


def test_replicas_join_end_and_leave_a_cut_batch():
    """A and D end two steps and one step into a launch (a launch of two steps ends
    in the buffer that it began in), C joins and A leaves: every change lays the
    mailboxes out anew over the old words."""
    A, B, C, D = replica(64, 64, 0), replica(300, 100, 1), replica(21, 21, 2), replica(120, 90, 3)
    with flb.Batch.open("local", 4, 64 << 20) as b:
        def step(n):
            assert b.step(n).launches() == ({"cut"}, 1)
        ka, kb, kd = b.add(A, 11), b.add(B), b.add(D, 10)
        b.set_sampling(0, 1)
        step(9)
        step(6)
        assert [b.replica_time(k) for k in (ka, kb, kd)] == [11, 15, 10]
        check(b.populations(ka), b.raw_sums(ka), A, 11)
        check(b.populations(kd), b.raw_sums(kd), D, 10)
        kc = b.add(C)
        b.set_sampling(0, 1, slot=kc)
        step(5)
        b.remove(ka)
        step(7)
        b.step(2)
        assert b.launches() == ({"step"}, 2)
        ka = b.add(A, 8)
        b.set_sampling(0, 1, slot=ka)
        step(6)
        step(40)
        b.sync()
        check(b.populations(ka), b.raw_sums(ka), A, 8)
        check(b.populations(kb), b.raw_sums(kb), B, 75)
        check(b.populations(kc), b.raw_sums(kc), C, 60)
        check(b.populations(kd), b.raw_sums(kd), D, 10)
