"""Calls of very many steps: launches of about 10 ms each, so that other streams'
kernels are not kept waiting, with the results of shorter calls."""
import numpy as np
import pytest

from paper_1204_6734_gb300 import flb, inputs

pytestmark = pytest.mark.gpu


def params(Lx, Ly, seed=3):
    return inputs.LatticeParams(Lx, Ly, 1.0, 0.1, 0.02, 1e-4, inputs.omega_groups(1.2, 0.9, 1.0), "local", "fp32",
                                seed=seed)


@pytest.mark.parametrize("Lx,Ly,n", [(21, 21, 30011), (300, 130, 9001)])
def test_lattice(Lx, Ly, n):
    out = []
    for cuts in ([n], [n // 3, n - n // 3]):
        with flb.Lattice(params(Lx, Ly)) as lat:
            lat.set_sampling(0, 7)
            launches = [lat.step(m).launches() for m in cuts]
            assert all(k in ({"resident"}, {"cut"}) and c > 1 for k, c in launches)
            out.append((lat.populations(), lat.raw_sums()))
    np.testing.assert_array_equal(out[0][0], out[1][0])
    assert out[0][1][2] == out[1][1][2]
    np.testing.assert_allclose(out[0][1][1], out[1][1][1], rtol=1e-10, atol=1e-12 * out[0][1][2] * 1e-4)


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


def test_another_stream_gets_in():
    torch = pytest.importorskip("torch")
    s, t = torch.cuda.Stream(), torch.cuda.Stream()
    with flb.Lattice(params(900, 900), stream=s) as a, flb.Lattice(params(900, 900, 4), stream=t) as b:
        for lat in (a, b):
            lat.step(5)
            lat.sync()
        a.step(20000)          # a third of a second
        assert a.launches()[0] == {"cut"}
        end = torch.cuda.Event()
        end.record(s)
        b.step(5)
        b.sync()
        assert not end.query()
        a.sync()
