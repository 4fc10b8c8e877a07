"""flb_batch_step on a stream that the caller captures: one launch per step goes
into the graph, whatever the call would launch otherwise, and nothing that the
call prepared counts as done until the graph has run -- steps taken directly
between the capture and the graph's launch see the same members."""
import numpy as np
import pytest

from paper_1204_6734_gb300 import flb, inputs

pytestmark = pytest.mark.gpu


def replica(Lx, Ly, r):
    return inputs.LatticeParams(Lx, Ly, 1.0, 0.1, 0.02, 1e-4, inputs.omega_groups(1.2, 0.9, 1.0), "local", "fp32",
                                seed=60 + r, replica=r)


@pytest.mark.parametrize("shapes", [[(21, 21)] * 300, [(64, 64)] * 8, [(700, 600), (900, 500)]])
@pytest.mark.parametrize("before", [0, 2, 4])
def test_steps_between_capture_and_launch(shapes, before):
    torch = pytest.importorskip("torch")
    ps = [replica(Lx, Ly, r) for r, (Lx, Ly) in enumerate(shapes)]
    s = torch.cuda.Stream()
    with flb.Batch(ps, stream=s) as b:
        b.set_sampling(0, 1)
        b.step(before)
        b.sync()
        g = torch.cuda.CUDAGraph()
        with torch.cuda.graph(g, stream=s):
            b.step(5)
            assert b.launches() == ({"step"}, 5)
        b.step(4)
        with torch.cuda.stream(s):
            g.replay()
        b.sync()
        assert b.t == before + 9
        for r in (0, len(ps) - 1):
            with flb.Lattice(ps[r], kernel="pipelined") as lat:
                lat.set_sampling(0, 1)
                lat.step(before + 9)
                np.testing.assert_array_equal(b.populations(r), lat.populations())
                assert b.raw_sums(r)[2] == lat.raw_sums()[2]
