"""The sums of a run do not depend on how its steps are cut into calls: every sampled
step of a lattice takes the same kernel in calls of any length, its FP32 partials go
to FP64 step by step, and only the order of the FP64 additions differs (1e-12)."""
import numpy as np
import pytest

from paper_1204_6734_gb300 import flb, inputs

pytestmark = pytest.mark.gpu


def params(Lx, Ly, precision="fp32", basis="local"):
    return inputs.LatticeParams(Lx, Ly, 1.0, 0.1, -0.05, 1e-4, inputs.omega_groups(1.1, 0.8, 1.0), basis, precision,
                                seed=5)


def run(p, cuts, warmup, every):
    with flb.Lattice(p) as lat:
        lat.set_sampling(warmup, every)
        for n in cuts:
            lat.step(n)
        return lat.populations(), lat.raw_sums()


@pytest.mark.parametrize("Lx,Ly", [(1, 1), (21, 21), (64, 64), (300, 130), (900, 900), (1100, 1000)])
@pytest.mark.parametrize("precision", ["fp32", "fp16dev"])
@pytest.mark.parametrize("warmup,every", [(0, 1), (3, 2), (5, 1)])
def test_cuts(Lx, Ly, precision, warmup, every):
    p = params(Lx, Ly, precision)
    f, (S1, S2, n) = run(p, [20], warmup, every)
    for cuts in ([1] * 20, [2] * 10, [1, 2, 16, 1], [4, 1, 1, 14]):
        g, (R1, R2, m) = run(p, cuts, warmup, every)
        np.testing.assert_array_equal(f, g)
        assert n == m
        np.testing.assert_allclose(S2, R2, rtol=1e-12, atol=1e-12 * n * p.kT)
        np.testing.assert_allclose(S1, R1, rtol=1e-12, atol=1e-12 * n * np.sqrt(p.kT))


def test_resumed_with_calls_of_one_step():
    p = params(64, 64)
    with flb.Lattice(p) as lat:
        lat.set_sampling(2, 1)
        lat.step(9)
        state = lat.checkpoint()
        lat.step(30)
        f, (S1, S2, n) = lat.populations(), lat.raw_sums()
    with flb.Lattice(p) as lat:
        lat.resume(state, 2, 1)
        for _ in range(30):
            lat.step(1)
        np.testing.assert_array_equal(f, lat.populations())
        R1, R2, m = lat.raw_sums()
    assert n == m
    np.testing.assert_allclose(S2, R2, rtol=1e-12, atol=1e-12 * n * p.kT)
    np.testing.assert_allclose(S1, R1, rtol=1e-12, atol=1e-12 * n * np.sqrt(p.kT))


@pytest.mark.parametrize("Lx,Ly", [(21, 21), (33, 65), (300, 130), (20, 601)])
@pytest.mark.parametrize("basis", ["standard", "local", "lut"])
def test_fp16_store_in_both_kernels(Lx, Ly, basis):
    """Captured steps take the one-step kernel: bit-identical states, and sums within the
    rounding of FP32 partials of at most 1024 products, 2^-14 sqrt(S2_ii S2_jj) a side."""
    torch = pytest.importorskip("torch")
    p = params(Lx, Ly, "fp16dev", basis)
    with flb.Lattice(p) as lat:
        lat.set_sampling(0, 1)
        k, _ = lat.step(11).launches()
        assert k in ({"resident"}, {"cut"})
        f, (S1, S2, n) = lat.populations(), lat.raw_sums()
    s = torch.cuda.Stream()
    with flb.Lattice(p, stream=s) as lat:
        lat.set_sampling(0, 1)
        g = torch.cuda.CUDAGraph()
        torch.cuda.synchronize()
        with torch.cuda.graph(g, stream=s):
            assert lat.step(11).launches() == ({"step"}, 11)
        with torch.cuda.stream(s):
            g.replay()
        np.testing.assert_array_equal(lat.populations(), f)
        R1, R2, m = lat.raw_sums()
    assert n == m
    d = np.sqrt(np.diag(R2))
    assert np.all(np.abs(S2 - R2) <= 2.0 ** -13 * np.outer(d, d))
    assert np.all(np.abs(S1 - R1) <= 2.0 ** -13 * np.sqrt(n) * d)
