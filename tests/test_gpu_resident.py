"""Many steps per launch with the populations in shared memory (the default on
lattices that fit the SMs) against one launch per step: the collision is the
same code on the same inputs, so populations are bit-identical; the sums are
formed from the same staged deviations, in FP32 partials of at most 1024
products cut differently, so each is within 2 x 2^-14 sqrt(S2_ii S2_jj) of the
other (the summation term of tests/tolerances.py, once per side)."""
import numpy as np
import pytest

from paper_1204_6734_gb300 import flb, inputs

pytestmark = pytest.mark.gpu


def params(Lx, Ly, basis="local", seed=5, ux0=0.1, uy0=-0.05, **kw):
    return inputs.LatticeParams(Lx, Ly, 1.0, ux0, uy0, 1e-4, inputs.omega_groups(1.1, 0.8, 1.0), basis, "fp32",
                                seed=seed, **kw)


def start_state(p):
    from paper_1204_6734_gb300.inputs import perturbation
    f0 = np.ones((9, p.Ly, p.Lx)) * np.array([4 / 9] + [1 / 9] * 4 + [1 / 36] * 4)[:, None, None]
    return f0 * (1 + 0.01 * perturbation(f0.shape, 7))


def run(p, cuts, kernel=None, warmup=2, every=2, f0=None):
    with flb.Lattice(p, kernel=kernel) as lat:
        lat.set_sampling(warmup, every)
        if f0 is not None:
            lat.set_populations(f0)
        for n in cuts:
            lat.step(n)
        f = lat.populations()
        return f, lat.raw_sums(), lat.conservation()


def close(a, b, n):
    (S1, S2, na), (R1, R2, nb) = a, b
    assert na == nb == n
    d = np.sqrt(np.diag(R2))
    assert np.all(np.abs(S2 - R2) <= 2 * 2.0 ** -14 * np.outer(d, d))
    assert np.all(np.abs(S1 - R1) <= 2 * 2.0 ** -14 * np.sqrt(n) * d)


# one node; single rows and columns; one block; cuts of one and of several rows;
# a cut across x; odd node counts (a pair's two nodes coincide in the middle)
SHAPES = [(1, 1), (1, 9), (9, 1), (2, 3), (21, 21), (32, 32), (64, 33), (33, 65), (300, 130), (257, 129), (4001, 20),
          (20, 601), (700, 300)]


@pytest.mark.parametrize("Lx,Ly", SHAPES)
@pytest.mark.parametrize("basis", ["standard", "local", "lut"])
def test_resident_equals_one_step_per_launch(Lx, Ly, basis):
    p = params(Lx, Ly, basis)
    f0 = start_state(p)
    got, sums, cons = run(p, [11], f0=f0)
    ref, rsums, rcons = run(p, [11], kernel="pipelined", f0=f0)
    np.testing.assert_array_equal(got, ref)
    np.testing.assert_allclose(cons, rcons, rtol=1e-12, atol=1e-9)
    close(sums, rsums, 5 * Lx * Ly)


@pytest.mark.parametrize("Lx,Ly", [(1, 1), (9, 1), (21, 21), (33, 65), (300, 130), (257, 129), (20, 601)])
@pytest.mark.parametrize("basis", ["standard", "local", "lut"])
def test_resident_fp16_store_equals_single_steps(Lx, Ly, basis):
    """The FP16 store: rounded to FP16 in every step, so bit-identical to calls of
    one step (which take the one-step kernel)."""
    p = params(Lx, Ly, basis)
    p.precision = "fp16dev"
    f0 = start_state(p)
    got, sums, _ = run(p, [11], f0=f0)
    ref, rsums, _ = run(p, [1] * 11, f0=f0)
    np.testing.assert_array_equal(got, ref)
    close(sums, rsums, 5 * Lx * Ly)


@pytest.mark.parametrize("Lx,Ly", [(21, 21), (64, 64), (300, 130)])
def test_launch_length_does_not_matter(Lx, Ly):
    p = params(Lx, Ly)
    f, (S1, S2, n), _ = run(p, [20], warmup=3, every=1)
    for cuts in ([3, 17], [5, 4, 6, 5], [1, 2, 16, 1]):
        g, (R1, R2, m), _ = run(p, cuts, warmup=3, every=1)
        np.testing.assert_array_equal(f, g)
        assert n == m
        if 1 not in cuts:   # calls of one or two steps take the one-step kernel, whose partials are cut differently
            np.testing.assert_allclose(S2, R2, rtol=1e-12, atol=1e-12 * n * p.kT)
            np.testing.assert_allclose(S1, R1, rtol=1e-12, atol=1e-12 * n * np.sqrt(p.kT))


@pytest.mark.parametrize("Lx,Ly", [(21, 21), (300, 130)])
def test_invalid_node_is_reported(Lx, Ly):
    p = params(Lx, Ly)
    f0 = start_state(p)
    x, y = Lx - 1, Ly // 2
    f0[:, y, x] = 0.0
    f0[1, y, x] = 1.0   # u = (1, 0): no basis
    where = []
    for kernel in (None, "pipelined"):
        with flb.Lattice(p, kernel=kernel) as lat:
            lat.set_populations(f0)
            lat.step(6)
            with pytest.raises(flb.FlbError) as e:
                lat.sync()
            assert e.value.code == flb.ERR_INVALID_VELOCITY
            where.append(flb.flb_error_location(lat.h)[1])
            with pytest.raises(flb.FlbError):
                lat.step(1)
    assert where[0] == where[1] == 0


@pytest.mark.parametrize("Lx,Ly,warmup,every,cuts", [
    (64, 32, 1, 4, [18]),               # several samples left by one launch
    (64, 32, 0, 3, [7, 50, 1, 42]),     # more than the buffers and the partial sums hold
    (256, 128, 2, 1, [40]),
    (32, 512, 5, 7, [3, 3, 30]),
    (21, 30, 1, 4, [18]),               # a side that is no power of two: one sample at a time
])
def test_structure_samples_of_long_launches(Lx, Ly, warmup, every, cuts):
    p = params(Lx, Ly)
    out = []
    for kernel in (None, "pipelined"):
        with flb.Lattice(p, kernel=kernel) as lat:
            lat.set_structure_sampling(warmup, every)
            for n in cuts:
                lat.step(n)
            out.append(lat.structure_factors() + (lat.populations(),))
    assert out[0][3] == out[1][3] == len(range(warmup, sum(cuts), every))
    for a, b in zip(out[0][:3] + out[0][4:], out[1][:3] + out[1][4:]):
        np.testing.assert_array_equal(a, b)


def test_captured_steps_take_the_one_step_kernel():
    import torch
    p = params(300, 130)
    s = torch.cuda.Stream()
    with flb.Lattice(p, stream=s) as lat:
        lat.step(5)
        torch.cuda.synchronize()
        g = torch.cuda.CUDAGraph()
        with torch.cuda.graph(g, stream=s):
            lat.step(6)
        with torch.cuda.stream(s):
            g.replay()
        f = lat.populations()
    ref, _, _ = run(p, [11], every=0)
    np.testing.assert_array_equal(f, ref)


def test_callers_workspace_keeps_its_size():
    import torch
    p = params(300, 130)
    n = flb.flb_workspace_bytes(p)
    ws = torch.empty(n, dtype=torch.uint8, device="cuda")
    with flb.Lattice(p, workspace=ws) as lat:
        lat.step(9)
        f = lat.populations()
    np.testing.assert_array_equal(f, run(p, [9], every=0)[0])
