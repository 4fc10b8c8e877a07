"""The batch tests on the kernel they were written for: one launch per step.

Small batches take many steps per launch of another kernel by default, so the
tile shapes, the graphs, the band edges and the runs of one replica are
stepped here with that kernel off, on the same inputs and with the same
tolerances, and every call is asked what it launched."""
import pytest

import test_gpu_batch as base
from paper_1204_6734_gb300 import flb, inputs

pytestmark = pytest.mark.gpu


@pytest.fixture(scope="module", autouse=True)
def _lib():
    torch = pytest.importorskip("torch")
    if not torch.cuda.is_available():
        pytest.skip("no CUDA device")
    flb.load()


@pytest.fixture
def seen(monkeypatch):
    """flb.Batch with one launch per step; the kinds of launches of each call."""
    kinds = []

    class OneStep(flb.Batch):
        def __init__(self, *args, **kw):
            super().__init__(*args, **{"kernel": "pipelined", **kw})

        def step(self, n):
            super().step(n)
            k, launches = self.launches()
            assert k <= {"step", "graph"} and launches == n
            kinds.append(k)
            return self

    monkeypatch.setattr(flb, "Batch", OneStep)
    yield kinds
    assert kinds and all(kinds)


@pytest.mark.parametrize("tile", base.TILES)
@pytest.mark.parametrize("basis", base.ALL_BASES)
def test_batch_equals_lattices_alone(basis, tile, seen):
    base.test_batch_equals_lattices_alone(basis, tile)


@pytest.mark.parametrize("basis", base.BASES)
def test_mixed_tiling_band_boundaries(basis, seen):
    base.test_mixed_tiling_band_boundaries(basis)


@pytest.mark.parametrize("tile", base.TILES)
@pytest.mark.parametrize("basis", base.BASES)
def test_batch_against_oracle_with_sampling(basis, tile, seen):
    base.test_batch_against_oracle_with_sampling(basis, tile)


@pytest.mark.parametrize("basis", base.ALL_BASES)
def test_batch_sampling_schedule_matches_lattice(basis, seen):
    base.test_batch_sampling_schedule_matches_lattice(basis)


@pytest.mark.parametrize("basis", base.BASES)
def test_graph_replay_equals_direct_launches(basis, seen):
    base.test_graph_replay_equals_direct_launches(basis)
    assert seen == [{"step"}, {"step"}, {"step", "graph"}, {"step", "graph"}]


@pytest.mark.parametrize("basis", base.BASES)
def test_membership_changes(basis, seen):
    base.test_membership_changes(basis)
    assert {"graph"} in seen


def test_invalid_replica_does_not_disturb_the_others(seen):
    base.test_invalid_replica_does_not_disturb_the_others()


@pytest.mark.parametrize("tile", ["64x12", "mixed"])
def test_many_runs_per_cta(tile, seen):
    base.test_many_runs_per_cta(tile)


def test_both_kernels_and_the_query():
    ps = base.uneven(inputs.LOCAL, n=4)
    with flb.Batch(ps) as b:
        b.step(5)
        assert b.launches() in (({"resident"}, 1), ({"cut"}, 1))
        b.step(2)
        assert b.launches() == ({"step"}, 2)
        b.set_kernel("pipelined")
        b.step(5)
        assert b.launches() == ({"step"}, 5)
        b.set_kernel("auto")
        b.step(0)
        assert b.launches() == ({"step"}, 5)
        b.step(3)
        assert b.launches() in (({"resident"}, 1), ({"cut"}, 1))
        with pytest.raises(flb.FlbError) as e:
            b.set_kernel("generic")
        assert e.value.code == flb.ERR_ARG
    with flb.Lattice(ps[0]) as lat:
        assert lat.step(7).launches() in (({"resident"}, 1), ({"cut"}, 1))
        assert lat.step(2).launches() == ({"step"}, 2)
