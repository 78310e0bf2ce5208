"""Failure detection without a GPU fault.

* Allocation failures: a plan whose allocation hook (hfx_options alloc /
  free) refuses memory reports HFX_ERR_OOM, gives back everything it took,
  and a plan whose per-call store cannot grow stays usable once memory is
  available again.
* Bounded waits: the tensor-core pipelines wait on mbarriers with a limit of
  one second of wall time.  The test-only switch
  HFX_TEST_STALL_Q2_PRODUCER=1 keeps the second product's producer warp from
  issuing its copies, so the consumers' waits run out; the call must return
  HFX_ERR_TIMEOUT (no trap, no hang) and the same plan must evaluate
  correctly afterwards.
"""
import numpy as np
import pytest

from paper_2412_11081_gb300 import hfx, inputs

pytestmark = pytest.mark.gpu


def rel(a, ref):
    a, ref = np.asarray(a, float), np.asarray(ref, float)
    return float(np.max(np.abs(a - ref)) / np.max(np.abs(ref)))


class CountingAllocator:
    """Device memory from PyTorch's caching allocator, with a budget of
    allocations after which it refuses (returns 0)."""

    def __init__(self, budget=10 ** 9):
        import torch
        self.torch = torch
        self.budget = budget
        self.live = {}
        self.allocs = 0
        self.frees = 0

    def alloc(self, n):
        if self.allocs >= self.budget:
            return 0
        self.allocs += 1
        p = self.torch.cuda.caching_allocator_alloc(n, 0, self.torch.cuda.current_stream())
        self.live[int(p)] = n
        return int(p)

    def free(self, p, n):
        self.frees += 1
        assert self.live.pop(p) == n
        self.torch.cuda.caching_allocator_delete(p)

    def hooks(self):
        return (self.alloc, self.free)


def test_plan_creation_out_of_memory_gives_back_what_it_took():
    pytest.importorskip("torch")
    w = inputs.diamond8()
    for budget in (0, 5, 30):
        a = CountingAllocator(budget)
        with pytest.raises(hfx.HfxError) as ei:
            hfx.Plan(w, allocator=a.hooks())
        assert ei.value.status == 2, (budget, ei.value)
        assert not a.live and a.frees == a.allocs, budget


def test_evaluation_out_of_memory_leaves_the_plan_usable():
    pytest.importorskip("torch")
    w = inputs.diamond8()
    a = CountingAllocator()
    with hfx.Plan(w, allocator=a.hooks()) as p:
        a.budget = a.allocs          # the per-call stores cannot grow any more
        with pytest.raises(hfx.HfxError) as ei:
            p.evaluate(w.lattice, w.positions)
        assert ei.value.status == 2
        a.budget = 10 ** 9
        E, F, S = p.evaluate(w.lattice, w.positions)
    with hfx.Plan(w) as q:
        ref = q.evaluate(w.lattice, w.positions)
    assert abs(E - ref[0]) <= 1e-12 * abs(ref[0]) and rel(F, ref[1]) <= 1e-12
    assert not a.live


@pytest.mark.parametrize("prec", [hfx.HFX_BF16X3, hfx.HFX_BF16X6])
def test_stalled_pipeline_wait_runs_out_and_plan_recovers(prec, monkeypatch):
    w = inputs.diamond8()
    with hfx.Plan(w, precision=prec) as p:
        ref = p.evaluate(w.lattice, w.positions)
        monkeypatch.setenv("HFX_TEST_STALL_Q2_PRODUCER", "1")
        with pytest.raises(hfx.HfxError) as ei:
            p.evaluate(w.lattice, w.positions)
        assert ei.value.status == 4, ei.value
        monkeypatch.delenv("HFX_TEST_STALL_Q2_PRODUCER")
        E, F, S = p.evaluate(w.lattice, w.positions)
    assert abs(E - ref[0]) <= 1e-12 * abs(ref[0]) and rel(F, ref[1]) <= 1e-12 and rel(S, ref[2]) <= 1e-12


@pytest.mark.parametrize("tiles", ["1", "2", "3"])
def test_stalled_pipeline_in_every_q2_shape(tiles, monkeypatch):
    """The producer warp stays out of the epilogue and nothing is read from an
    accumulator that was not handed over, whichever way the row tiles are
    divided over the warps; diamond8's and a 13-orbital cell's tiles (one and
    several of 128 rows)."""
    monkeypatch.setenv("HFX_Q2_TILES", tiles)
    for w in (inputs.diamond8(), inputs.tiny_model([13], [50], [0], np.eye(3) * 3.4, [[0.1, 0.2, 0.0]], r_c=1.4, seed=3)):
        with hfx.Plan(w, precision=hfx.HFX_BF16X6) as p:
            ref = p.evaluate(w.lattice, w.positions)
            monkeypatch.setenv("HFX_TEST_STALL_Q2_PRODUCER", "1")
            with pytest.raises(hfx.HfxError) as ei:
                p.evaluate(w.lattice, w.positions)
            assert ei.value.status == 4, ei.value
            monkeypatch.delenv("HFX_TEST_STALL_Q2_PRODUCER")
            E, F, S = p.evaluate(w.lattice, w.positions)
        assert abs(E - ref[0]) <= 1e-12 * abs(ref[0]) and rel(S, ref[2]) <= 1e-12


def test_wide_plan_without_room_for_two_y_stores():
    """n_ao > 16: the tensor-memory kernels keep two Y stores, the warp-level
    ones one.  Whichever store of the first evaluation cannot be had, the plan
    goes on with one Y store and gives the same result; one that gets no more
    memory at all says so and works again afterwards."""
    pytest.importorskip("torch")
    rng = np.random.default_rng(5)
    pos = np.array([[0.1, 0.2, 0.0], [1.6, 1.5, 1.7]]) + rng.normal(0, 0.05, (2, 3))
    w = inputs.cut_density(inputs.tiny_model([18, 7], [23, 11], [0, 1], np.eye(3) * 3.3, pos, r_c=1.4, seed=5), 4.0)

    class Refusing(CountingAllocator):
        refuse = ()

        def alloc(self, n):
            self.allocs += 1
            if self.allocs in self.refuse:
                self.refused = getattr(self, "refused", 0) + 1
                return 0
            p = self.torch.cuda.caching_allocator_alloc(n, 0, self.torch.cuda.current_stream())
            self.live[int(p)] = n
            return int(p)

    a = Refusing()
    with hfx.Plan(w, precision=hfx.HFX_BF16X6, allocator=a.hooks()) as p:
        made = a.allocs
        two = p.evaluate(w.lattice, w.positions, stats=True)
        launches, stores = p.stats.kernel_launches, a.allocs - made
    assert not a.live and stores >= 6
    for k in range(1, stores + 1):
        a = Refusing()
        with hfx.Plan(w, precision=hfx.HFX_BF16X6, allocator=a.hooks()) as p:
            a.refuse = (a.allocs + k,)
            E, F, S = p.evaluate(w.lattice, w.positions, stats=True)
            assert a.refused == 1 and p.stats.kernel_launches != launches, k   # (the other kernels ran)
            assert abs(E - two[0]) <= 1e-5 * abs(two[0]) and rel(F, two[1]) <= 1e-5 and rel(S, two[2]) <= 1e-5
            assert rel(p.evaluate(w.lattice, w.positions)[1], F) <= 1e-12
        assert not a.live
    a = Refusing()
    with hfx.Plan(w, precision=hfx.HFX_BF16X6, allocator=a.hooks()) as p:
        a.refuse = range(a.allocs + 2, 10 ** 9)
        with pytest.raises(hfx.HfxError) as ei:
            p.evaluate(w.lattice, w.positions)
        assert ei.value.status == 2
        a.refuse = ()
        E, F, S = p.evaluate(w.lattice, w.positions)
        assert rel(F, two[1]) <= 1e-5
    assert not a.live


@pytest.mark.parametrize("prec", [hfx.HFX_FP64, hfx.HFX_BF16X6])
def test_list_rebuild_out_of_memory_leaves_the_plan_usable(prec):
    """Memory that runs out while stale pair lists are made again: the old ones
    are gone by then, so the next call makes them, at whatever geometry."""
    pytest.importorskip("torch")
    w = inputs.diamond8()
    far = w.positions + np.random.default_rng(2).normal(0, 0.3, w.positions.shape)
    a = CountingAllocator()
    with hfx.Plan(w, precision=prec, allocator=a.hooks()) as p:
        ref = p.evaluate(w.lattice, w.positions)
        for more in (0, 7, 20):
            a.budget = a.allocs + more
            with pytest.raises(hfx.HfxError) as ei:
                p.evaluate(w.lattice, far)
            assert ei.value.status == 2
            a.budget = 10 ** 9
            E, F, S = p.evaluate(w.lattice, w.positions)
            assert abs(E - ref[0]) <= 1e-12 * abs(ref[0]) and rel(F, ref[1]) <= 1e-12
    assert not a.live
