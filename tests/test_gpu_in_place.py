"""Steps in place (mixed-mode simulations of a capacity of 2^25 particles or more):
near the capacity, around a batch, after a start-up and under the adjoint.

Near the capacity: an in-place step keeps its holes and the next step's samples
follow behind its slots, so that they can reach past a capacity that holds the
particles, and the sorted layout, with room to spare.  Such a step packs its slots
first; no step fails that sorted steps would take."""
import numpy as np
import pytest

from paper_2007_13091_gb300 import workloads as wl

pytestmark = pytest.mark.gpu


def _buckets(count):
    return int((count + count // 32 + 4).sum())


@pytest.mark.parametrize("sampling,K", [("energy_matched", 0), ("maxwell", 2)])
def test_samples_past_the_slots(sampling, K):
    """82,944 cells of about 200 particles whose mass exceeds rho by what one and a
    half steps collide: hardly a cell samples in the first two steps, in the third
    nearly all of them fill up to N_min = 400.  The capacity lies half-way between
    what sorted steps and what slots left in place would need."""
    import torch
    from paper_2007_13091_gb300 import ugkwp
    cfg = wl.uniform_box(n=(24, 24, 24), Kn=7.1e-3, N_ref=200, precision="mixed", K=K)
    cfg["params"].update(sampling=sampling, N_min=400)
    nc = len(cfg["mesh"]["tets"])

    def sim(cap):
        p = dict(cfg["params"], particle_capacity=cap)
        return ugkwp.Simulation(cfg["mesh"], cfg["W0"], p, stream=torch.cuda.Stream())

    first = sim(1 << 26)
    first.step(1)
    wp = first.moments(ugkwp.WP)
    st = first.state_native()
    st["W"] = wl.conservative(0.85 * wp[0], np.zeros(3), 0.85 * wp[0], K)
    first.set_state_native(st)
    count = np.bincount(st["cell"], minlength=nc)
    need, wide, n_sam = [], [], []
    for _ in range(3):
        first.step(1)
        n = first.last("n_sam").astype(np.int64)
        n_sam.append(int(n.sum()))
        need.append(_buckets(count + n))  # the slots behind which sorted steps sample next
        count = first.last("surv_count").astype(np.int64)
    # the first step after an import sorts, the second would stay in place
    assert 8 * n_sam[1] <= count.sum() and n_sam[2] > 4 * (n_sam[1] + nc)
    sorted_need, in_place_need = need[1] + n_sam[2], need[0] + n_sam[1] + n_sam[2]
    cap = (sorted_need + in_place_need) // 2
    assert cap - sorted_need > nc and cap >= max(need) and cap >= 1 << 25
    assert need[0] + 5 * n_sam[1] + 4 * nc <= cap

    alone, member = sim(cap), sim(cap)
    batch = ugkwp.Batch([member])  # a batch's members sort in every step
    for s in (alone, member):
        s.set_state_native(st)
    del st
    for n in (1, 2):  # the step that packs is the second of a replayed pair
        alone.step(n)
        batch.step(n)
        batch.sync()
    alone.sync()
    for k in ("n_sam", "surv_count", "surv_mass", "pflux"):
        assert np.array_equal(alone.last(k), first.last(k)), k
        assert np.array_equal(member.last(k), first.last(k)), k
    for w in (ugkwp.W, ugkwp.WP):
        assert np.array_equal(alone.moments(w), first.moments(w))
    batch.close()
    a, b = alone.state_native(), first.state_native()
    oa, ob = np.argsort(a["id"]), np.argsort(b["id"])
    for k in ("id", "cell", "m", "e"):
        assert np.array_equal(a[k][oa], b[k][ob]), k
    for k in ("x", "u"):
        assert np.array_equal(a[k][:, oa], b[k][:, ob]), k


def test_members_step_in_place_again_after_their_batches():
    """A member sorts while it is in a batch, and steps in place as before once its
    last batch is freed: the particles of its image then lie out of cell order.
    Everything equals, bit for bit, a simulation that was in no batch."""
    import torch
    from paper_2007_13091_gb300 import ugkwp
    cfg = wl.cavity(n=6, Kn=0.3, N_ref=80, precision="mixed", order=2)
    cfg["params"]["particle_capacity"] = 1 << 25
    a, b = (ugkwp.Simulation(cfg["mesh"], cfg["W0"], cfg["params"], stream=torch.cuda.Stream()) for _ in range(2))

    def backward_steps():  # in cell order from slot to slot; only overflow slots when sorted
        x, y = a.state_native(), b.state_native()
        ox, oy = np.argsort(x["id"]), np.argsort(y["id"])
        for k in ("id", "cell", "m"):
            assert np.array_equal(x[k][ox], y[k][oy]), k
        for k in ("x", "u"):
            assert np.array_equal(x[k][:, ox], y[k][:, oy]), k
        assert np.array_equal(x["W"], y["W"])
        assert np.array_equal(a.moments(ugkwp.WP), b.moments(ugkwp.WP))
        return [int((np.diff(s["cell"]) < 0).sum()) for s in (x, y)]

    a.step(5)
    b.step(5)
    inplace = backward_steps()[1]
    assert inplace > 1000
    one = ugkwp.Batch([a])
    two = ugkwp.Batch([a])
    one.step(3)
    one.sync()
    one.close()
    a.step(2)  # alone, but still in the second batch
    a.sync()
    two.step(2)
    two.sync()
    b.step(7)
    assert backward_steps()[0] < 100
    two.close()
    for n in (1, 2, 2):
        a.step(n)
        b.step(n)
        got = backward_steps()
    assert got[0] > 1000
    never = ugkwp.Batch([a])  # created and freed between steps in place
    never.close()
    a.step(3)
    b.step(3)
    backward_steps()


@pytest.mark.parametrize("order", [1, 2])
def test_start_up_and_adjoint_in_place(order):
    """Steps in place after a gas-kinetic start-up, and the steps that an adjoint call
    records, equal sorted ones bit for bit, and so does what the call returns."""
    import torch
    from paper_2007_13091_gb300 import ugkwp
    cfg = wl.wall_channel(n=(9, 4, 5), Kn=0.2, N_ref=70, precision="mixed", order=order)
    sims = []
    for cap in (1 << 25, 1 << 19):
        p = dict(cfg["params"], particle_capacity=cap)
        sims.append(ugkwp.Simulation(cfg["mesh"], cfg["W0"], p, stream=torch.cuda.Stream()))
    unsorted = []
    for s in sims:
        s.gks_steps(4)
        s.step(3)
        s.out = [s.adjoint(f, 6, [1]) for f in (0, 1)]
        unsorted.append(int((np.diff(s.state_native()["cell"]) < 0).sum()))
        s.step(2)
    a, b = sims
    assert unsorted[0] > unsorted[1] + 1000
    for x, y in zip(a.out, b.out):
        assert np.array_equal(x, y) and np.all(np.isfinite(x)) and x[0] != 0.0
    for w in (ugkwp.W, ugkwp.WP):
        assert np.array_equal(a.moments(w), b.moments(w))
    for k in ("n_sam", "surv_count", "surv_mass", "pflux"):
        assert np.array_equal(a.last(k), b.last(k)), k
