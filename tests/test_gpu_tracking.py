"""The tracking's shortcuts against the oracle, which walks every particle: the
inside test in binary32 with a margin, the collision threshold, and the exit
faces decided in binary32 for binary64 particles.  Meshes far from the origin
make the margins as large as the cells (everything is walked exactly), the
Knudsen numbers go from gas that nearly all collides to gas that hardly does."""
import numpy as np
import pytest

from paper_2007_13091_gb300 import workloads as wl
from tests.test_gpu_parity import run_teacher_forced

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("precision", ["fp64", "mixed"])
@pytest.mark.parametrize("offset,Kn", [(0.0, 2e-3), (0.0, 1.0), (30.0, 0.02), (1000.0, 0.1)])
def test_shortcuts_teacher_forced(precision, offset, Kn):
    cfg = wl.uniform_box(n=(3, 4, 5), U=(0.3, -0.2, 0.9), Kn=Kn, N_ref=60, precision=precision, bc_type="wall",
                         jitter_amount=0.15)
    cfg["mesh"] = dict(cfg["mesh"], nodes=cfg["mesh"]["nodes"] + offset * np.array([1.0, -0.7, 0.4]))
    cfg["params"]["sampling"] = "energy_matched"
    gsim, osim = run_teacher_forced(cfg, warm_steps=3, launch=(11, 3, 128, -1))
    c = osim.last("counters")
    assert c["n_crossings"] > 0 and c["n_wall_hits"] > 0
    st = gsim.step(1, stats=True)
    osim.step()
    d = osim.last("counters")
    assert st["n_crossings"] == d["n_crossings"] and st["n_wall_hits"] == d["n_wall_hits"]
    assert st["n_collided"] == d["n_collided"]


@pytest.mark.parametrize("precision,K,n", [("fp64", 0, 5), ("fp64", 2, 4), ("mixed", 0, 7), ("mixed", 5, 4)])
def test_particle_moments_after_steps(precision, K, n):
    """W^p of a stepped case (buckets with holes, an odd number of slots) against
    the sums over the exported particles.  Each particle's value is rounded to a
    quantum of 2^-50 of the largest cell's (about 1e-15 of a cell's W^p), summed
    over some hundred particles: 1e-12 relative, 1e-12 absolute."""
    from paper_2007_13091_gb300 import ugkwp
    cfg = wl.cavity(n=n, N_ref=60, precision=precision, K=K)
    s = ugkwp.Simulation(cfg["mesh"], cfg["W0"], cfg["params"])
    s.step(4)
    st = s.state()
    nodes, tets = cfg["mesh"]["nodes"], cfg["mesh"]["tets"]
    vol = np.abs(wl._volumes(nodes, tets))
    e2 = (st["u"] ** 2).sum(0) + (st["e"] if K else 0.0)
    phi = np.stack([st["m"], *(st["m"] * st["u"]), 0.5 * st["m"] * e2])
    WP = np.stack([np.bincount(st["cell"], p, len(tets)) for p in phi]) / vol
    np.testing.assert_allclose(s.moments(ugkwp.WP), WP, rtol=1e-12, atol=1e-12)
    np.testing.assert_allclose(s.moments(ugkwp.WH), st["W"] - WP, rtol=1e-11, atol=1e-11)


def _by_id(st):
    o = np.argsort(st["id"])
    return [st["id"][o], st["cell"][o], st["m"][o], st["x"][:, o], st["u"][:, o], st["e"][o]]


@pytest.mark.parametrize("flow,sampling,K", [("cavity", "maxwell", 0), ("cavity", "maxwell", 2),
                                             ("channel", "energy_matched", 0), ("cavity", "gp1", 0)])
def test_in_place_steps_equal_sorted_steps(flow, sampling, K):
    """A mixed-mode simulation of a capacity from 2^25 on leaves its particles in
    their slots in most steps; a smaller one sorts them in every step.  Both give
    the same bits: fields, particles, counts, W^p, through single and replayed
    steps, an import half-way and a batch."""
    import torch
    from paper_2007_13091_gb300 import ugkwp
    if flow == "cavity":
        cfg = wl.cavity(n=6, Kn=0.3, N_ref=80, precision="mixed", order=2, K=K)
    else:
        cfg = wl.wall_channel(n=(9, 4, 5), Kn=0.2, N_ref=70, precision="mixed")
    cfg["params"]["sampling"] = sampling
    sims = []
    for cap in (1 << 25, 1 << 19):
        p = dict(cfg["params"], particle_capacity=cap)
        sims.append(ugkwp.Simulation(cfg["mesh"], cfg["W0"], p, stream=torch.cuda.Stream()))
    big, small = sims
    unsorted = 0

    def same():
        a, b = big.state_native(), small.state_native()
        for x, y in zip(_by_id(a), _by_id(b)):
            assert np.array_equal(x, y)
        assert np.array_equal(a["W"], b["W"]) and a["t"] == b["t"]
        for k in ("n_sam", "surv_count", "surv_mass", "pflux"):
            assert np.array_equal(big.last(k), small.last(k)), k
        assert np.array_equal(big.moments(ugkwp.WP), small.moments(ugkwp.WP))
        return int((np.diff(a["cell"]) < 0).sum()) - int((np.diff(b["cell"]) < 0).sum())

    for n in (1, 1, 2, 3, 4, 1, 6):
        sa, sb = big.step(n, stats=True), small.step(n, stats=True)
        assert {k: v for k, v in sa.items()} == {k: v for k, v in sb.items()}
        unsorted = max(unsorted, same())
    assert unsorted > 100  # steps in place did happen
    st = big.state()
    big.set_state(st)
    small.set_state(st)
    for s in sims:
        s.step(5)
    same()
    batch = ugkwp.Batch(sims)
    batch.step(5)
    batch.sync()
    batch.close()
    same()


def test_largest_tracking_grid():
    """2^20 blocks of 256 threads, the largest grid that is accepted, on some 2.6e6
    particles: its 2^23 warps reserve two runs of 320 slots each, past 2^32 slots,
    and every particle is tracked once all the same (fields and counts equal those
    of the default grid, bit for bit)."""
    import torch
    from paper_2007_13091_gb300 import ugkwp
    cfg = wl.cavity(n=14, Kn=0.5, N_ref=160, precision="mixed", order=1)
    a, b = (ugkwp.Simulation(cfg["mesh"], cfg["W0"], cfg["params"], stream=torch.cuda.Stream()) for _ in range(2))
    ugkwp.ugkwp_set_launch_cfg(a.handle, 1 << 20, 4, 256)
    for k in range(3):
        sa, sb = a.step(1, stats=True), b.step(1, stats=True)
        assert sa == sb
        assert k > 0 or sa["n_tracked"] >= 10 * (32 * 8192)  # runs of ten tiles
    assert 2 * (1 << 20) * 8 * 320 > 1 << 32
    assert np.array_equal(a.moments(ugkwp.WP), b.moments(ugkwp.WP))
    assert np.array_equal(a.state_native()["W"], b.state_native()["W"])
    for k in ("pflux", "surv_count", "surv_mass"):
        assert np.array_equal(a.last(k), b.last(k)), k


@pytest.mark.parametrize("precision", ["fp64", "mixed"])
def test_past_the_capacity_no_particle_is_left(precision):
    """A step that does not fit the capacity writes no particle; none of the slots
    it left unwritten is read afterwards: the simulation has no particles until a
    step fits, and says so in the image, in W^p and in the sums per cell."""
    from paper_2007_13091_gb300 import ugkwp
    cfg = wl.shock_tube(nx=20, ny=2, nz=2, precision=precision)
    cfg["params"]["particle_capacity"] = 1000  # far below the 480 x 50 sampled particles
    s = ugkwp.Simulation(cfg["mesh"], cfg["W0"], cfg["params"])
    for n in (1, 2, 1):
        s.step(n)
        with pytest.raises(ugkwp.UgkwpError) as e:
            s.moments(ugkwp.WP)
        assert e.value.code == ugkwp.E_CAPACITY
        assert not s.moments(ugkwp.WP).any()
        assert s.state()["id"].size == 0 and s.state_native()["id"].size == 0
        assert not s.last("surv_count").any() and not s.last("surv_mass").any()
