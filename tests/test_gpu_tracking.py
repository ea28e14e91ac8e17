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
