"""The wave flux's faces in tiles: a grid that does not cover them takes the tiles
from a counter (one simulation at first order; a fused batch, whose blocks also
take the other members' tiles).  Which warp computes a face changes nothing: the
states equal those of a grid that covers every face, bit for bit.
"""
import pytest

from paper_2007_13091_gb300 import ugkwp, workloads as wl
from tests.test_gpu_batch import _assert_same, _sim

pytestmark = pytest.mark.gpu


def _cfg(n, order, seed, precision="mixed"):
    c = wl.cavity(n=n, N_ref=60, Kn=0.05, precision=precision, order=order, seed=seed)
    c["params"]["sampling"] = "energy_matched"
    return c


@pytest.mark.parametrize("blocks", [1, 3, 5])
@pytest.mark.parametrize("order", [1, 2])
def test_few_wave_blocks(order, blocks):
    """1,296 tets: 2,376 interior and 432 boundary faces (87.75 tiles of 32)."""
    import torch
    cfg = _cfg(6, order, 7)
    a, c = _sim(cfg, torch.cuda.Stream()), _sim(cfg, torch.cuda.Stream())
    d = ugkwp.ugkwp_get_launch_cfg(a.handle)
    ugkwp.ugkwp_set_launch_cfg(a.handle, d["particle_blocks"], blocks, d["track_threads"], d["smem_carveout"])
    a.step(3)
    c.step(3)
    _assert_same(a, c)


@pytest.mark.parametrize("order", [1, 2])
def test_batch_members_share_the_blocks(order):
    """Four members of uneven size on six flux blocks: the small ones' blocks
    cover their faces, the others' do not."""
    import torch
    cfgs = [_cfg(n, order, 20 + n) for n in (2, 7, 3, 9)]
    batched = [_sim(c, torch.cuda.Stream()) for c in cfgs]
    alone = [_sim(c, torch.cuda.Stream()) for c in cfgs]
    for s in batched:
        d = ugkwp.ugkwp_get_launch_cfg(s.handle)
        ugkwp.ugkwp_set_launch_cfg(s.handle, d["particle_blocks"], 6, d["track_threads"], d["smem_carveout"])
    b = ugkwp.Batch(batched)
    b.step(3)
    b.sync()
    for x, y in zip(batched, alone):
        y.step(3)
        _assert_same(x, y)
    b.close()


def test_wave_blocks_hold_in_start_up_steps():
    """Second-order start-up steps take the grid the caller chose: four blocks, on
    four of the chip's SMs, take far longer (some 38 times, bound by the binary64
    pipe; at least 5 is asked) than the default, with the same bits."""
    import torch
    cfg = _cfg(24, 2, 5)
    few, default = _sim(cfg, torch.cuda.Stream()), _sim(cfg, torch.cuda.Stream())
    d = ugkwp.ugkwp_get_launch_cfg(few.handle)
    ugkwp.ugkwp_set_launch_cfg(few.handle, d["particle_blocks"], 4, d["track_threads"], d["smem_carveout"])
    ms = []
    for s in (few, default):
        s.gks_steps(3)
        ugkwp.ugkwp_timing_enable(s.handle, True)
        s.gks_steps(5)
        ms.append(ugkwp.ugkwp_timing_read(s.handle)[0]["flux_o2"])
    _assert_same(few, default)
    assert ms[0] > 5 * ms[1]
