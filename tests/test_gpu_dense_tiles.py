"""Tiles of thousands of records, which the gridder splits over several CTAs, and dense
prediction tiles, which the degridder takes in runs: an array core on a small mesh, at
every tile side, next to the thresholds of the split.

Bars: planes are FP32 sums of n terms per cell in a fixed order, error growing like
sqrt(n) eps at worst n eps / 2: with 40 k records over a core of 400 cells and 64 taps,
6400 terms a cell, 2e-5 of the largest cell bounds it with room; predictions as in
tests/test_gpu_predict.py (1e-6 of the largest)."""
import numpy as np
import pytest

from tests.gpu_util import oracle_config, plan_config, rel_err, to_device
from visgen.workloads import tiny_wstack

pytestmark = pytest.mark.gpu


@pytest.fixture(scope="module")
def rk():
    import __graft_entry__
    __graft_entry__.build()
    import torch
    assert torch.cuda.is_available(), "GPU tests need a CUDA device"
    from paper_2601_19714_gb300 import rick
    rick.load()
    return rick


@pytest.mark.parametrize("tile,nvis", [(32, 8191), (32, 8193), (32, 40_000), (16, 40_000), (64, 70_000)])
@pytest.mark.parametrize("sparse", [False, True])
def test_split_tiles_match_oracle(rk, tile, nvis, sparse):
    import torch

    import oracle as orc
    orc.build()
    img, obs = tiny_wstack(nvis + tile, nvis=nvis, N=256, Nw=1)
    # most visibilities inside one tile (off its edges), a tenth over the whole disk
    obs.uvw[nvis // 10:, :2] *= 0.03
    obs.uvw[nvis // 10:, :2] += (8 if tile > 16 else 4) / img.fov
    dev = to_device(obs)
    with rk.Plan(plan_config(img, 1, tile=tile)) as plan:
        grids = torch.zeros((1, 1, 256, 256), dtype=torch.complex64, device="cuda")
        wsum = torch.empty(1, dtype=torch.float64, device="cuda")
        args = (dev["uvw"], dev["chan_scale"], dev["vis"], dev["weight"], None, dev["nrow"])
        plan.bin(*args, wsum)
        plan.grid_binned(0, 1, 0, 1, grids, sparse=sparse)
        g = grids.cpu().numpy()[0, 0]
        again = torch.zeros_like(grids)
        plan.grid_binned(0, 1, 0, 1, again, sparse=sparse)
        assert torch.equal(torch.view_as_real(again), torch.view_as_real(grids))   # a fixed order of additions
        plan.sync_status()
        G = orc.grid_plane(oracle_config(orc, img), obs.uvw, obs.chan_scale, obs.vis, obs.weight, None, plane=0)
        assert rel_err(g, G) <= 2e-5
        if not sparse and tile == 32:
            model = torch.zeros((1, 256, 256), dtype=torch.float32, device="cuda")
            r = np.random.default_rng(1)
            p, q = r.integers(100, 156, (2, 20))
            model[0, q, p] = torch.from_numpy(r.random(20).astype(np.float32)).cuda()
            vis = torch.empty((nvis, 1), dtype=torch.complex64, device="cuda")
            plan.predict(args[0], args[1], args[3], None, nvis, model, vis)
            at = r.integers(0, nvis, 50)
            want = orc.predict(oracle_config(orc, img), obs.uvw[at], obs.chan_scale, obs.weight[at], None,
                               image=model.cpu().numpy()[0].astype(np.float64))
            assert rel_err(vis.cpu().numpy()[at, 0], want) <= 1e-6
