"""The gridder's paths by kernel support (1 to 3 and 9 to 16 general, 4, 5 to 8)
and tile side, with footprints on every tile edge, against the oracle's planes.

Bar: FP32 sums of a few hundred terms per cell, the parity bar of gridded planes
(1e-6 of the plane's largest cell)."""
import numpy as np
import pytest

from tests.gpu_util import oracle_config, plan_config, rel_err, to_device
from visgen.workloads import GAUSS_SIGMA_S7, tiny_wstack

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


@pytest.mark.parametrize("S", [1, 2, 3, 4, 5, 6, 7, 8, 9, 13, 16])
@pytest.mark.parametrize("tile", [16, 32, 64])
def test_planes_match_oracle_at_every_support(rk, S, tile):
    import torch

    import oracle as orc
    orc.build()
    img, obs = tiny_wstack(S * 100 + tile, nvis=4003, N=256, Nw=2)
    img = img.with_(S=S, kernel="gauss", kernel_param=max(GAUSS_SIGMA_S7 * S / 7.0, 0.5))
    dev = to_device(obs)
    with rk.Plan(plan_config(img, 1, tile=tile)) as plan:
        grids = torch.full((1, 2, 256, 256), float("nan"), dtype=torch.complex64, device="cuda")
        wsum = torch.empty(1, dtype=torch.float64, device="cuda")
        plan.grid(dev["uvw"], dev["chan_scale"], dev["vis"], dev["weight"], None, dev["nrow"], 0, 2, grids, wsum)
        g = grids.cpu().numpy()[0]
    cfg = oracle_config(orc, img)
    for k in range(2):
        G = orc.grid_plane(cfg, obs.uvw, obs.chan_scale, obs.vis, obs.weight, None, plane=k)
        assert rel_err(g[k], G) <= 1e-6, (S, tile, k)
