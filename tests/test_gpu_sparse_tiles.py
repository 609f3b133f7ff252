"""Sparse gridding of launches whose tile count is no multiple of a warp: a 256^2 mesh
with tiles of 64 has 16 tiles a plane.  Only the launch's own tiles may be listed:
the planes after its range keep what they held, and the image equals that of the
dense calls (bar as in tests/test_gpu_columns.py: two FP32 transforms of the same
planes, 6e-6 of the peak)."""
import pytest

from tests.gpu_util import oracle_config, plan_config, rel_err, taper_gain, to_device
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


def _two_channels(obs):
    import numpy as np
    obs.chan_scale = np.ones(2)
    obs.vis = np.repeat(np.asarray(obs.vis).reshape(-1, 1), 2, 1)
    obs.weight = np.repeat(np.asarray(obs.weight).reshape(-1, 1), 2, 1)
    return obs


@pytest.mark.parametrize("Nw,k0,k1", [(1, 0, 1), (3, 0, 3), (3, 1, 2)])
def test_launch_lists_only_its_own_tiles(rk, Nw, k0, k1):
    import torch

    import oracle as orc
    orc.build()
    img, obs = tiny_wstack(70 + Nw + k0, nvis=2000, N=256, Nw=Nw)
    obs = _two_channels(obs)
    dev = to_device(obs)
    guard = 2
    with rk.Plan(plan_config(img, 2, tile=64)) as plan:
        grids = torch.full((k1 - k0 + guard, 256, 256), 7.0 + 7.0j, dtype=torch.complex64, device="cuda")
        grids[:k1 - k0] = 0   # unreached tiles are not written
        wsum = torch.empty(2, dtype=torch.float64, device="cuda")
        plan.bin(dev["uvw"], dev["chan_scale"], dev["vis"], dev["weight"], None, dev["nrow"], wsum)
        plan.grid_binned(0, 1, k0, k1, grids[:k1 - k0], sparse=True)
        plan.sync_status()
        assert bool((grids[k1 - k0:] == 7.0 + 7.0j).all())
        for k in range(k0, k1):
            G = orc.grid_plane(oracle_config(orc, img), obs.uvw, obs.chan_scale[:1], obs.vis[:, :1], obs.weight[:, :1],
                               None, plane=k)
            # FP32 sums of some tens of terms a cell
            assert rel_err(grids[k - k0].cpu().numpy(), G) <= 1e-5


@pytest.mark.parametrize("Nw", [1, 3])
def test_image_of_odd_plane_count_equals_dense_calls(rk, Nw):
    import torch
    img, obs = tiny_wstack(80 + Nw, nvis=2000, N=256, Nw=Nw)
    dev = to_device(obs)
    args = (dev["uvw"], dev["chan_scale"], dev["vis"], dev["weight"], None, dev["nrow"])
    with rk.Plan(plan_config(img, 1, tile=64)) as plan:
        got, ref = (torch.zeros((1, 256, 256), dtype=torch.float32, device="cuda") for _ in range(2))
        plan.dirty_image(*args, got)
        grids = torch.empty((1, Nw, 256, 256), dtype=torch.complex64, device="cuda")
        wsum = torch.empty(1, dtype=torch.float64, device="cuda")
        plan.grid(*args, 0, Nw, grids, wsum)
        plan.fft_wplanes(grids, Nw)
        plan.phase_correct_reduce(grids, 0, 1, 0, Nw, wsum, ref)
        A = torch.from_numpy(taper_gain(plan.taper())).cuda()
        assert float(((got - ref).abs() * A).max() / (ref.abs() * A).max()) <= 6e-6
        plan.sync_status()
