"""The column pass on the plan's own grid memory (pruned to the reached tiles,
rows outside the image left out) and the cropped row pass, against the
separate calls on whole planes (rick_grid, rick_fft_wplanes,
rick_phase_correct_reduce; rick_model_to_wplanes, rick_fft_wplanes_forward,
rick_degrid_binned), at every transform length and tile side and with padding.

Bar: both sides are FP32 transforms of the same gridded planes, each within
3e-6 of the RMS of FP64 (tests/test_gpu_fft.py), so the taper-weighted images
and the predictions differ by at most 6e-6 of their peak."""
import numpy as np
import pytest

from tests.gpu_util import plan_config, taper_gain, to_device
from visgen.workloads import tiny_wstack

pytestmark = pytest.mark.gpu
TOL = 6e-6


@pytest.fixture(scope="module")
def rk():
    import __graft_entry__
    __graft_entry__.build()
    import torch
    assert torch.cuda.is_available(), "GPU tests need a CUDA device"
    from paper_2601_19714_gb300 import rick
    rick.load()
    return rick


CASES = [(256, 256, 16, True), (256, 512, 32, False), (512, 512, 64, False), (256, 1024, 32, True),
         (1024, 1024, 16, False), (1024, 2048, 16, True), (2048, 2048, 64, False), (2048, 4096, 32, True),
         (4096, 4096, 16, False), (512, 4096, 64, True), (4096, 8192, 16, True), (4096, 8192, 32, False),
         (8192, 8192, 64, True), (512, 8192, 32, False), (8192, 16384, 32, True)]


@pytest.mark.parametrize("N,Ng,tile,fold", CASES)
def test_own_grid_path_equals_separate_calls(rk, N, Ng, tile, fold):
    import torch
    img, obs = tiny_wstack(N + Ng + tile, nvis=3001, N=N, Nw=5, n_src=3)
    dev = to_device(obs)
    args = (dev["uvw"], dev["chan_scale"], dev["vis"], dev["weight"], None, dev["nrow"])
    with rk.Plan(plan_config(img, 1, tile=tile, hermitian_fold=fold, grid_size=Ng if Ng != N else 0)) as plan:
        P = plan.cfg.stored_planes
        got = torch.zeros((1, N, N), dtype=torch.float32, device="cuda")
        plan.dirty_image(*args, got)
        grids = torch.empty((1, P, Ng, Ng), dtype=torch.complex64, device="cuda")
        wsum = torch.empty(1, dtype=torch.float64, device="cuda")
        ref = torch.zeros_like(got)
        plan.grid(*args, 0, P, grids, wsum)
        plan.fft_wplanes(grids, P)
        plan.phase_correct_reduce(grids, 0, 1, 0, P, wsum, ref)
        A = torch.from_numpy(taper_gain(plan.taper())).cuda()
        err = float(((got - ref).abs() * A).max() / (ref.abs() * A).max())
        assert err <= TOL, err
        # prediction of the (taper-safe) central part of that image
        q = N // 4
        model = torch.zeros_like(ref)
        model[:, q:-q, q:-q] = ref[:, q:-q, q:-q] * A[q:-q, q:-q].float()
        vis = torch.empty((dev["nrow"], 1), dtype=torch.complex64, device="cuda")
        want = torch.zeros_like(vis)
        plan.predict(*args[:2], args[3], None, dev["nrow"], model, vis)
        plan.bin_predict(*args[:2], args[3], None, dev["nrow"])
        plan.model_to_wplanes(model, 0, 1, 0, P, grids)
        plan.fft_wplanes_forward(grids, P)
        plan.degrid_binned(grids, 0, 1, 0, P, want)
        err = float((vis - want).abs().max() / want.abs().max())
        assert err <= TOL, err
        plan.sync_status()
