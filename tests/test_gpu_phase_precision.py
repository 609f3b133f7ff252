"""The phase screen of the separate reduction far along a long stack of planes: only
plane k = 4088 of 4096 is not zero, so the complex image's argument is that plane's
phase 2 pi w_k (n - 1), k steps of the plane spacing from the first.

Bar: the phase is carried in 64-bit turns, whose top 32 bits are rounded to FP32 (half
a unit of 2^-24 half-turns: 9.4e-8 rad) before sincospif (2 ulp, 1.7e-7) and two fused
multiply-adds (1.2e-7): 5e-7.  Turns and steps of 32 bits are 3e-6 rad off there."""
import numpy as np
import pytest

from tests.gpu_util import plan_config
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


@pytest.mark.parametrize("k0", [0, 4080])
def test_phase_of_a_late_plane(rk, k0):
    import torch
    N, Nw, k = 256, 4096, 4088
    img, _ = tiny_wstack(0, nvis=8, N=N, Nw=Nw)
    with rk.Plan(plan_config(img, 1)) as plan:
        grids = torch.zeros((1, Nw - k0, N, N), dtype=torch.complex64, device="cuda")
        grids[0, k - k0] = 1.0
        image = torch.zeros((1, N, N), dtype=torch.float32, device="cuda")
        cplx = torch.zeros((1, N, N), dtype=torch.complex64, device="cuda")
        plan.phase_correct_reduce(grids, 0, 1, k0, Nw, torch.ones(1, dtype=torch.float64, device="cuda"), image, cplx)
        plan.sync_status()
        got = cplx[0].cpu().numpy().astype(np.complex128)
    x = (np.arange(N) - N // 2) * (img.fov / N)
    r2 = x[:, None] ** 2 + x ** 2
    turn = (img.w_min + (k + 0.5) * (img.w_max - img.w_min) / Nw) * (-r2 / (1 + np.sqrt(1 - r2)))
    sign = 1 - 2 * ((np.arange(N)[:, None] + np.arange(N)) & 1)
    err = np.abs(sign * got / np.abs(got) - np.exp(2j * np.pi * turn)).max()
    print(f"first plane {k0}: {err:.2e}")
    assert err <= 5e-7
    assert np.array_equal(image[0].cpu().numpy(), cplx[0].real.cpu().numpy())
