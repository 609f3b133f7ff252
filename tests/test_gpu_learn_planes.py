"""Learned training on more w-planes than the plane phasors' share of shared memory
holds (422), next to it and far beyond, against FP64 numpy with the bars of
tests/test_gpu_learn_kernels.py."""
import numpy as np
import pytest

from tests.test_gpu_learn_kernels import _reference
from visgen.workloads import KB_BETA_S4

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


@pytest.mark.parametrize("Nw", [422, 423, 447, 1000])
def test_field_gradient_with_many_planes(rk, Nw):
    import torch
    N, L, nvis, ns, npr, fov, w = 64, 2, 700, 3, 40, 0.02, 150.0
    r = np.random.default_rng(Nw)
    rad, t = 0.4 * N / fov * np.sqrt(r.random(nvis)), 2 * np.pi * r.random(nvis)
    uvw = np.stack([rad * np.cos(t), rad * np.sin(t), w * (2 * r.random(nvis) - 1)], 1)
    W = (0.5 + r.random(nvis)).astype(np.float32)
    src = np.concatenate([N * (0.2 + 0.6 * r.random((ns, 2))), 0.1 + r.random((ns, 1))], 1).astype(np.float32)
    probes = r.integers(N // 4, 3 * N // 4, (npr, 2)).astype(np.int32)
    table = (0.3 * r.standard_normal((Nw * (L + 1) ** 2, 16))).astype(np.float32)
    cfg = rk.Config(N=N, n_wplanes=Nw, support=4, n_channels=1, fov_rad=fov, w_min=-w, w_max=w, kernel="table",
                    kernel_param=KB_BETA_S4)
    dev = lambda a: torch.from_numpy(a).cuda()  # noqa: E731
    learn = rk.Learn(cfg, L, dev(uvw), dev(W))
    loss, idft, grad = (torch.empty(n, device="cuda") for n in ((1,), (npr, 2), (table.size,)))
    learn.field_grad(dev(table), src, probes, grad, loss, idft)
    I, D, want_loss, want = _reference(N, Nw, L, fov, w, uvw, W.astype(np.float64), table.astype(np.float64),
                                       src.astype(np.float64), probes)
    got, top = idft.cpu().numpy(), np.abs(np.stack([I, D])).max()
    assert np.abs(got[:, 0] - I).max() <= 1e-5 * top and np.abs(got[:, 1] - D).max() <= 1e-5 * top
    assert abs(float(loss) - want_loss) <= 1e-4 * want_loss
    assert np.abs(grad.cpu().numpy().reshape(want.shape) - want).max() <= 1e-4 * np.abs(want).max()
