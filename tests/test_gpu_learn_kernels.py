"""The training objective's kernels at the sizes where their work split can go
wrong (probe counts around a warp, visibility counts around a staged block, the
smallest mesh), against the same sums in FP64 numpy.

Bars: a term's phases are exact to a few 1e-7 turns, so a sum of random-phase terms
is within 1e-5 of its largest value; the table gradient multiplies by I - D, of the
size of I here (random table), so 1e-4 of its largest entry."""
import numpy as np
import pytest

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


def _reference(N, Nw, L, fov, w, uvw, W, table, src, probes):
    g = lambda s: np.where(np.abs(s) <= 2, np.i0(KB_BETA_S4 * np.sqrt(np.maximum(0, 1 - (s / 2) ** 2))), 0) / np.i0(KB_BETA_S4)  # noqa: E731
    x, wt = np.polynomial.legendre.leggauss(24)
    nodes = (np.arange(4)[:, None] - 1.5 + 0.5 * x).ravel()
    taper = (np.cos(2 * np.pi / N * (np.arange(N) - N // 2)[:, None] * nodes) * g(nodes) * np.tile(0.5 * wt, 4)).sum(1)
    lm = (src[:, :2] - N // 2) * fov / N
    n = np.sqrt(1 - (lm ** 2).sum(1))
    V = (src[:, 2] / n * np.exp(-2j * np.pi * (uvw[:, :2] @ lm.T + uvw[:, 2:] * (n - 1)))).sum(1) * W
    sx = uvw[:, :2] * fov + N / 2 - 2
    first = np.floor(sx).astype(int) + 1
    f = sx - np.floor(sx)
    k = np.clip(np.floor((uvw[:, 2] + w) * Nw / (2 * w)), 0, Nw - 1).astype(int)
    a = np.arange(4)
    at = np.minimum((f * L).astype(int), L - 1)
    r = f * L - at
    gx = g(a + 1 - 2 - f[:, :, None])
    taps = gx[:, 1, :, None] * gx[:, 0, None, :]
    corners = [(dy, dx, (r[:, 0] if dx else 1 - r[:, 0]) * (r[:, 1] if dy else 1 - r[:, 1])) for dy in (0, 1) for dx in (0, 1)]
    tab = table.reshape(Nw, L + 1, L + 1, 4, 4)
    for dy, dx, c in corners:
        taps = taps + c[:, None, None] * tab[k, at[:, 1] + dy, at[:, 0] + dx]
    P = probes - N // 2
    plm = P * fov / N
    pn = np.sqrt(1 - (plm ** 2).sum(1))
    scale = pn / (taper[probes[:, 0]] * taper[probes[:, 1]])
    wk = -w + (k + 0.5) * 2 * w / Nw if Nw > 1 else 0 * k
    E = [np.exp(2j * np.pi * (first[:, d, None, None] + a - N // 2) * P[:, d][None, :, None] / N) for d in (0, 1)]
    c = scale * V[:, None] * np.exp(2j * np.pi * wk[:, None] * (pn - 1))
    term = np.einsum("np,npb,npa->npba", c, E[1], E[0]).real
    I = np.einsum("npba,nba->p", term, taps) / W.sum()
    D = (pn * V[:, None] * np.exp(2j * np.pi * (uvw[:, :2] @ plm.T + uvw[:, 2:] * (pn - 1)))).real.sum(0) / W.sum()
    ge = 2 * (I - D) / (D ** 2).sum() / W.sum()
    gt = np.einsum("p,npba->nba", ge, term)
    grad = np.zeros_like(tab)
    for dy, dx, cw in corners:
        np.add.at(grad, (k, at[:, 1] + dy, at[:, 0] + dx), cw[:, None, None] * gt)
    return I, D, ((I - D) ** 2).sum() / (D ** 2).sum(), grad.reshape(table.shape)


@pytest.mark.parametrize("N,Nw,L,nvis,ns,npr", [(64, 1, 1, 1, 1, 1), (128, 3, 4, 127, 2, 31), (128, 2, 8, 129, 64, 32),
                                               (256, 5, 3, 1003, 3, 33), (2048, 4, 16, 3001, 7, 64)])
def test_field_gradient_matches_fp64(rk, N, Nw, L, nvis, ns, npr):
    import torch
    r = np.random.default_rng(N + nvis)
    fov, w = 0.02, 150.0
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
    tab, loss, idft = dev(table), torch.empty(1, device="cuda"), torch.empty((npr, 2), device="cuda")
    # a gradient buffer that is 4-byte aligned only, then an aligned one: added to the same sum
    buf = torch.zeros(table.size + 1, device="cuda")
    odd, grad = buf[1:], torch.zeros(table.size, device="cuda")
    learn.field_grad(tab, src, probes, grad, loss, idft)
    learn.field_grad(tab, src, probes, odd, loss, idft, accumulate=True, grad_scale=0.5)
    I, D, want_loss, want = _reference(N, Nw, L, fov, w, uvw, W.astype(np.float64), table.astype(np.float64),
                                       src.astype(np.float64), probes)
    got = idft.cpu().numpy()
    top = np.abs(np.stack([I, D])).max()
    assert np.abs(got[:, 0] - I).max() <= 1e-5 * top and np.abs(got[:, 1] - D).max() <= 1e-5 * top
    assert abs(float(loss) - want_loss) <= 1e-4 * want_loss
    for g, scale in ((grad, 1.0), (odd, 0.5)):
        assert np.abs(g.cpu().numpy().reshape(want.shape) - scale * want).max() <= 1e-4 * np.abs(want).max()
