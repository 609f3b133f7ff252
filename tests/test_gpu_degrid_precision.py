"""The rounding of the degridder's footprint sums: planes of a model amplified by
1/taper, as a prediction's are, handed straight to rick_degrid_binned, against the
same sums in FP64 with the same FP32 taps.

Bar: the RMS error of one chain of fused multiply-adds along every footprint row and
one over the rows (a rounding per cell), restated here in FP32; 10 % more covers tap
coefficients that the host's two fits may round differently.  Sums whose products are
rounded before they are added are 1.2 (support 4) to 1.4 (support 7) times as far off here."""
import math

import numpy as np
import pytest

pytestmark = pytest.mark.gpu
DEGREE = 11
f4, f8 = np.float32, np.float64


@pytest.fixture(scope="module")
def rk():
    import __graft_entry__
    __graft_entry__.build()
    import torch
    assert torch.cuda.is_available(), "GPU tests need a CUDA device"
    from paper_2601_19714_gb300 import rick
    rick.load()
    return rick


def _fma(a, b, c):
    return (np.asarray(a, f8) * np.asarray(b, f8) + np.asarray(c, f8)).astype(f4)


def _kernel(S, s):
    beta = math.pi * math.sqrt(0.25 * S * S - 0.8)
    return np.where(np.abs(s) <= S / 2, np.i0(beta * np.sqrt(np.maximum(0, 1 - (2 * s / S) ** 2))) / np.i0(beta), 0)


def _taps(S, f):
    """The S taps at the fractions f: FP32 Horner of the degree-DEGREE Chebyshev fits."""
    t = _fma(2, f, -1)
    out = []
    for a in range(S):
        c = np.polynomial.chebyshev.Chebyshev.interpolate(lambda t: _kernel(S, a + 1 - 0.5 * S - 0.5 * (t + 1)), DEGREE)
        m = np.zeros(DEGREE + 1)
        q = np.polynomial.chebyshev.cheb2poly(c.coef)
        m[:len(q)] = q
        acc = np.full_like(t, m[DEGREE], dtype=f4)
        for k in range(DEGREE - 1, -1, -1):
            acc = _fma(acc, t, f4(m[k]))
        out.append(acc * f4(1 - 2 * (a & 1)))   # the checkerboard sign of the tap
    return out


def _planes(S, N, g):
    model = np.zeros((N, N))
    at = (N * (0.5 + 0.7 * (g.random((200, 2)) - 0.5))).astype(int)
    model[at[:, 0], at[:, 1]] = g.exponential(0.3, 200)
    x, wt = np.polynomial.legendre.leggauss(24)
    s = (np.arange(S)[:, None] - 0.5 * S + 0.5 + 0.5 * x).ravel()
    taper = (np.cos(2 * np.pi / N * (np.arange(N) - N // 2)[:, None] * s) * _kernel(S, s) * np.tile(0.5 * wt, S)).sum(1)
    sign = 1 - 2 * ((np.arange(N)[:, None] + np.arange(N)) & 1)
    return np.fft.fft2(model * sign / (taper[:, None] * taper)).astype(np.complex64)


@pytest.mark.parametrize("S", [4, 5, 6, 7, 8])
def test_footprint_sums_round_once_a_cell(rk, S):
    import torch
    N, n, fov = 256, 20_000, 2.0 ** -6
    g = np.random.default_rng(S)
    F = _planes(S, N, g)
    ij = g.integers(0, N - S, (n, 2))
    f = (g.integers(0, 1 << 24, (n, 2)) / 2.0 ** 24).astype(f4)   # positions are exact
    uvw = np.zeros((n, 3))
    uvw[:, :2] = (ij - 1 + f.astype(f8) + 0.5 * S - N / 2) / fov
    gx, gy = _taps(S, f[:, 0]), _taps(S, f[:, 1])
    s0 = (1 - 2 * (ij.sum(1) & 1)).astype(f4)
    exact, chain = [], []
    for part in (F.real, F.imag):
        cells = [[part[ij[:, 1] + b, ij[:, 0] + a] for a in range(S)] for b in range(S)]
        acc, sum64 = np.zeros(n, f4), 0.0
        for b in range(S):
            row, row64 = np.zeros(n, f4), 0.0
            for a in range(S):
                row = _fma(s0 * gx[a], cells[b][a], row)
                row64 = row64 + (s0 * gx[a]).astype(f8) * cells[b][a]
            acc, sum64 = _fma(gy[b], row, acc), sum64 + gy[b].astype(f8) * row64
        exact.append(sum64)
        chain.append(acc)
    cfg = rk.Config(N=N, n_wplanes=1, support=S, n_channels=1, fov_rad=fov, w_min=-1.0, w_max=1.0, kernel="kb",
                    kernel_param=math.pi * math.sqrt(0.25 * S * S - 0.8))
    dev = lambda a: torch.from_numpy(np.ascontiguousarray(a)).cuda()  # noqa: E731
    with rk.Plan(cfg) as plan:
        plan.bin_predict(dev(uvw), dev(np.ones(1)), dev(np.ones((n, 1), f4)), None, n)
        vis = torch.zeros((n, 1), dtype=torch.complex64, device="cuda")
        plan.degrid_binned(dev(F.reshape(1, 1, N, N)), 0, 1, 0, 1, vis)
        plan.sync_status()
        got = vis.cpu().numpy()[:, 0]
    rms = lambda re, im: math.sqrt(np.mean((re - exact[0]) ** 2 + (im - exact[1]) ** 2))  # noqa: E731
    err, bar = rms(got.real.astype(f8), got.imag.astype(f8)), rms(chain[0].astype(f8), chain[1].astype(f8))
    print(f"S={S}: {err / bar:.4f} of the chains' error ({bar / math.sqrt(np.mean(exact[0] ** 2 + exact[1] ** 2)):.2e})")
    assert err <= 1.1 * bar
