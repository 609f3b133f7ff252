"""Tiles split over several CTAs, with the number of records that reach a tile set
exactly: at the thresholds of the split, with more chunks than a tile may have, and
with every tile of a mesh split; and the memory that a reservation takes, which the
splitting does not add to.

Bar of the planes: FP32 sums of n terms a cell in a fixed order, 2e-5 of the largest
cell as in tests/test_gpu_dense_tiles.py (at most 20 k terms a cell here, whose signs
vary)."""
import numpy as np
import pytest

from visgen.workloads import GAUSS_SIGMA_S7, KB_BETA_S8

pytestmark = pytest.mark.gpu
FOV = 2.0 ** -6   # positions in cells are exact


@pytest.fixture(scope="module")
def rk():
    import __graft_entry__
    __graft_entry__.build()
    import torch
    assert torch.cuda.is_available(), "GPU tests need a CUDA device"
    from paper_2601_19714_gb300 import rick
    rick.load()
    return rick


def _grid_and_compare(rk, tile, S, kernel, param, first, frac, N=256, sparse=False):
    """Grids visibilities whose footprints start at the cells `first`; returns the plan's bin offsets."""
    import torch

    import oracle as orc
    orc.build()
    n = len(first)
    g = np.random.default_rng(n + tile)
    uvw = np.zeros((n, 3))
    uvw[:, :2] = (first - 1 + frac + 0.5 * S - N / 2) / FOV
    vis = (g.standard_normal((n, 1)) + 1j * g.standard_normal((n, 1))).astype(np.complex64)
    weight = (0.5 + g.random((n, 1))).astype(np.float32)
    one = np.ones(1)
    dev = lambda a: torch.from_numpy(a).cuda()  # noqa: E731
    cfg = rk.Config(N=N, n_wplanes=1, support=S, n_channels=1, fov_rad=FOV, w_min=-1.0, w_max=1.0, kernel=kernel,
                    kernel_param=param, tile=tile)
    with rk.Plan(cfg) as plan:
        grids = torch.zeros((1, 1, N, N), dtype=torch.complex64, device="cuda")
        wsum = torch.empty(1, dtype=torch.float64, device="cuda")
        plan.bin(dev(uvw), dev(one), dev(vis), dev(weight), None, n, wsum)
        plan.grid_binned(0, 1, 0, 1, grids, sparse=sparse)
        again = torch.zeros_like(grids)
        plan.grid_binned(0, 1, 0, 1, again, sparse=sparse)
        plan.sync_status()
        assert torch.equal(torch.view_as_real(again), torch.view_as_real(grids))   # a fixed order of additions
        offsets = plan.bin_offsets().astype(np.int64)
    ocfg = orc.Config(N=N, Nw=1, S=S, kernel=kernel, kernel_param=param, fov=FOV, w_min=-1.0, w_max=1.0)
    G = orc.grid_plane(ocfg, uvw, one, vis, weight, None, plane=0)
    assert np.abs(grids[0, 0].cpu().numpy() - G).max() <= 2e-5 * np.abs(G).max()
    return offsets


@pytest.mark.parametrize("tile,n", [(32, 8191), (32, 8192), (32, 8193), (32, 12_287), (32, 12_288), (32, 12_289),
                                    (16, 8191), (16, 8192), (64, 32_767), (64, 32_768), (64, 32_769),
                                    (32, 600_001)])   # the last: 147 chunks, of which 128 are made
@pytest.mark.parametrize("sparse", [False, True])
def test_exact_number_of_records_in_one_tile(rk, tile, n, sparse):
    g = np.random.default_rng(n)
    S = 7
    # footprints wholly inside the tile (1, 2) of the mesh
    first = np.stack([tile + g.integers(0, tile - S + 1, n), 2 * tile + g.integers(0, tile - S + 1, n)], 1)
    frac = g.integers(0, 1 << 24, (n, 2)) / 2.0 ** 24
    off = _grid_and_compare(rk, tile, S, "gauss", GAUSS_SIGMA_S7, first, frac, sparse=sparse)
    key = (2 * (256 // tile) + 1) * 4
    assert off[key + 1] - off[key] == n == off[-1]   # every record in the tile's own bin, none beyond it


def test_every_tile_split(rk):
    """1.05 M records over 256 tiles of 16 with S = 8: each reaches about two tiles."""
    n, S = 1_050_001, 8
    g = np.random.default_rng(3)
    first = g.integers(0, 256 - S, (n, 2))
    frac = g.integers(0, 1 << 24, (n, 2)) / 2.0 ** 24
    _grid_and_compare(rk, 16, S, "kb", KB_BETA_S8, first, frac)


@pytest.mark.parametrize("tile", [16, 32, 64])
def test_reservation_takes_forty_bytes_a_record(rk, tile):
    import torch
    n = 32_000_000
    cfg = rk.Config(N=256, n_wplanes=1, support=7, n_channels=1, fov_rad=FOV, w_min=-1.0, w_max=1.0, kernel="gauss",
                    kernel_param=GAUSS_SIGMA_S7, tile=tile)
    with rk.Plan(cfg) as plan:
        torch.cuda.synchronize()
        before = torch.cuda.mem_get_info()[0]
        plan.reserve(n)
        taken = before - torch.cuda.mem_get_info()[0]
    # key, rank, two records of 16 bytes; three lists of a tile index per T records; allocation granules
    assert taken <= (40 + 12 / tile) * n + (32 << 20), taken / n
