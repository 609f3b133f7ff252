"""The cropped row passes of the smallest meshes (64 threads a row, radix 4 and 8) on
every padding: the plan's own grid path against the separate calls, with the bar of
tests/test_gpu_columns.py."""
import pytest

from tests import test_gpu_columns as columns

pytestmark = pytest.mark.gpu
rk = columns.rk


@pytest.mark.parametrize("N,Ng,tile,fold", [(64, 256, 16, False), (64, 256, 32, True), (128, 256, 16, True),
                                            (128, 256, 64, False), (64, 512, 64, True), (128, 512, 32, False)])
def test_own_grid_path_of_small_padded_meshes(rk, N, Ng, tile, fold):
    columns.test_own_grid_path_equals_separate_calls(rk, N, Ng, tile, fold)
