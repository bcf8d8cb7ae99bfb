"""The block that one CTA of a layer's cluster finishes alone: 32 a side only in FP32 and
only where it holds two levels or more, else 16 at most (or a row per CTA)."""
import pytest

from host_plan import coarse_sides
from synth import configs


@pytest.fixture(scope="module")
def folder(tmp_path_factory):
    return tmp_path_factory.mktemp("hostplan")


@pytest.mark.parametrize("N,levels,precision,side", [
    (128, 4, 0, 32), (128, 5, 0, 32), (128, 3, 0, 16), (128, 2, 0, 16), (128, 1, 0, 16),
    (128, 4, 1, 16), (128, 5, 1, 16), (64, 3, 0, 16), (64, 4, 1, 16), (32, 3, 0, 16), (32, 3, 1, 16), (16, 2, 0, 8)])
def test_coarse_side(folder, N, levels, precision, side):
    n_sub = N // 4
    g = configs.small_lgs_config(n_sub=n_sub, N=N, n_layers=2, levels=levels, order=2, precision=precision)
    assert coarse_sides(g, 0, 1, folder) == [side, side]
