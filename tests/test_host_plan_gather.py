"""Shared memory of the separate gather, from the host plan alone: a plan that is accepted
can be launched (220 KB a CTA), also where one node row has more pupil-edge terms than fit."""
import pytest

from gather_systems import many_edge_terms
from host_plan import gather_sizes

LIMIT = 220 * 1024


@pytest.fixture(scope="module")
def folder(tmp_path_factory):
    return tmp_path_factory.mktemp("hostplan")


@pytest.mark.parametrize("n_tt", [20, 56, 60])
def test_an_accepted_plan_can_launch_its_gather(folder, n_tt):
    bands, smem, terms = gather_sizes(many_edge_terms(n_tt), 64, 2, folder)
    assert bands == 512 or smem <= 108 * 1024
    # 501 terms a sensor (more where tip/tilt removal adds its own), 8 bytes each beside the row's nodes
    assert (terms * 8 + 512 * 8 > LIMIT) == (n_tt >= 56)
    assert smem <= LIMIT
