"""Hybrid Gauss-Seidel on few large macros (a launch per colour from three rounds a cluster on) and on small
macros (all colours in one launch), by the check of test_gpu_gs.py."""

import pytest

import test_gpu_gs as G

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("macros,level", [(1, 6), (2, 6), (2, 5), (24, 4), (24, 5)])
def test_colours_of_few_and_of_small_macros(macros, level):
    G.test_colours_follow_the_definition(macros, level)
