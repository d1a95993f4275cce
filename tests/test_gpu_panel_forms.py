"""The panel's kernels on both sides of the rule that gives a level's columns to chunks of planes (6, 10, 12 and 32
planes by the number of columns), the pointwise ones with one, few and sixteen planes a thread; the comparison and its
tolerance are those of the smaller panels' test."""
import pytest

import test_gpu_panel as panel

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("shape", [(64, 64, 1, 2), (64, 66, 5, 2), (64, 66, 6, 2), (104, 100, 9, 2), (104, 100, 10, 2),
                                   (130, 130, 11, 2), (130, 130, 12, 2), (160, 158, 31, 2), (160, 158, 32, 2), (34, 20, 3, 2), (260, 258, 17, 2),
                                   (260, 258, 1, 2), (138, 446, 5, 2),
                                   (170, 170, 33, 2), (170, 170, 65, 2)],
                         ids=lambda s: "x".join(map(str, s)))
def test_kernels_match_the_oracle_on_every_level(shape):
    panel.test_kernels_match_the_oracle_on_every_level(shape)
