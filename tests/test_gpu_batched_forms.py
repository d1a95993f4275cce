"""The batched solver's forms by shared memory (k_batched.cu): tiles with per-column factors at and beyond what two
blocks of an SM hold, columns with and without them. The comparison is that of the other forms' test."""
import pytest

import test_gpu_tiles as tiles

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("shapes", [[(128, 64, 128), (192, 64, 120)], [(64, 64, 144), (128, 128, 161)], [(40, 24, 256), (96, 36, 1)]],
                         ids=["two-blocks", "beyond", "columns"])
@pytest.mark.parametrize("square", [True, False], ids=["square", "oblong"])
@pytest.mark.parametrize("lam", [None, 1e3], ids=["varying", "constant"])
def test_batched_forms_reach_the_single_solves(shapes, square, lam):
    tiles.test_batched_forms_reach_the_single_solves(shapes, square, lam)
