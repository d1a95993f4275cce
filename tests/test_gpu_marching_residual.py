"""The residual kernels that march through the planes, on grids large enough that no pointwise one takes them: two
columns per thread (nx a multiple of 64, even ny), one column with tiles (of 32 only) and, above 131072 columns in
native FP64, without. The comparisons and their tolerances are those of the smaller grids' tests."""
import pytest

import test_gpu_tiles as tiles
import test_zz_no_alloc as noalloc
from gpu_common import PREC_IDS, PRECS

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("shape", [(256, 132, 9), (224, 160, 9), (370, 370, 3), (192, 172, 1), (192, 172, 2)],
                         ids=lambda s: "x".join(map(str, s)))
@pytest.mark.parametrize("prec", PRECS, ids=PREC_IDS)
def test_residual_matches_oracle(prec, shape):
    tiles.test_pointwise_residual_matches_oracle(prec, shape)


@pytest.mark.parametrize("square", [True, False], ids=["square", "oblong"])
@pytest.mark.parametrize("shape", [(512, 68, 9), (256, 132, 33)], ids=lambda s: "x".join(map(str, s)))
@pytest.mark.parametrize("prec", PRECS, ids=PREC_IDS)
def test_fused_restriction_equals_the_marching_residual_and_the_restriction(prec, shape, square):
    tiles.test_restrict_tile_equals_the_two_kernels(prec, shape, square, None)


def test_noalloc_residual(monkeypatch):
    monkeypatch.setattr(noalloc, "CASES", [(256, 132, 9, 1), (224, 160, 9, 2), (370, 370, 3, 3)])
    noalloc.test_noalloc_residual_matches_regular_entry_point_and_oracle()
