"""The fused SpMV of CG where its blocks take several planes (large grids) and on rows that end inside a warp, folded and
not; the comparison and its tolerances are those of the small grids' test, whose blocks take one or two planes."""
import pytest

import test_gpu_tiles as tiles
from gpu_common import PREC_IDS, PRECS

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("shape", [(640, 136, 33), (66, 600, 32), (130, 1200, 17), (200, 96, 5), (34, 700, 33), (78, 131, 17), (88, 180, 45),
                                   (88, 90, 203)],
                         ids=lambda s: "x".join(map(str, s)))
@pytest.mark.parametrize("prec", PRECS, ids=PREC_IDS)
def test_cg_spmv_matches_oracle(prec, shape):
    tiles.test_cg_spmv_matches_oracle(prec, shape)
