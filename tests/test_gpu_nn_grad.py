"""Parameter gradients of the network where the marching weight-gradient kernels (tiles of 64 x 8
columns, the (tile, plane) steps dealt to the blocks in contiguous ranges) can go wrong: a tile with
rows beyond ny, y wrapping more than once inside a tile's halo (ny = 2), one plane, blocks that cross
from one tile to the next in mid-column (more steps than blocks), three tile columns. The comparison
and its tolerance are those of the layer-by-layer gradient test."""
import pytest

import test_gpu_nn as nn_tests

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("shape", [(1, 2, 64), (40, 34, 128), (7, 12, 192), (2, 6, 64)],
                         ids=lambda s: "x".join(map(str, s)))
@pytest.mark.parametrize("cin", [1, 2])
def test_marching_gradients_match_oracle(shape, cin):
    nn_tests.test_gradient_matches_oracle_layers_with_bf16_storage(shape, cin)
