"""Each side of the rules that deal levels to kernel forms by size: both forms under the comparisons, and their
tolerances, of the forms' own tests."""
import pytest
import torch

import test_gpu_tiles as tiles
from gpu_common import PREC_IDS, PRECS, make_problem
from paper_1402_3545_gb300 import tpmg

pytestmark = pytest.mark.gpu


def ids(s):
    return "x".join(map(str, s))


# FP32: tiles from 16 planes; where there is the two-column sweep (nx a multiple of 64) up to 32768 columns, up to 58368
# from 24 planes and up to 65536 beyond 64
@pytest.mark.parametrize("lam", [None, 1e3], ids=["varying", "constant"])
@pytest.mark.parametrize("shape", [(256, 128, 16), (256, 132, 16), (256, 132, 23), (256, 228, 24),
                                   (256, 232, 24), (256, 256, 64), (256, 256, 65), (512, 130, 65), (352, 132, 17), (96, 704, 40), (352, 132, 15)], ids=ids)
def test_fp32_tridiag(shape, lam):
    tiles.test_tile_line_solve_and_tridiag_match_oracle(tpmg.F32, shape, lam)


# FP32, lambda^2 varying, from 262144 columns: the four-column tile of a warp up to 64 planes
@pytest.mark.parametrize("shape", [(512, 256, 17), (512, 260, 17), (512, 260, 64), (512, 260, 65), (512, 510, 17), (512, 512, 17),
                                   (512, 516, 64), (512, 516, 65)], ids=ids)
def test_fp32_line_solve(shape):
    tiles.test_tile_line_solve_and_tridiag_match_oracle(tpmg.F32, shape, None)


# the pointwise Residual's planes per thread: one to four on small levels, fewer blocks with the norm, sixteenths beyond
@pytest.mark.parametrize("shape", [(8, 8, 256), (34, 20, 8), (64, 64, 29), (64, 64, 256), (128, 128, 13), (192, 126, 29),
                                   (192, 126, 67), (370, 330, 7)], ids=ids)
@pytest.mark.parametrize("prec", PRECS, ids=PREC_IDS)
def test_residual_planes(prec, shape):
    tiles.test_pointwise_residual_matches_oracle(prec, shape)
    nx, ny, nz = shape
    op = tiles.operator(nx, ny, nz, None, nlevels=1)
    u, f = tiles.fields((nz, ny, nx), prec, 3)
    r, norm = [torch.empty_like(u) for _ in range(2)], torch.zeros(1, dtype=torch.float64, device="cuda")
    tpmg.residual(op.op, 1, prec, u, f, r[0], u.numel())
    tpmg.residual(op.op, 1, prec, u, f, r[1], u.numel(), norm_out=norm)
    assert torch.equal(*r)
    op.close()


# FP32 Residual + RestrictSmooth: tiles from 6 planes, or up to 131072 fine columns; the marching form else
@pytest.mark.parametrize("lam", [None, 1e3], ids=["varying", "constant"])
@pytest.mark.parametrize("shape", [(512, 256, 5), (512, 258, 5), (512, 258, 6), (512, 258, 1)], ids=ids)
def test_fp32_residual_restriction(shape, lam):
    tiles.test_restrict_tile_equals_the_two_kernels(tpmg.F32, shape, True, lam)


# native FP64 levels between cyclic reduction and chunks of planes: up to 512, 608, 752 and 912 columns
@pytest.mark.parametrize("lam,shape", [(None, s) for s in ((20, 20, 80), (20, 20, 81), (24, 24, 64), (24, 24, 128), (24, 24, 129),
                                                          (26, 24, 48), (26, 24, 49), (32, 24, 80), (32, 24, 81))] +
                         [(1e3, s) for s in ((20, 20, 65), (16, 32, 256), (24, 24, 200), (24, 24, 201), (26, 24, 160), (26, 24, 161),
                                             (32, 24, 40), (32, 24, 41), (32, 24, 96), (32, 24, 97))],
                         ids=lambda v: ids(v) if isinstance(v, tuple) else ("varying" if v is None else "constant"))
def test_fp64_columns(shape, lam, monkeypatch):
    monkeypatch.setattr(tiles, "make_problem", lambda *size: make_problem(*size, lam=lam))
    tiles.test_chunked_columns_match_oracle(shape)
