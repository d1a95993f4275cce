"""Grids with more rows than a launch takes blocks in y (65535): the forms on whole-column tiles, whose grid has a
block row per one, two or four rows of columns."""
import pytest
import torch

from gpu_common import host
from paper_1402_3545_gb300 import tpmg

pytestmark = pytest.mark.gpu


def operator(nx, ny, nz, nlevels):
    return tpmg.Operator(nx, ny, nz, 1e-2, 1e-2, 1e-2, 1.0 / nz, 1e3, nlevels=nlevels)


@pytest.mark.parametrize("prec", [tpmg.F32, tpmg.DW], ids=["f32", "dw"])
def test_smooth(prec):
    """The tile variant against the plane-marching one, which takes any number of rows: the same bits."""
    nx, ny, n = 64, 131076, 64 * 131076
    op = operator(nx, ny, 1, 1)
    dt = torch.float32 if prec == tpmg.F32 else torch.float64
    u, f = (torch.randn(n, dtype=dt, device="cuda") for _ in range(2))
    out = []
    for variant in (0, 3):
        tpmg.set_variant(op.op, prec, 1, variant)
        out.append(torch.empty_like(u))
        tpmg.smooth(op.op, 1, prec, 0.8, u, f, out[-1], n)
    assert torch.equal(*out)
    op.close()


def test_residual_and_restriction():
    nx, ny, n = 128, 131076, 128 * 131076
    op = operator(nx, ny, 1, 2)
    u, f = (torch.randn(n, dtype=torch.float32, device="cuda") for _ in range(2))
    fc, uc, r, fc2, uc2 = (torch.empty(m, dtype=torch.float32, device="cuda") for m in (n // 4, n // 4, n, n // 4, n // 4))
    tpmg.residual_restrict_smooth(op.op, 1, tpmg.F32, 0.8, u, f, fc, uc, n, n // 4)
    tpmg.residual(op.op, 2, tpmg.F32, u, f, r, n)
    tpmg.restrict_smooth(op.op, 1, tpmg.F32, 0.8, r, fc2, uc2, n, n // 4)
    assert torch.equal(fc, fc2) and torch.equal(uc, uc2)
    op.close()


def test_line_solve_and_tridiag():
    """Columns are independent: the first rows are those of a short grid with the same coefficients, bit for bit."""
    nx, ny, nz, few = 128, 65540, 16, 64
    op, small = operator(nx, ny, nz, 1), operator(nx, few, nz, 1)
    n, m = nx * ny * nz, nx * few * nz
    b = torch.randn(nz, ny, nx, dtype=torch.float32, device="cuda")
    x, z = torch.empty_like(b), torch.empty_like(b)
    tpmg.line_solve(op.op, 1, tpmg.F32, b, x, n)
    want = torch.empty(nz, few, nx, dtype=torch.float32, device="cuda")
    for rows in (slice(0, few), slice(ny - few, ny)):
        tpmg.line_solve(small.op, 1, tpmg.F32, b[:, rows].contiguous(), want, m)
        assert torch.equal(x[:, rows], want)
    rr, rz = (torch.zeros(1, dtype=torch.float64, device="cuda") for _ in range(2))
    tpmg.cg_fused_tridiag(op.op, tpmg.F32, 0.0, b, torch.zeros_like(b), z, rr, rz, n)
    assert (z - x).abs().max() <= 1e-5 * x.abs().max()
    # <r, r> in FP32 partial sums of at most 128 x 16 terms each: below 2048 * 2^-24 of it
    assert abs(host(rr)[0] / float((b.double() ** 2).sum()) - 1.0) < 2048 * 2.0 ** -24
    op.close()
    small.close()
