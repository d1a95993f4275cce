"""The norms' partial sums: all of them lie in the first half of the operator's buffer (the second half is for the
second sum of CG), on the grids whose kernels write the most for their size."""
import pytest
import torch

from gpu_common import host
from paper_1402_3545_gb300 import tpmg

pytestmark = pytest.mark.gpu


class Block:
    """A device block of the library's, as an array of doubles."""

    def __init__(self, address, nbytes):
        self.__cuda_array_interface__ = {"shape": (nbytes // 8,), "typestr": "<f8", "data": (address, False), "version": 3}


def matching_blocks(held, norm):
    """The blocks whose first half adds up to the squared norm."""
    out = []
    for address, nbytes in held.items():
        half = torch.as_tensor(Block(address, nbytes), device="cuda")[:nbytes // 16]
        if nbytes <= 1 << 20 and abs(float(half.sum()) - norm ** 2) <= 1e-9 * norm ** 2:
            out.append(nbytes)
    return out


@pytest.mark.parametrize("kind,shape,level", [("box", (224, 200, 48), 1), ("box", (224, 200, 48), 2), ("box", (64, 64, 128), 2),
                                              ("panel", (512, 130, 8), 2), ("panel", (64, 66, 33), 2), ("panel", (34, 2, 7), 2)],
                         ids=lambda v: "x".join(map(str, v)) if isinstance(v, tuple) else str(v))
def test_partial_sums_fit_their_half(kind, shape, level):
    held = {}

    def alloc(nbytes):
        p = torch.cuda.caching_allocator_alloc(nbytes)
        held[p] = nbytes
        return p

    tpmg.set_allocator(alloc, torch.cuda.caching_allocator_delete)
    try:
        nx, ny, nz = shape
        if kind == "box":
            op = tpmg.Operator(nx, ny, nz, 1e-2, 1.0 / nx, 1.0 / ny, 1.0 / nz, 1e3, nlevels=2)
        else:
            op = tpmg.PanelOperator(nx, ny, nz, 1e-4, 1.0, 1e-3, nlevels=2)
        n = op.level_n(level)
        u, f = (torch.randn(n, dtype=torch.float64, device="cuda") for _ in range(2))
        r, norm = torch.empty_like(u), torch.zeros(1, dtype=torch.float64, device="cuda")
        if kind == "box":
            tpmg.residual(op.op, level, tpmg.F64, u, f, r, n, norm_out=norm)
        else:
            tpmg.panel_residual(op.op, level, u, f, r, n, norm_out=norm)
        got = host(norm)[0]
        assert abs(got - float(r.norm())) <= 1e-12 * got
        assert len(matching_blocks(held, got)) == 1
        op.close()
    finally:
        tpmg.use_cuda_allocator()
