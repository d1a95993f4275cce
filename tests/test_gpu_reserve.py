"""What tpmg_op_reserve promises: the workspace that a solver of that precision needs is there afterwards, so that
solves, cycles and single applications allocate nothing."""
import numpy as np
import pytest
import torch

from gpu_common import PRECS, make_problem
from paper_1402_3545_gb300 import tpmg, workloads

pytestmark = pytest.mark.gpu


@pytest.fixture
def blocks():
    """The device blocks the library asks for, by address, from PyTorch's allocator."""
    held = {}

    def alloc(nbytes):
        p = torch.cuda.caching_allocator_alloc(nbytes)
        held[p] = nbytes
        return p

    tpmg.set_allocator(alloc, torch.cuda.caching_allocator_delete)
    yield held
    tpmg.use_cuda_allocator()


# finest level, one in double-word, three and more in native FP64 below it, 128^2 columns the uppermost of them; levels
# of at most 4096 columns only; a single level beyond double-word's reach
@pytest.mark.parametrize("shape,lam,levels", [((512, 512, 16), 4e6, 5), ((128, 96, 12), None, 3), ((64, 64, 32), 1e8, 1)],
                         ids=["ill-conditioned", "small", "no-double-word"])
@pytest.mark.parametrize("prec", PRECS + [tpmg.MIXED], ids=["f64", "dw", "f32", "mixed"])
def test_nothing_is_allocated_after_reserve(blocks, prec, shape, lam, levels):
    p = make_problem(*shape, lam=None if lam is None else lam / 1e3 * workloads.lambda2_varying(*shape[:2]))
    op = tpmg.Operator.from_problem(p, nlevels=levels)
    tpmg.op_reserve(op.op, prec)
    before = dict(blocks)
    dt = torch.float32 if prec == tpmg.F32 else torch.float64
    f = torch.randn(p.n, dtype=dt, device="cuda")
    u = torch.zeros_like(f)
    prm = tpmg.default_params(prec=prec, tol=0.0, max_iter=2)
    tpmg.mg_solve(op.op, prm, f, u, p.n)
    if prec != tpmg.MIXED:
        tpmg.vcycle(op.op, prm, f, u, p.n)
        tpmg.cg_solve(op.op, prm, f, u, p.n)
        for l in range(1, op.L + 1):
            n, w = op.level_n(l), torch.empty_like(f)
            tpmg.apply_A(op.op, l, prec, f[:n], w[:n], n)
            tpmg.line_solve(op.op, l, prec, f[:n], w[:n], n)
            tpmg.smooth(op.op, l, prec, 0.8, f[:n], u[:n], w[:n], n)
            tpmg.residual(op.op, l, prec, f[:n], u[:n], w[:n], n)
            if l < op.L:
                m, c = op.level_n(l + 1), [torch.empty(n, dtype=dt, device="cuda") for _ in range(2)]
                tpmg.restrict_smooth(op.op, l, prec, 0.8, f[:m], *c, m, n)
                if prec == tpmg.DW:
                    tpmg.residual_restrict_smooth(op.op, l, prec, 0.8, u[:m], f[:m], *c, m, n)
                tpmg.prolongate(op.op, l + 1, prec, c[0], w[:m], n, m)
    torch.cuda.synchronize()
    new = sorted(nb for a, nb in blocks.items() if a not in before)
    assert not new, (len(new), sum(new))
    op.close()
