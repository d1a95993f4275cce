"""How much the kernels round: attainable residuals, single applications against wider arithmetic, and long sums
against 64-bit ones."""
import numpy as np
import pytest
import torch

from gpu_common import dev, make_problem
from paper_1402_3545_gb300 import tpmg

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("shape,lam", [((128, 128, 128), None), ((128, 64, 128), 1e3)], ids=["varying", "constant"])
def test_double_word_attains_the_refinement_s_residual(shape, lam):
    """Cycles without end settle where the rounding of the stored iterate and of the residual does. The double-word
    and the mixed solver store the same pairs and form the residual by the same kernel, and what either adds to the
    iterate is rounded relative to the correction, so both settle at the same height; a factor of 2 allows for their
    corrections' different spectra. A smoother that rounds relative to u itself settles several times higher."""
    p = make_problem(*shape, lam=lam)
    op = tpmg.Operator.from_problem(p)
    f = dev(p.rhs(), tpmg.F64)
    level = {}
    for prec in (tpmg.DW, tpmg.MIXED):
        res = tpmg.mg_solve(op.op, tpmg.default_params(prec=prec, tol=0.0, max_iter=40), f, torch.zeros_like(f), p.n)
        level[prec] = np.median(res["history"][-10:])
    assert level[tpmg.DW] < 2.0 * level[tpmg.MIXED], level
    op.close()
