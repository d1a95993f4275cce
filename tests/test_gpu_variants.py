"""A tile variant changes the schedule of a level that sweeps its columns, and nothing on a level that does not."""
import pytest
import torch

from gpu_common import make_problem
from paper_1402_3545_gb300 import tpmg

pytestmark = pytest.mark.gpu


# native FP64 levels in chunks of planes, by cyclic reduction and on the sweep, with tiles (nx a multiple of 32)
@pytest.mark.parametrize("shape", [(128, 128, 64), (96, 64, 33), (64, 64, 16), (64, 64, 8), (256, 130, 16)],
                         ids=lambda s: "x".join(map(str, s)))
@pytest.mark.parametrize("norm", [False, True], ids=["plain", "norm"])
def test_fp64_smooth_is_that_of_the_untuned_level(shape, norm):
    p = make_problem(*shape)
    op = tpmg.Operator.from_problem(p, nlevels=1)
    u, f = (torch.randn(p.n, dtype=torch.float64, device="cuda") for _ in range(2))
    nrm = torch.zeros(1, dtype=torch.float64, device="cuda") if norm else None

    def run():
        o = torch.empty_like(u)
        tpmg.smooth(op.op, 1, tpmg.F64, 0.8, u, f, o, p.n, norm_out=nrm)
        return o

    untuned = run()
    for v in range(tpmg.NUM_VARIANTS):
        tpmg.set_variant(op.op, tpmg.F64, 1, v)
        assert torch.equal(run(), untuned), v
    op.close()
