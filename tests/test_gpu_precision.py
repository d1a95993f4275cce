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


@pytest.mark.parametrize("cin,shape", [(2, (64, 256, 256)), (1, (64, 1024, 1024))], ids=["2^22", "2^26"])
def test_gradient_sums_of_one_sign_match_64_bit_sums(cin, shape):
    """A network whose layers pass channel 0 of x on (centre taps 1, the last layer's 1/16) and a target x - d: with
    the values chosen here no activation and no data gradient rounds (BF16 x in [1, 2), d of 8 bits down to 2^-12, a
    power of two of cells), so what remains are the gradients' own sums of 2^22 and 2^26 terms of one sign:
    S_ci(tap) = sum_p d4(p) x_ci(p + tap) and sum_p d4(p), times 1/16 below the last layer.

    Tolerances, of each element: the tensor cores cut off at most a unit in the last place (2^-23) per MMA. 16 -> 16
    layers: 256 MMAs to an accumulator. First and last: one, and the result's own rounding, below 2^-22. Biases: the
    result's rounding and those of many partial sums, which average out, below 2^-23."""
    nz, ny, nx = shape
    n = nx * ny * nz
    W = [np.zeros((16, cin, 27)), np.zeros((16, 16, 27)), np.zeros((16, 16, 27)), np.zeros((1, 16, 27))]
    W[0][:, 0, 13] = 1.0
    for w in W[1:3]:
        w[:, :, 13] = np.eye(16)
    W[3][0, :, 13] = 1.0 / 16.0
    net = tpmg.Network(cin, np.concatenate([np.concatenate([w.ravel(), np.zeros(w.shape[0])]) for w in W]).astype(np.float32))
    g = torch.Generator(device="cuda")
    g.manual_seed(11)

    def mantissa():
        return 1.0 + torch.randint(0, 128, shape, generator=g, device="cuda").float() / 128.0

    x = torch.stack([mantissa() for _ in range(cin)], dim=-1)
    d = torch.ldexp(mantissa(), -torch.randint(1, 13, shape, generator=g, device="cuda"))
    loss, grad = net.loss_grad(x.reshape(-1), (x[..., 0] - d).reshape(-1), shape)
    grad = grad.double().cpu().numpy()
    S = np.zeros((cin, 27))
    for dz in (-1, 0, 1):
        to, frm = slice(max(0, -dz), nz - max(0, dz)), slice(max(0, dz), nz - max(0, -dz))
        for dy in (-1, 0, 1):
            for dx in (-1, 0, 1):
                for ci in range(cin):
                    S[ci, ((dz + 1) * 3 + dy + 1) * 3 + dx + 1] = float(
                        (d[to].double() * x[frm][..., ci].roll((-dy, -dx), (1, 2))).sum())
    S, B = S * 2.0 / n, float(d.double().sum()) * 2.0 / n
    n1, n2 = 16 * cin * 27, 16 * 16 * 27
    at = np.cumsum([0, n1, 16, n2, 16, n2, 16, 16 * 27, 1])
    part = [grad[a:b] for a, b in zip(at[:-1], at[1:])]
    cut = 2.0 ** -23
    want = [np.tile(S.ravel() / 16, 16), B / 16, np.tile(S[0] / 16, 256), B / 16, np.tile(S[0] / 16, 256), B / 16,
            np.tile(S[0], 16), B]
    tol = [2 * cut, cut, 256 * cut, cut, 256 * cut, cut, 2 * cut, cut]
    off = [np.abs(p / w - 1.0).max() for p, w in zip(part, want)]
    assert all(o < t for o, t in zip(off, tol)), off
    net.close()


@pytest.mark.parametrize("what,shape,by", [("box", (130, 66, 3), 0), ("box", (130, 66, 3), 1), ("box", (32, 32, 8), 0),
                                           ("box", (64, 62, 96), 0), ("panel", (66, 64, 5), 0)],
                         ids=["vector", "any-alignment", "cells", "pairs-of-cells", "panel"])
def test_prolongation_rounds_once_relative_to_the_fine_field(what, shape, by):
    """u_f + P u_c with a correction of a tenth of u_f, as in a V-cycle, in native FP64 against extended precision.
    The correctly rounded sum has the r.m.s. error e of one rounding; P u_c adds at most five of a tenth of its size:
    sqrt(1 + 5 / 100) e. 1.25 e leaves room for that, not for more than one rounding at u_f's size."""
    nx, ny, nz = shape
    n, nc = nx * ny * nz, nx * ny * nz // 4
    rng = np.random.default_rng(17)
    uf, uc = rng.standard_normal((nz, ny, nx)), 0.1 * rng.standard_normal((nz, ny // 2, nx // 2))
    t = torch.empty(n + 2, dtype=torch.float64, device="cuda")[by:by + n]
    t.copy_(torch.from_numpy(uf.ravel()))
    if what == "box":
        op = tpmg.Operator(nx, ny, nz, 1e-2, 1.0 / nx, 1.0 / ny, 1.0 / nz, 1e3, nlevels=2)
        tpmg.prolongate(op.op, 2, tpmg.F64, dev(uc, tpmg.F64), t, nc, n)
        e = np.pad(uc.astype(np.longdouble), ((0, 0), (1, 1), (1, 1)), mode="wrap")
    else:
        op = tpmg.PanelOperator(nx, ny, nz, 1e-4, 1.0, 1e-3, nlevels=2)
        tpmg.panel_prolongate(op.op, 2, dev(uc, tpmg.F64), t, nc, n)
        e = np.pad(uc.astype(np.longdouble), ((0, 0), (1, 1), (1, 1)))
    exact = uf.astype(np.longdouble)
    c, ldx = e[:, 1:-1, 1:-1], {0: e[:, 1:-1, :-2], 1: e[:, 1:-1, 2:]}
    for b, y in ((0, slice(None, -2)), (1, slice(2, None))):
        for a, x in ((0, slice(None, -2)), (1, slice(2, None))):
            exact[:, b::2, a::2] += (9 * c + 3 * ldx[a] + 3 * e[:, y, 1:-1] + e[:, y, x]) / 16
    rms = lambda v: float(np.sqrt(np.mean((v.astype(np.longdouble) - exact) ** 2)))
    got = t.cpu().numpy().reshape(nz, ny, nx)
    assert rms(got) < 1.25 * rms(exact.astype(np.float64)), (rms(got), rms(exact.astype(np.float64)))
    op.close()
