"""The forms that the hot kernels take by size and alignment, at the edges of each: whole-column tiles in shared
memory (Smooth, line solve, Residual + RestrictSmooth, the fused Tridiag of CG), columns in chunks of planes, the
pointwise Residual, 16-byte Prolongate and conversions, the marching SpMV of CG, the batched solver's tiles and the
solver loop on the device. Forms that replace another bit for bit are compared with it, the others with the FP64
oracle under the tolerances of gpu_common."""
import numpy as np
import pytest
import torch

import oracle
from gpu_common import PREC_IDS, PRECS, TOL, dev, host, make_problem, oracle_levels, rel, tol_inverse
from paper_1402_3545_gb300 import tpmg, workloads

pytestmark = pytest.mark.gpu
RHO = 0.8


def fields(shape, prec, seed, count=2):
    rng = np.random.default_rng(seed)
    return [dev(rng.standard_normal(shape), prec) for _ in range(count)]


def operator(nx, ny, nz, lam, square=True, nlevels=2):
    """lam None: lambda^2 varies by column; square: cx == cy"""
    l2 = workloads.lambda2_varying(nx, ny) if lam is None else lam
    h = 1.0 / max(nx, ny)
    return tpmg.Operator(nx, ny, nz, 1e-2, h, h if square else 0.75 * h, 1.0 / nz, l2, nlevels=nlevels)


# above 4096 columns, so that no small-level kernel takes them: rows of 128, 64 and 32 FP32 columns a tile, and
# what has FP32 or no tiles only; below and at the rules' plane counts, and one plane more than a tile holds
@pytest.mark.parametrize("lam", [None, 1e3], ids=["varying", "constant"])
@pytest.mark.parametrize("square", [True, False], ids=["square", "oblong"])
@pytest.mark.parametrize("shape", [(128, 34, 1), (128, 34, 2), (64, 66, 15), (64, 66, 16), (96, 44, 17), (32, 132, 16),
                                   (128, 34, 127), (64, 66, 128), (128, 34, 129)], ids=lambda s: "x".join(map(str, s)))
@pytest.mark.parametrize("prec", [tpmg.F32, tpmg.DW], ids=["f32", "dw"])
def test_tile_smooth_equals_the_marching_one(prec, shape, square, lam):
    nx, ny, nz = shape
    op = operator(nx, ny, nz, lam, square)
    n = nx * ny * nz
    u, f = fields((nz, ny, nx), prec, nx + nz)

    def run(variant, norm):
        tpmg.set_variant(op.op, prec, 2, variant)
        o, nrm = torch.empty_like(u), torch.zeros(1, dtype=torch.float64, device="cuda")
        tpmg.smooth(op.op, 2, prec, RHO, u, f, o, n, norm_out=nrm if norm else None)
        return host(o), host(nrm)[0]

    for norm in (False, True):
        (a, na), (b, nb) = run(0, norm), run(3, norm)
        assert np.array_equal(a, b), (norm, np.abs(a - b).max())
        assert abs(na - nb) <= 1e-6 * nb
    op.close()


@pytest.mark.parametrize("lam", [None, 1e3], ids=["varying", "constant"])
@pytest.mark.parametrize("shape", [(128, 34, 15), (128, 34, 16), (64, 66, 17), (96, 44, 128), (48, 88, 33)],
                         ids=lambda s: "x".join(map(str, s)))
@pytest.mark.parametrize("prec", [tpmg.F32, tpmg.DW], ids=["f32", "dw"])
def test_tile_line_solve_and_tridiag_match_oracle(prec, shape, lam):
    nx, ny, nz = shape
    p = make_problem(nx, ny, nz, lam=lam)
    op = tpmg.Operator.from_problem(p, nlevels=2)
    cx, cy, v = oracle.problem_coefficients(p)
    tol = tol_inverse(prec, cx, cy, v)
    r, q = fields((nz, ny, nx), prec, nz)
    r0, q0 = (host(t).reshape(nz, ny, nx) for t in (r, q))
    x = torch.empty_like(r)
    tpmg.line_solve(op.op, 2, prec, r, x, p.n)
    assert rel(host(x), oracle.line_solve(r0, cx, cy, v)) < tol
    alpha = 0.37
    z, rr, rz = torch.empty_like(r), *(torch.zeros(1, dtype=torch.float64, device="cuda") for _ in range(2))
    tpmg.cg_fused_tridiag(op.op, prec, alpha, r, q, z, rr, rz, p.n)
    r1 = r0 - alpha * q0
    z1 = oracle.line_solve(r1, cx, cy, v)
    assert rel(host(r), r1) < TOL[prec] and rel(host(z), z1) < tol
    assert abs(host(rr)[0] - (r1 * r1).sum()) < max(TOL[prec], 1e-7) * (r1 * r1).sum()
    assert abs(host(rz)[0] - (r1 * z1).sum()) < max(tol, 1e-7) * abs((r1 * z1).sum())
    op.close()


@pytest.mark.parametrize("lam", [None, 1e3], ids=["varying", "constant"])
@pytest.mark.parametrize("square", [True, False], ids=["square", "oblong"])
@pytest.mark.parametrize("shape", [(256, 66, 1), (256, 66, 15), (256, 66, 16), (128, 130, 33), (192, 88, 128),
                                   (128, 130, 256)], ids=lambda s: "x".join(map(str, s)))
@pytest.mark.parametrize("prec", [tpmg.F32, tpmg.DW], ids=["f32", "dw"])
def test_restrict_tile_equals_the_two_kernels(prec, shape, square, lam):
    nx, ny, nz = shape
    op = operator(nx, ny, nz, lam, square)
    n = nx * ny * nz
    u, f = fields((nz, ny, nx), prec, nz)
    got = []
    for fuse in (True, False):
        tpmg.set_fusion(op.op, fuse)
        fc, uc = (torch.empty(n // 4, dtype=u.dtype, device="cuda") for _ in range(2))
        tpmg.residual_restrict_smooth(op.op, 1, prec, RHO, u, f, fc, uc, n, n // 4)
        got.append((host(fc), host(uc)))
    assert np.array_equal(got[0][0], got[1][0])
    assert np.array_equal(got[0][1], got[1][1])
    op.close()


# chunk sizes change above 64 and 128 planes and end at 256; 8, 4 or 2 columns a block by the level's size; whole and
# part-filled rows of chunks. The rule's edges: cyclic reduction up to 8, 32 or 12 planes and on 256 columns above 64;
# 10240 and 16384 columns with tiles, 4 and 24 planes without
@pytest.mark.parametrize("shape", [(2, 2, 64), (6, 4, 65), (34, 10, 128), (66, 62, 129), (34, 10, 256), (66, 62, 1),
                                   (182, 182, 5), (130, 130, 24), (130, 130, 25), (16, 16, 9), (16, 16, 65), (32, 32, 32),
                                   (32, 32, 33), (64, 64, 12), (64, 64, 13), (128, 80, 9), (128, 128, 24), (128, 128, 25)],
                         ids=lambda s: "x".join(map(str, s)))
def test_chunked_columns_match_oracle(shape):
    nx, ny, nz = shape
    p = make_problem(nx, ny, nz)
    op = tpmg.Operator.from_problem(p, nlevels=2)
    lv = oracle_levels(*oracle.problem_coefficients(p), 2)
    tol = tol_inverse(tpmg.F64, *lv[2])
    u, f = fields((nz, ny, nx), tpmg.F64, nz)
    uh, fh = (host(t).reshape(nz, ny, nx) for t in (u, f))
    ref, rn = oracle.smooth(uh, fh, *lv[2], RHO), np.linalg.norm(oracle.residual(uh, fh, *lv[2]))
    for norm in (None, torch.zeros(1, dtype=torch.float64, device="cuda")):
        o = torch.empty_like(u)
        tpmg.smooth(op.op, 2, tpmg.F64, RHO, u, f, o, p.n, norm_out=norm)
        assert rel(host(o), ref) < tol
    assert abs(host(norm)[0] - rn) < 1e-7 * rn
    tpmg.line_solve(op.op, 2, tpmg.F64, f, o, p.n)
    assert rel(host(o), oracle.line_solve(fh, *lv[2])) < tol
    fc, uc = (torch.empty(p.n // 4, dtype=torch.float64, device="cuda") for _ in range(2))
    tpmg.restrict_smooth(op.op, 1, tpmg.F64, RHO, f, fc, uc, p.n, p.n // 4)
    assert rel(host(fc), oracle.restrict(fh)) < TOL[tpmg.F64]
    assert rel(host(uc), RHO * oracle.line_solve(oracle.restrict(fh), *lv[1])) < tol
    op.close()


@pytest.mark.parametrize("shape", [(96, 44, 1), (96, 44, 9), (160, 204, 3), (182, 182, 5), (190, 34, 17)],
                         ids=lambda s: "x".join(map(str, s)))
@pytest.mark.parametrize("prec", PRECS, ids=PREC_IDS)
def test_pointwise_residual_matches_oracle(prec, shape):
    nx, ny, nz = shape
    p = make_problem(nx, ny, nz)
    op = tpmg.Operator.from_problem(p, nlevels=2)
    u, f = fields((nz, ny, nx), prec, nz)
    r, nrm = torch.empty_like(u), torch.zeros(1, dtype=torch.float64, device="cuda")
    tpmg.residual(op.op, 2, prec, u, f, r, p.n, norm_out=nrm)
    ref = oracle.residual(host(u).reshape(nz, ny, nx), host(f).reshape(nz, ny, nx), *oracle.problem_coefficients(p))
    assert rel(host(r), ref) < TOL[prec]
    assert abs(host(nrm)[0] - np.linalg.norm(ref)) < max(TOL[prec], 1e-7) * np.linalg.norm(ref)
    op.close()


def offset_copy(t, by):
    """t's values at an address that is `by` elements off a 16-byte boundary"""
    b = torch.empty(t.numel() + 4, dtype=t.dtype, device="cuda")[by:by + t.numel()]
    b.copy_(t.reshape(-1))
    return b


@pytest.mark.parametrize("shape", [(130, 66, 3), (132, 64, 2), (256, 34, 5)], ids=lambda s: "x".join(map(str, s)))
@pytest.mark.parametrize("prec", [tpmg.F64, tpmg.F32], ids=["f64", "f32"])
def test_prolongate_forms_agree(prec, shape):
    """16-byte segments, one coarse column a thread where nxc is odd, and any alignment: in FP32 the same bits."""
    nx, ny, nz = shape
    op = operator(nx, ny, nz, 1e3)
    n = nx * ny * nz
    uf, = fields((nz, ny, nx), prec, 3, 1)
    uc, = fields((nz, ny // 2, nx // 2), prec, 4, 1)
    a, b = uf.clone().reshape(-1), offset_copy(uf, 1)
    for t in (a, b):
        tpmg.prolongate(op.op, 2, prec, uc, t, n // 4, n)
    ref = oracle.prolongate_add(host(uc).reshape(nz, ny // 2, nx // 2), host(uf).reshape(nz, ny, nx))
    assert rel(host(a), ref) < TOL[prec] and rel(host(b), ref) < TOL[prec]
    if prec == tpmg.F32:
        assert torch.equal(a, b)
    op.close()


@pytest.mark.parametrize("by", [0, 1])
def test_conversion_alignment_and_edges(by):
    """Double-word units' conversions (omega^2 = 0, so A = I) on both alignments: exponents at the limits of the
    integer form, ties of the rounding, zeros and values whose low part leaves the float range."""
    nx, ny, nz = 6, 2, 3
    rng = np.random.default_rng(5)
    e = np.array([-74, -75, 126, -73, 0, -126, -149, 125])
    x = np.ldexp(1.0 + rng.random(36), np.resize(e, 36)) * np.resize([1.0, -1.0], 36)
    x[:6] = [0.0, -0.0, np.ldexp(1 + 2.0 ** -24, -74), np.ldexp(1 + 3 * 2.0 ** -24, 100), 2.0 ** -74, 1.0]
    op = tpmg.Operator(nx, ny, nz, 0.0, 1.0 / nx, 1.0 / ny, 1.0 / nz, 1.0, 1)
    y = offset_copy(torch.empty(36, dtype=torch.float64, device="cuda"), by)
    tpmg.apply_A(op.op, 1, tpmg.DW, offset_copy(dev(x, tpmg.F64), by), y, 36)
    with np.errstate(under="ignore"):
        hi = x.astype(np.float32)
        lo = (x - hi.astype(np.float64)).astype(np.float32)
    assert np.array_equal(host(y), hi.astype(np.float64) + lo.astype(np.float64))
    op.close()


@pytest.mark.parametrize("shape", [(2, 2, 1), (6, 4, 15), (64, 10, 16), (34, 18, 17), (130, 8, 33)],
                         ids=lambda s: "x".join(map(str, s)))
@pytest.mark.parametrize("prec", PRECS, ids=PREC_IDS)
def test_cg_spmv_matches_oracle(prec, shape):
    nx, ny, nz = shape
    p = make_problem(nx, ny, nz)
    op = tpmg.Operator.from_problem(p, nlevels=1)
    u, pp, z, q = fields((nz, ny, nx), prec, nz, 4)
    uh, ph, zh, qh = (host(t).reshape(nz, ny, nx) for t in (u, pp, z, q))
    sg = torch.zeros(1, dtype=torch.float64, device="cuda")
    alpha, beta = 0.3, -0.6
    tpmg.cg_fused_spmv(op.op, prec, alpha, beta, u, pp, z, q, sg, p.n)
    p1 = zh + beta * ph
    q1 = oracle.apply_A(zh, *oracle.problem_coefficients(p)) + beta * qh
    assert rel(host(u), uh + alpha * ph) < TOL[prec] and rel(host(pp), p1) < TOL[prec] and rel(host(q), q1) < TOL[prec]
    assert abs(host(sg)[0] - (p1 * q1).sum()) <= max(TOL[prec], 1e-7) * np.linalg.norm(p1) * np.linalg.norm(q1)
    op.close()


@pytest.mark.parametrize("what", ["max_iter", "zero_rhs", "nonfinite", "converges"])
@pytest.mark.parametrize("solve", ["mg", "cg"])
def test_loop_on_the_device_equals_plain_launches(solve, what):
    p = make_problem(32, 16, 16)
    op = tpmg.Operator.from_problem(p, nlevels=2)
    f = dev(p.rhs(), tpmg.F64)
    if what == "zero_rhs":
        f.zero_()
    if what == "nonfinite":
        f.view(-1)[5] = float("nan")
    got = []
    for graph in (1, 0):
        u = torch.zeros_like(f)
        prm = tpmg.default_params(prec=tpmg.F64, tol=1e-8, max_iter=3 if what == "max_iter" else 200, use_graph=graph)
        run = tpmg.mg_solve if solve == "mg" else tpmg.cg_solve
        try:
            info = run(op.op, prm, f, u, p.n)
            got.append((info["iters"], info["converged"], list(info["history"]), host(u)))
        except tpmg.TpmgError as e:
            got.append((e.status,))
    assert len(got[0]) == len(got[1])
    for a, b in zip(*got):
        assert np.array_equal(a, b, equal_nan=True)
    op.close()


@pytest.mark.parametrize("shapes", [[(48, 40, 17), (96, 36, 16), (64, 64, 1)], [(64, 64, 200), (8, 8, 256), (32, 16, 140)],
                                    [(256, 64, 33), (64, 128, 150), (192, 64, 20)]], ids=["columns", "long", "tiles"])
@pytest.mark.parametrize("square", [True, False], ids=["square", "oblong"])
@pytest.mark.parametrize("lam", [None, 1e3], ids=["varying", "constant"])
def test_batched_forms_reach_the_single_solves(shapes, square, lam):
    """32-column and vector tiles in one batch: what the single mixed solver reaches, to its tolerance."""
    ops = [operator(nx, ny, nz, lam, square, 2 if nx % 4 or ny % 4 else 3) for nx, ny, nz in shapes]
    fs = [fields((nz, ny, nx), tpmg.F64, nz, 1)[0] for nx, ny, nz in shapes]
    us = [torch.zeros_like(f) for f in fs]
    prm = tpmg.default_params(prec=tpmg.MIXED, tol=1e-6, max_iter=60)
    res = tpmg.mg_solve_batched([o.op for o in ops], prm, fs, us)
    for o, f, u, r in zip(ops, fs, us, res["problems"]):
        u1 = torch.zeros_like(f)
        single = tpmg.mg_solve(o.op, prm, f, u1, f.numel())
        assert abs(single["iters"] - r["iters"]) <= 1 and single["converged"] == r["converged"]
        r1, r2 = (torch.empty_like(f) for _ in range(2))
        tpmg.residual(o.op, o.L, tpmg.F64, u, f, r1, f.numel())
        tpmg.residual(o.op, o.L, tpmg.F64, u1, f, r2, f.numel())
        if r["converged"]:  # Eq. 10 with the FP64 residual
            assert r1.norm() < 1.01e-6 * f.norm() and r2.norm() < 1.01e-6 * f.norm()
    for o in ops:
        o.close()
