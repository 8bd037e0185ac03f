"""The kernels whose work is cut by size, at the sizes where the cuts can go wrong
(one warp, warps that are not full, remainders of eight columns, the largest
N_tv, ragged last CTAs), against the oracle: the coarse apply of many vectors, SAP
on clusters of CTAs, the coarse GMRES inside a two-grid cycle, the many
right-hand-side stencil, the tensor-core coarse apply with 4-byte fragments, and
inner products and updates.  The bounds are those of the same operations in
test_gpu_mg.py, test_gpu_links16.py, test_gpu_operator.py and test_gpu_blas.py; for
FP32 vectors 1e-5 of sum |a_i b_i|, a hundred roundings of 2^-24 times sqrt(n) of
the at most 4099 terms a sum has here."""
import functools

import numpy as np
import pytest

import synth
from oracle import dirac, mg
from tests.gpu_util import norm_rel_err, rel_err

pytestmark = pytest.mark.gpu

SHAPES = {
    # SAP blocks of one warp, n2 = 6 (less than one residue of eight columns)
    "ntv3": dict(dims=(8, 4, 4, 4), agg=(2, 2, 2, 2), sap=(4, 2, 2, 2), ntv=3),
    # two warps a SAP block, n2 = 20 (two and a half residues)
    "ntv10": dict(dims=(8, 8, 4, 4), agg=(4, 2, 2, 2), sap=(4, 4, 2, 2), ntv=10),
    # 81 sites: the third warp is not full; n2 = 48, the largest
    "ntv24": dict(dims=(6, 6, 6, 6), agg=(3, 3, 3, 3), sap=(3, 3, 3, 3), ntv=24),
    # eight warps a SAP block, n2 = 24
    "ntv12": dict(dims=(8, 8, 8, 8), agg=(4, 4, 4, 4), sap=(4, 4, 4, 4), ntv=12),
}
PHYS = dict(m0=-0.1, csw=1.5, bc=(1, 1, 1, -1))


@functools.lru_cache(maxsize=None)
def oracle_parts(name):
    s = SHAPES[name]
    U = synth.gauge_field(s["dims"], 0.25, 311)
    op = dirac.WilsonClover(U, PHYS["m0"], PHYS["csw"], bc=PHYS["bc"])
    W = synth.uniform_vectors(s["dims"], s["ntv"], 17)
    P = mg.Interpolation(W, s["agg"])
    C = mg.CoarseOperator(mg.coarse_operator(op, P), P.cdims, P.ntv)
    return U, op, W, P, C


def make(name, precision, **kw):
    from paper_1509_06865_gb300 import Context
    s = SHAPES[name]
    ctx = Context(s["dims"])
    ctx.set_params(agg=s["agg"], sap_block=s["sap"], n_tv=s["ntv"], precision=precision, **PHYS, **kw)
    ctx.load_gauge(oracle_parts(name)[0])
    return ctx


@pytest.mark.parametrize("prec,tol", [(0, 1e-12), (1, 1e-5)], ids=["fp64", "mixed"])
@pytest.mark.parametrize("name", list(SHAPES))
def test_coarse_apply_many(name, prec, tol):
    U, op, W, P, C = oracle_parts(name)
    ctx = make(name, prec)
    ctx.set_test_vectors(W)
    X = np.array([P.restrict(x) for x in synth.gaussian_vectors(SHAPES[name]["dims"], 16, 5)])
    for nrhs in (1, 3, 4, 5, 8, 9, 16):
        Y = ctx.coarse_apply_nrhs(X[:nrhs], 0.07)
        for r in range(nrhs):
            assert rel_err(Y[r], C.apply(X[r], 0.07)) < tol, (nrhs, r)
    ctx.close()


@pytest.mark.parametrize("prec,tol", [(0, 1e-11), (1, 2e-5)], ids=["fp64", "mixed"])
@pytest.mark.parametrize("name", list(SHAPES))
def test_sap_block_shapes(name, prec, tol):
    U, op, W, P, C = oracle_parts(name)
    s = SHAPES[name]
    ctx = make(name, prec, sap_mr_iters=3)
    b, z0 = synth.gaussian_vectors(s["dims"], 2, 8)
    got = ctx.sap(b, 0.1 * z0, 0.05, cycles=2)
    assert norm_rel_err(got, mg.SAP(op, s["sap"]).smooth(b, 0.1 * z0, 0.05, 2, 3)) < tol
    ctx.close()


@pytest.mark.parametrize("dims,sap", [((16, 8, 8, 8), (2, 2, 2, 2)), ((16, 16, 8, 8), (2, 2, 2, 2)),
                                      ((12, 12, 12, 6), (3, 3, 3, 1)), ((16, 8, 16, 16), (4, 4, 4, 2))],
                         ids=["256 x 16 sites", "512 x 16 sites", "192 x 27 sites", "128 x 128 sites"])
def test_sap_fp64_many_blocks(dims, sap):
    """Blocks a colour on both sides of the line between the two FP64 forms on 152 SMs, warps of them not full."""
    from paper_1509_06865_gb300 import FP64, Context
    U = synth.gauge_field(dims, 0.25, 311)
    op = dirac.WilsonClover(U, PHYS["m0"], PHYS["csw"], bc=PHYS["bc"])
    ctx = Context(dims)
    ctx.set_params(agg=sap, sap_block=sap, n_tv=2, precision=FP64, sap_mr_iters=3, outer_restart=1, **PHYS)
    ctx.load_gauge(U)
    b, z0 = synth.gaussian_vectors(dims, 2, 8)
    got = ctx.sap(b, 0.1 * z0, 0.05, cycles=1)
    assert norm_rel_err(got, mg.SAP(op, sap).smooth(b, 0.1 * z0, 0.05, 1, 3)) < 1e-11
    ctx.close()


@pytest.mark.parametrize("prec,tol", [(0, 1e-9), (1, 1e-4)], ids=["fp64", "mixed"])
@pytest.mark.parametrize("deflate", [1, 0], ids=["deflated", "plain"])
@pytest.mark.parametrize("name", list(SHAPES))
def test_two_grid_cycle_shapes(name, deflate, prec, tol):
    U, op, W, P, C = oracle_parts(name)
    s = SHAPES[name]
    kw = dict(coarse_tol=0.0, coarse_maxiter=7, coarse_restart=4, sap_cycles=1, sap_mr_iters=2)
    B = mg.TwoGrid(op, W, dict(mg.DEFAULT_PARAMS, agg=s["agg"], sap_block=s["sap"], ntv=s["ntv"], smoother="sap",
                               coarse_deflate=bool(deflate), **kw))
    ctx = make(name, prec, coarse_deflate=deflate, **kw)
    ctx.set_test_vectors(W)
    r = synth.gaussian_vectors(s["dims"], 1, 12)[0]
    assert norm_rel_err(ctx.mg_cycle(r, 0.05), B(r, 0.05)) < tol
    ctx.close()


@pytest.mark.parametrize("nrhs", [1, 4, 5, 13])
def test_tensor_core_apply_rows_off_16_bytes(nrhs):
    """n2 = 20: a link row is 40 bytes."""
    from paper_1509_06865_gb300 import LINKS_BF16
    U, op, W, P, C = oracle_parts("ntv10")
    ctx = make("ntv10", 1, coarse_links=LINKS_BF16)
    ctx.set_test_vectors(W)
    X = np.array([P.restrict(x) for x in synth.gaussian_vectors(SHAPES["ntv10"]["dims"], nrhs, 6)])
    Y = ctx.coarse_apply_nrhs(X, 0.03)
    for r in range(nrhs):
        assert norm_rel_err(Y[r], C.apply(X[r], 0.03)) < 2e-2, r
    ctx.close()


@pytest.mark.parametrize("dims", [(5, 3, 4, 7), (16, 8, 4, 5), (24, 24, 24, 2), (32, 16, 32, 2)],
                         ids=["420 sites", "4 CTAs a timeslice", "runs of 54 CTAs", "runs of 64 CTAs"])
@pytest.mark.parametrize("nrhs", [2, 5])
def test_stencil_many_fields_ragged(dims, nrhs):
    from paper_1509_06865_gb300 import OP_D, OP_Q, PREC_F32, Context
    U = synth.gauge_field(dims, 0.3, 41)
    op = dirac.WilsonClover(U, 0.0, 1.0)
    x = synth.gaussian_vectors(dims, nrhs, 9)
    ctx = Context(dims)
    ctx.load_gauge(U)
    for which in (OP_Q, OP_D):
        y = ctx.apply(x, 0.04, which, PREC_F32)
        for r in range(nrhs):
            want = op.Q_sigma(x[r], 0.04) if which == OP_Q else op.D_sigma(x[r], 0.04)
            assert norm_rel_err(y[r], want) < 1e-6
    ctx.close()


@pytest.mark.parametrize("prec", ["f32", "f64-ds", "f64"])
@pytest.mark.parametrize("n", [1, 31, 1024, 4099])
@pytest.mark.parametrize("k", [1, 9, 16, 17, 32])
def test_inner_products_and_updates(k, n, prec):
    import torch
    from paper_1509_06865_gb300 import PREC_F32, PREC_F64, Context
    dt = np.complex64 if prec == "f32" else np.complex128
    rng = np.random.default_rng(100 * k + n)
    X = (rng.standard_normal((k, n + n % 2)) + 1j * rng.standard_normal((k, n + n % 2))).astype(dt)
    y = (rng.standard_normal(n) + 1j * rng.standard_normal(n)).astype(dt)
    c = rng.standard_normal(k) + 1j * rng.standard_normal(k)
    ctx = Context((4, 4, 4, 4))
    ctx.set_params(n_tv=8, agg=(2, 2, 2, 2), sap_block=(2, 2, 2, 2), precision=1, blas_ds=0 if prec == "f64" else 1)
    Xd, yd = torch.from_numpy(X).cuda(), torch.from_numpy(y).cuda()
    torch.cuda.synchronize()
    p = [v.data_ptr() for v in Xd]
    P = PREC_F32 if prec == "f32" else PREC_F64
    bound = 1e-5 if prec == "f32" else 2.0 ** -40
    X64, y64 = X[:, :n].astype(np.complex128), y.astype(np.complex128)
    d = ctx.multidot_dev(p, yd.data_ptr(), n, P)
    assert np.all(np.abs(d - X64.conj() @ y64) <= bound * (np.abs(X64) @ np.abs(y64)))
    ctx.multi_axpy_dev(p, c, yd.data_ptr(), n, P)
    assert np.all(np.abs(yd.cpu().numpy() - (y64 + c @ X64)) <= bound * (np.abs(y64) + np.abs(c) @ np.abs(X64)))
    ctx.close()


@pytest.mark.parametrize("prec", [0, 1], ids=["fp64", "mixed"])
def test_solve_with_a_basis_of_more_vectors_than_a_launch_takes(prec):
    """FGMRES minimises the residual over its whole basis, so 100 steps without a restart end
    no further from the solution than 70.  sigma lies deep inside the spectrum, where the
    cycle is a poor preconditioner, and 1e-13 is out of reach."""
    name = "ntv3"
    U, op, W, P, C = oracle_parts(name)
    b = synth.gaussian_vectors(SHAPES[name]["dims"], 1, 23)[0]
    res = {}
    for steps in (70, 100):
        ctx = make(name, prec, outer_restart=100, outer_maxiter=steps)
        ctx.set_test_vectors(W)
        x, st = ctx.solve(b, 1.7, 1e-13)
        assert st["outer_iters"] == steps and not st["converged"]
        res[steps] = np.linalg.norm(b - op.Q_sigma(x, 1.7)) / np.linalg.norm(b)
        ctx.close()
    assert res[100] <= res[70] * (1 + 1e-6)


@pytest.mark.parametrize("prec,tol", [(0, 1e-12), (1, 1e-5)], ids=["fp64", "mixed"])
@pytest.mark.parametrize("ntv", [2, 10])
def test_restriction_cut_by_test_vectors(ntv, prec, tol):
    """256 aggregates: the test vectors go to several CTAs, 10 of them unevenly."""
    from paper_1509_06865_gb300 import Context
    dims, agg = (8, 8, 8, 8), (2, 2, 2, 2)
    W = synth.uniform_vectors(dims, ntv, 19)
    P = mg.Interpolation(W, agg)
    ctx = Context(dims)
    ctx.set_params(agg=agg, sap_block=(4, 4, 4, 4), n_tv=ntv, precision=prec, **PHYS)
    ctx.load_gauge(synth.gauge_field(dims, 0.25, 29))
    ctx.set_test_vectors(W)
    r = synth.gaussian_vectors(dims, 1, 3)[0]
    ec = P.restrict(r)
    assert rel_err(ctx.restrict(r), ec) < tol
    assert rel_err(ctx.prolong(ec), P.prolong(ec)) < tol
    ctx.close()
