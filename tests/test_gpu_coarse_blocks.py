"""The coarse GMRES on few blocks of many rows, which small lattices reach through
coarse_blocks: its matvec in several passes and chunks of sites, basis slices in global
memory (all of them at the restarts of 30 below, but for the smallest blocks), one lane a
row in the sums over vectors, more rows than 1024 and more sites than the staged neighbour
table holds, FP64 rows in several runs.  Against the oracle with the bounds that the
two-grid cycles have elsewhere: 1e-9 in FP64, 1e-4 in FP32.  The FP32 sums have an order
that does not depend on where vectors and parts of sums are kept, so FP32 results agree
bit for bit whatever the restart length decides about that."""
import functools

import numpy as np
import pytest

import synth
from oracle import dirac, mg
from tests.gpu_util import norm_rel_err

pytestmark = pytest.mark.gpu

SHAPES = {
    "256 sites of 6 rows": dict(dims=(8, 8, 8, 8), agg=(2, 2, 2, 2), sap=(4, 4, 4, 4), ntv=3),
    "128 sites of 20 rows": dict(dims=(8, 8, 8, 4), agg=(2, 2, 2, 2), sap=(4, 4, 4, 2), ntv=10),
    "16 sites of 40 rows": dict(dims=(8, 8, 8, 8), agg=(4, 4, 4, 4), sap=(4, 4, 4, 4), ntv=20),
    "16 sites of 48 rows": dict(dims=(6, 6, 6, 6), agg=(3, 3, 3, 3), sap=(3, 3, 3, 3), ntv=24),
}
PHYS = dict(m0=-0.1, csw=1.5, bc=(1, 1, 1, -1))
SIGMA = 0.05


@functools.lru_cache(maxsize=None)
def parts(name):
    s = SHAPES[name]
    U = synth.gauge_field(s["dims"], 0.25, 311)
    op = dirac.WilsonClover(U, PHYS["m0"], PHYS["csw"], bc=PHYS["bc"])
    return U, op, synth.uniform_vectors(s["dims"], s["ntv"], 17), synth.gaussian_vectors(s["dims"], 1, 12)[0]


@functools.lru_cache(maxsize=None)
def oracle_cycle(name, deflate, restart, maxiter):
    s = SHAPES[name]
    U, op, W, r = parts(name)
    B = mg.TwoGrid(op, W, dict(mg.DEFAULT_PARAMS, agg=s["agg"], sap_block=s["sap"], ntv=s["ntv"], smoother="sap",
                               coarse_deflate=bool(deflate), coarse_tol=0.0, coarse_maxiter=maxiter,
                               coarse_restart=restart, sap_cycles=1, sap_mr_iters=2))
    return B(r, SIGMA)


def cycle(name, **kw):
    from paper_1509_06865_gb300 import Context
    s = SHAPES[name]
    U, op, W, r = parts(name)
    ctx = Context(s["dims"])
    ctx.set_params(agg=s["agg"], sap_block=s["sap"], n_tv=s["ntv"], sap_cycles=1, sap_mr_iters=2,
                   **dict(PHYS, coarse_tol=0.0, **kw) if "coarse_tol" not in kw else dict(PHYS, **kw))
    ctx.load_gauge(U)
    ctx.set_test_vectors(W)
    z = ctx.mg_cycle(r, SIGMA)
    ctx.close()
    return z


@pytest.mark.parametrize("prec,tol", [(0, 1e-9), (1, 1e-4)], ids=["fp64", "mixed"])
@pytest.mark.parametrize("deflate,restart", [(1, 4), (1, 30), (0, 30)], ids=["restart 4", "restart 30", "plain"])
@pytest.mark.parametrize("blocks", [1, 2, 3])
@pytest.mark.parametrize("name", list(SHAPES))
def test_few_blocks(name, blocks, deflate, restart, prec, tol):
    z = cycle(name, precision=prec, coarse_blocks=blocks, coarse_deflate=deflate, coarse_restart=restart, coarse_maxiter=7)
    assert norm_rel_err(z, oracle_cycle(name, deflate, restart, 7)) < tol


@pytest.mark.parametrize("links", ["level", "bf16", "f16"])
@pytest.mark.parametrize("blocks", [1, 3])
@pytest.mark.parametrize("name", list(SHAPES))
def test_bits_do_not_depend_on_where_vectors_are_kept(name, blocks, links):
    from paper_1509_06865_gb300 import LINKS_BF16, LINKS_F16, LINKS_LEVEL
    kw = dict(precision=1, coarse_blocks=blocks, coarse_maxiter=4,
              coarse_links={"level": LINKS_LEVEL, "bf16": LINKS_BF16, "f16": LINKS_F16}[links])
    assert np.array_equal(cycle(name, coarse_restart=4, **kw), cycle(name, coarse_restart=30, **kw))


@pytest.mark.parametrize("links", ["bf16", "f16"])
@pytest.mark.parametrize("name", list(SHAPES))
def test_few_blocks_16_bit_links(name, links):
    """The same links on as many blocks as there are rows for (128 each): FP32 roundings apart."""
    from paper_1509_06865_gb300 import LINKS_BF16, LINKS_F16
    kw = dict(precision=1, coarse_maxiter=7, coarse_restart=30, coarse_links=LINKS_BF16 if links == "bf16" else LINKS_F16)
    many = cycle(name, **kw)
    for blocks in (1, 2):
        assert norm_rel_err(cycle(name, coarse_blocks=blocks, **kw), many) < 1e-4


def test_no_room_for_parts():
    """384 rows of 48 a site and a basis of 31: what is left of the shared memory takes the neighbour vectors
    of one site (3.4 KB) and no parts of sums, with a basis of 20 both.  The solve stops in less than 20 steps."""
    name = "16 sites of 48 rows"
    kw = dict(precision=1, coarse_blocks=2, coarse_restart=31)
    assert np.array_equal(cycle(name, coarse_maxiter=33, coarse_tol=0.1, **kw),
                          cycle(name, coarse_maxiter=20, coarse_tol=0.1, **kw))
