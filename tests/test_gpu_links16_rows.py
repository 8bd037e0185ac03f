"""The coarse operator with 16-bit links on one vector where a row starts on 4, 8 and 16
bytes (odd N_tv, even, a multiple of 4), against the oracle with the bounds of the other
16-bit links: 2e-2 for BF16, 3e-3 for IEEE half."""
import numpy as np
import pytest

import synth
from oracle import dirac, mg
from tests.gpu_util import norm_rel_err

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("links,tol", [("bf16", 2e-2), ("f16", 3e-3)])
@pytest.mark.parametrize("ntv", [3, 9, 10, 12, 24])
def test_one_vector(ntv, links, tol):
    from paper_1509_06865_gb300 import LINKS_BF16, LINKS_F16, Context
    dims, agg = (8, 8, 4, 4), (4, 4, 2, 2)
    U = synth.gauge_field(dims, 0.25, 311)
    op = dirac.WilsonClover(U, -0.1, 1.5)
    W = synth.uniform_vectors(dims, ntv, 17)
    P = mg.Interpolation(W, agg)
    C = mg.CoarseOperator(mg.coarse_operator(op, P), P.cdims, P.ntv)
    ctx = Context(dims)
    ctx.set_params(m0=-0.1, csw=1.5, agg=agg, sap_block=(4, 4, 2, 2), n_tv=ntv, precision=1,
                   coarse_links=LINKS_BF16 if links == "bf16" else LINKS_F16)
    ctx.load_gauge(U)
    ctx.set_test_vectors(W)
    x = P.restrict(synth.gaussian_vectors(dims, 1, 6)[0])
    assert norm_rel_err(ctx.coarse_apply(x, 0.03), C.apply(x, 0.03)) < tol
    if links == "f16":   # a launch a vector
        X = np.array([x, 2 * x])
        Y = ctx.coarse_apply_nrhs(X, 0.03)
        assert norm_rel_err(Y[0], C.apply(x, 0.03)) < tol and np.array_equal(Y[1], 2 * Y[0])
    ctx.close()
