"""A SAP block of more than 256 sites is an accepted parameter, the operator works with it, and
whatever sweeps over it returns MGEIG_ECUDA, in both precisions; the context goes on."""
import numpy as np
import pytest

import synth

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("precision", [0, 1], ids=["fp64", "mixed"])
@pytest.mark.parametrize("sap", [(4, 4, 4, 8), (4, 4, 8, 8)], ids=["512 sites", "1024 sites"])
def test_large_blocks(sap, precision):
    from paper_1509_06865_gb300 import Context, MgeigError, check_params
    from paper_1509_06865_gb300._lib import ECUDA
    dims = (8, 8, 16, 16)
    kw = dict(agg=(4, 4, 4, 4), n_tv=4, precision=precision, outer_restart=2)
    assert check_params(dims, sap_block=sap, **kw) == 0
    ctx = Context(dims)
    ctx.set_params(sap_block=sap, **kw)
    ctx.load_gauge(synth.gauge_field(dims, 0.25, 311))
    x = synth.gaussian_vectors(dims, 1, 8)[0]
    y = ctx.apply(x[None], 0.05)
    for call in (lambda: ctx.sap(x, 0 * x, 0.05, cycles=1), lambda: ctx.setup(5)):
        with pytest.raises(MgeigError) as e:
            call()
        assert e.value.code == ECUDA
    assert np.array_equal(ctx.apply(x[None], 0.05), y)
    ctx.set_params(sap_block=(4, 4, 4, 4), **kw)
    assert np.all(np.isfinite(ctx.sap(x, 0 * x, 0.05, cycles=1)))
    ctx.close()
