"""mgeig_get_launch_count counts every kernel of a call: one more Schwarz cycle is two
more sweeps, one launch each, in FP64 (a launch as clusters) as in FP32."""
import pytest

import synth

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("precision", [0, 1], ids=["fp64", "mixed"])
def test_schwarz_sweeps_are_counted(precision):
    from paper_1509_06865_gb300 import Context
    dims = (8, 4, 4, 4)
    ctx = Context(dims)
    ctx.set_params(agg=(2, 2, 2, 2), sap_block=(2, 2, 2, 2), n_tv=4, precision=precision)
    ctx.load_gauge(synth.gauge_field(dims, 0.25, 311))
    b, z = synth.gaussian_vectors(dims, 2, 8)
    took = []
    for cycles in (1, 4):
        n = ctx.launch_count()
        ctx.sap(b, z, 0.05, cycles=cycles)
        took.append(ctx.launch_count() - n)
    ctx.close()
    assert took[1] - took[0] == 3 * 2
