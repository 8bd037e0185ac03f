"""Inner products with few vectors and updates by few: the kernels for 2, 4, 6, 8 and 16
vectors at their edges, FP32 vectors of one value per load (odd length, 8-byte aligned)
included.  The bounds are those of the other tests of these calls: 1e-5 of sum |a_i b_i| in
FP32 (a hundred roundings of 2^-24), 2^-40 of it in double-float arithmetic and FP64.  A
vector's inner product has the same bits whatever the number of vectors beside it."""
import numpy as np
import pytest

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("prec", ["f32", "f32-8", "f64-ds", "f64"])
@pytest.mark.parametrize("n", [33, 3070, 300002])
def test_few_vectors(n, prec):
    import torch
    from paper_1509_06865_gb300 import PREC_F32, PREC_F64, Context
    f32 = prec.startswith("f32")
    dt, P, bound = (np.complex64, PREC_F32, 1e-5) if f32 else (np.complex128, PREC_F64, 2.0 ** -40)
    shift = 1 if prec == "f32-8" else 0   # vectors that start 8 bytes off a 16-byte boundary
    rng = np.random.default_rng(n)
    K = 17
    X = (rng.standard_normal((K, n + 3)) + 1j * rng.standard_normal((K, n + 3))).astype(dt)
    X = np.ascontiguousarray(X[:, :(n + 3) // 2 * 2])
    y = (rng.standard_normal(n) + 1j * rng.standard_normal(n)).astype(dt)
    c = rng.standard_normal(K) + 1j * rng.standard_normal(K)
    ctx = Context((4, 4, 4, 4))
    ctx.set_params(n_tv=8, agg=(2, 2, 2, 2), sap_block=(2, 2, 2, 2), precision=1, blas_ds=0 if prec == "f64" else 1)
    Xd = torch.from_numpy(X).cuda()
    p = [v.data_ptr() + 8 * shift for v in Xd]
    X64, y64 = X[:, shift:shift + n].astype(np.complex128), y.astype(np.complex128)
    alone = None
    for k in (1, 2, 3, 4, 5, 6, 7, 8, 9, 11, 17):
        yd = torch.from_numpy(y).cuda()
        torch.cuda.synchronize()
        d = ctx.multidot_dev(p[:k], yd.data_ptr(), n, P)
        assert np.all(np.abs(d - X64[:k].conj() @ y64) <= bound * (np.abs(X64[:k]) @ np.abs(y64))), k
        alone = d[0] if alone is None else alone
        assert d[0] == alone, k
        ctx.multi_axpy_dev(p[:k], c[:k], yd.data_ptr(), n, P)
        want, size = y64 + c[:k] @ X64[:k], np.abs(y64) + np.abs(c[:k]) @ np.abs(X64[:k])
        assert np.all(np.abs(yd.cpu().numpy() - want) <= bound * size), k
    ctx.close()
