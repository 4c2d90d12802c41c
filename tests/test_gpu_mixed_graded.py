"""The mixed forms on matrices whose rows are graded: every row of U carries
single precision relative to itself.

theta = diag(2^-30 .. 1) X with X of a decaying spectrum.  The FP32 chain
(products, QR, triangular products) works row by row, so a row of U has errors
of some 2^-24 relative to its own norm, times s_1 / s_10 = 4.5 for the ten
leading vectors compared and the few operations a row passes: of the order of
1e-6 to 1e-5.  The bar is 1e-4; rows rounded on the scale of the largest one
were off by 0.3."""
import numpy as np
import pytest

from tests.gpu_util import rrsvd_device

pytestmark = pytest.mark.gpu


def _graded(m, n, seed):
    rng = np.random.default_rng(seed)

    def haar(a, b):
        return np.linalg.qr(rng.standard_normal((a, b)) + 1j * rng.standard_normal((a, b)))[0]

    r = min(m, n)
    X = (haar(m, r) * np.exp(-np.arange(r) / 6.0)) @ haar(n, r).conj().T
    return X * (2.0 ** -np.linspace(0, 30, m))[:, None]


@pytest.mark.parametrize("form", ["tf32", "bf16"])
@pytest.mark.parametrize("m,n,k,p,products", [
    (400, 400, 40, 20, 0),     # the digit products
    (1201, 400, 40, 20, 0),
    (400, 400, 40, 20, 2),     # the double-float products
    (120, 100, 30, 10, 0),     # below the size rule of the digit products
])
def test_small_rows_of_U_keep_their_bits(lib, form, m, n, k, p, products):
    from paper_1504_00992_gb300 import binding as B
    A = _graded(m, n, m + n)
    U, s, _ = np.linalg.svd(A, full_matrices=False)
    plan = B.rrsvd_plan_create(m, n, k, p, 2, 1, {"tf32": B.TEBD_PREC_TF32, "bf16": B.TEBD_PREC_BF16}[form], 3)
    try:
        if products:
            B.rrsvd_plan_set_tuning(plan, {"products": products})
        out = rrsvd_device(B, plan, A[None])
    finally:
        B.rrsvd_plan_destroy(plan)
    u = out["U"][0]
    g = u.conj().T @ u
    assert np.abs(g - np.eye(k)).max() <= 1e-12       # Q = Q_f (I + D) to FP64
    assert np.abs(out["sigma"][0] - s[:k]).max() <= 1e-10 * s[0]
    ph = np.einsum("ij,ij->j", U[:, :10].conj(), u[:, :10])
    ref = U[:, :10] * (ph / np.abs(ph))
    err = np.linalg.norm(u[:, :10] - ref, axis=1) / np.linalg.norm(ref, axis=1)
    assert err.max() <= 1e-4
