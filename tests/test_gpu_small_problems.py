"""Small FP64 problems: the QR with the matrix in shared memory, on clusters of
eight to one CTAs by the size of the batch (bit for bit the same), and its
truncations against what the input was made of, at sizes around its rows per
lane, its register blocks and its smallest and largest matrices.

Bars, set before the first run: a theta of exact rank k comes back to 1e-12 of
its norm (FP64 QRs, products and Jacobi, each a few l eps with l <= 60), the
factors are orthonormal to 1e-12."""
import numpy as np
import pytest

from paper_1504_00992_gb300 import inputs as I
from tests.gpu_util import rrsvd_device, truncated

pytestmark = pytest.mark.gpu

SIZES = [
    (2, 2, 1, 1, 1),       # the smallest: l = 2
    (17, 16, 4, 2, 2),
    (33, 31, 10, 3, 1),    # one past a register block of rows
    (64, 64, 32, 10, 2),
    (65, 96, 20, 11, 0),
    (96, 80, 12, 6, 2),
    (129, 60, 40, 19, 1),  # columns of Q in memory on one side
    (1200, 50, 5, 3, 1),   # tall and narrow
    (240, 250, 46, 5, 1),  # l = 51: the largest matrices that fit
    (270, 250, 46, 5, 1),  # one side past it
]


def _run(B, theta, k, p, q, batch):
    plan = B.rrsvd_plan_create(theta.shape[0], theta.shape[1], k, p, q, batch, B.TEBD_PREC_FP64, 3)
    try:
        return rrsvd_device(B, plan, np.repeat(theta[None], batch, axis=0))
    finally:
        B.rrsvd_plan_destroy(plan)


@pytest.mark.parametrize("m,n,k,p,q", SIZES)
def test_small_truncations(lib, m, n, k, p, q):
    from paper_1504_00992_gb300 import binding as B
    sig = np.where(np.arange(min(m, n)) < k, np.exp(-np.arange(min(m, n)) / max(2.0, 0.2 * k)), 0.0)
    theta = I.haar_theta(m, n, sig, seed=m + n)
    first = None
    for batch in (1, 20, 40, 160):     # clusters of up to eight, four and two CTAs, and one CTA
        out = _run(B, theta, k, p, q, batch)
        one = {x: out[x][0] for x in ("sigma", "U", "Vh", "w", "rank")}
        if first is None:
            first = one
        for x in one:
            assert np.array_equal(one[x], first[x]), (x, batch)
    d = truncated(first["U"], first["sigma"], first["Vh"]) - theta
    assert np.linalg.norm(d) <= 1e-12 * np.linalg.norm(theta)
    r = int(first["rank"])
    assert np.abs(first["U"][:, :r].conj().T @ first["U"][:, :r] - np.eye(r)).max() <= 1e-12
    assert np.abs(first["Vh"][:r] @ first["Vh"][:r].conj().T - np.eye(r)).max() <= 1e-12
