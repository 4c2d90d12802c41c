"""The FP64 form's products and QRs from digit splits on the tensor cores (the
path of problems with l >= 40, m, n >= 128) against the same truncation on the
FP64 pipe (GEMM tiles forced), on the same theta and Omega, at the edges of
the rule, of the 128 x 32 output tiles and of the 16- and 64-deep k steps, on
graded, degenerate, rank-deficient and scaled inputs; one-site expectation
values spread over many CTAs against NumPy.

Bars, set before the first run: both paths carry FP64-level errors, so
singular values agree to 1e-12 s_1, the truncated theta to 1e-10 of its norm
and w to 1e-12 (the project's bars for two FP64 codes on the same Omega)."""
import numpy as np
import pytest

from paper_1504_00992_gb300 import inputs as I
from tests.gpu_util import rrsvd_device, truncated

pytestmark = pytest.mark.gpu


def _both(B, theta, k, p, q, seed=5):
    batch, m, n = theta.shape
    out = []
    for tiles in (0, 32):
        plan = B.rrsvd_plan_create(m, n, k, p, q, batch, B.TEBD_PREC_FP64, seed)
        try:
            if tiles:
                B.rrsvd_plan_set_tuning(plan, {"tiles": [tiles] * 6})
            out.append(rrsvd_device(B, plan, theta))
        finally:
            B.rrsvd_plan_destroy(plan)
    return out


def _agree(theta, a, b):
    for t in range(theta.shape[0]):
        s1, nrm = b["sigma"][t][0], np.linalg.norm(theta[t])
        r = min(a["rank"][t], b["rank"][t])
        assert abs(int(a["rank"][t]) - int(b["rank"][t])) <= 2      # values at the 1e-14 cutoff
        assert np.abs(a["sigma"][t][:r] - b["sigma"][t][:r]).max() <= 1e-12 * s1
        d = truncated(a["U"][t], a["sigma"][t], a["Vh"][t]) - truncated(b["U"][t], b["sigma"][t], b["Vh"][t])
        assert np.linalg.norm(d) <= 1e-10 * nrm
        assert abs(a["w"][t] - b["w"][t]) <= 1e-12
        # orthonormal factors over the kept rank
        U, Vh = a["U"][t][:, :r], a["Vh"][t][:r]
        assert np.abs(U.conj().T @ U - np.eye(r)).max() <= 1e-12
        assert np.abs(Vh @ Vh.conj().T - np.eye(r)).max() <= 1e-12


@pytest.mark.parametrize("m,n,k,p,q,batch", [
    (128, 128, 30, 10, 2, 3),     # the smallest sizes of the rule
    (129, 193, 32, 10, 1, 2),     # one past a row tile and a k step
    (517, 131, 45, 13, 2, 2),     # odd sizes, several row tiles
    (640, 256, 118, 22, 1, 2),    # l = 140: five column tiles
    (300, 420, 150, 10, 1, 2),    # l = 160: the widest factor in shared memory
    (350, 420, 190, 10, 1, 2),    # l = 200: factors in global memory
    (1030, 2049, 60, 20, 0, 1),   # no power round: the sketch's basis is the last one
])
def test_digit_products_agree_with_the_fp64_pipe(lib, m, n, k, p, q, batch):
    from paper_1504_00992_gb300 import binding as B
    sig = I.exp_spectrum(min(m, n), max(4.0, 0.15 * k))
    theta = np.stack([I.synthetic_theta(m, n, sig, seed=300 + t) for t in range(batch)])
    _agree(theta, *_both(B, theta, k, p, q))


@pytest.mark.parametrize("kind", ["graded", "degenerate", "low_rank", "tiny", "huge"])
def test_digit_products_on_hard_inputs(lib, kind):
    from paper_1504_00992_gb300 import binding as B
    m, n, k, p, q = 260, 200, 50, 14, 2
    if kind == "graded":            # down to rounding level: the sketch is numerically singular
        sig = np.exp(-0.6 * np.arange(n))
    elif kind == "degenerate":      # quadruplets of equal values, the cut between two of them
        sig = np.exp(-0.25 * (np.arange(n) // 4))
        k = 48
    elif kind == "low_rank":        # exact rank below k
        sig = np.where(np.arange(n) < 20, np.exp(-0.2 * np.arange(n)), 0.0)
    else:
        sig = I.exp_spectrum(n, 8.0) * (1e-40 if kind == "tiny" else 1e40)
    theta = np.stack([I.haar_theta(m, n, sig, seed=40 + t) for t in range(2)])
    a, b = _both(B, theta, k, p, q)
    if kind == "low_rank":          # beyond the rank both keep rounding-level values or none
        for t in range(2):
            assert np.abs(a["sigma"][t] - b["sigma"][t]).max() <= 1e-12 * b["sigma"][t][0]
            d = truncated(a["U"][t], a["sigma"][t], a["Vh"][t]) - theta[t]
            assert np.linalg.norm(d) <= 1e-10 * np.linalg.norm(theta[t])
    else:
        _agree(theta, a, b)


@pytest.mark.parametrize("d,chi", [(3, 12), (5, 40), (2, 129)])
def test_expectation_over_many_ctas(lib, d, chi):
    from paper_1504_00992_gb300 import binding as B
    rng = np.random.default_rng(d)
    dims, caps = [64, d, 64], [min(64, chi), min(64, chi)]
    cl, cr = caps
    sh = [(64, 1, cl), (d, cl, cr), (64, cr, 1)]
    gam = [rng.standard_normal(s) + 1j * rng.standard_normal(s) for s in sh]
    lam = []
    for c in caps:
        v = np.exp(-np.arange(c) / 9.0)
        lam.append(v / np.linalg.norm(v))
    op = rng.standard_normal((d, d)) + 1j * rng.standard_normal((d, d))
    sim = B.Tebd(3, 2, 0, 2, 1, 0, d_site=dims, chi_bond=caps)
    try:
        sim.set_mps(gam, lam)
        got = sim.expect(1, op)
    finally:
        sim.close()
    w = (lam[0] ** 2)[:, None] * (lam[1] ** 2)[None, :]
    terms = np.einsum("iac,ij,jac,ac->ac", gam[1].conj(), op, gam[1], w)
    assert abs(got - terms.sum()) <= 1e-13 * np.abs(terms).sum() * d
