"""The mixed forms' FP32 QRs (Cholesky QR from digits, Householder for what it
gives up), their small SVD's FP32 sweeps on one CTA and on a cluster, at the
edges of their sizes and on inputs whose sketches are singular; the theta
contraction from digits with the gate applied in place, and the rebuild on
many CTAs, against the same update on the FP64 pipe.

Bars, set before the first run.  Truncations: errors (singular values,
Frobenius) at most 1.05 of the FP64 form's on the same Omega plus 1e-8 s_1,
factors orthonormal to 1e-11; exactly rank-deficient inputs come back to 3e-6
of their norm (the mixed forms' bars).  Bond updates: both sides are FP64-level,
so Schmidt values agree to 1e-11, w to 1e-12, observables to 1e-10."""
import numpy as np
import pytest

from paper_1504_00992_gb300 import inputs as I
from tests.gpu_util import rrsvd_device, truncated

pytestmark = pytest.mark.gpu


def _run(B, theta, k, p, q, prec):
    batch, m, n = theta.shape
    plan = B.rrsvd_plan_create(m, n, k, p, q, batch, prec, 11)
    try:
        return rrsvd_device(B, plan, theta)
    finally:
        B.rrsvd_plan_destroy(plan)


def _orthonormal(out, t):
    r = int(out["rank"][t])
    U, Vh = out["U"][t][:, :r], out["Vh"][t][:r]
    assert np.abs(U.conj().T @ U - np.eye(r)).max() <= 1e-11
    assert np.abs(Vh @ Vh.conj().T - np.eye(r)).max() <= 1e-11


@pytest.mark.parametrize("m,n,k,p,q", [
    (256, 256, 38, 10, 1),     # l = 48: the smallest of the rule
    (257, 700, 60, 5, 2),      # one past a row block and a column tile
    (2100, 300, 64, 64, 1),    # two whole column tiles
    (330, 420, 150, 10, 1),    # l = 160: the widest on one CTA
    (420, 330, 150, 11, 1),    # l = 161: a cluster
    (700, 650, 220, 42, 2),    # l = 262
    (400, 330, 300, 20, 1),    # l = 320: the widest of the cluster form
    (400, 340, 315, 10, 0),    # l = 325: the Jacobi kernels alone; no power round
])
def test_mixed_form_over_its_sizes(lib, m, n, k, p, q):
    from paper_1504_00992_gb300 import binding as B
    sig = I.exp_spectrum(min(m, n), max(4.0, 0.15 * k))
    theta = np.stack([I.synthetic_theta(m, n, sig, seed=70 + t) for t in range(2)])
    a = _run(B, theta, k, p, q, B.TEBD_PREC_TF32)
    b = _run(B, theta, k, p, q, B.TEBD_PREC_FP64)
    for t in range(2):
        ea, eb = (np.abs(x["sigma"][t] - sig[:k]).max() for x in (a, b))
        assert ea <= 1.05 * eb + 1e-8
        fa, fb = (np.linalg.norm(truncated(x["U"][t], x["sigma"][t], x["Vh"][t]) - theta[t]) for x in (a, b))
        assert fa <= 1.05 * fb + 1e-8
        _orthonormal(a, t)


@pytest.mark.parametrize("l", [60, 180])
@pytest.mark.parametrize("kind", ["one_entry", "one_row", "rank_3", "graded"])
def test_mixed_form_on_singular_sketches(lib, kind, l):
    from paper_1504_00992_gb300 import binding as B
    m, n, k = 300, 280, l - 10
    if kind == "one_entry":
        theta = np.zeros((m, n), dtype=np.complex128)
        theta[7, 11] = 0.5 + 0.25j
    elif kind == "one_row":
        theta = np.zeros((m, n), dtype=np.complex128)
        theta[5] = np.exp(1j * np.arange(n)) / np.sqrt(n)
    elif kind == "rank_3":
        theta = I.haar_theta(m, n, np.array([1.0, 0.5, 1e-3]), seed=3)
    else:
        theta = I.haar_theta(m, n, np.exp(-0.6 * np.arange(n)), seed=4)
    out = _run(B, theta[None], k, 10, 2, B.TEBD_PREC_TF32)
    d = truncated(out["U"][0], out["sigma"][0], out["Vh"][0]) - theta
    assert np.linalg.norm(d) <= 3e-6 * np.linalg.norm(theta)
    assert np.abs(out["sigma"][0][0] - np.linalg.norm(theta, 2)) <= 1e-8


@pytest.mark.parametrize("dims,caps,bond", [
    ([64, 3, 3, 64], [64, 70, 64], 1),
    ([64, 4, 2, 2, 4, 64], [64, 100, 33, 97, 64], 2),   # the smallest contraction depth but one
    ([40, 5, 6, 33], [40, 40, 33], 1),    # 30 physical indices: the largest gate applied in place
    ([40, 5, 5, 39], [40, 50, 39], 1),
])
def test_contraction_from_digits(lib, dims, caps, bond):
    from paper_1504_00992_gb300 import binding as B
    rng = np.random.default_rng(sum(dims))
    chi = [1] + caps + [1]
    gam = [(rng.standard_normal((d, chi[s], chi[s + 1])) + 1j * rng.standard_normal((d, chi[s], chi[s + 1])))
           / np.sqrt(2.0 * d * chi[s]) for s, d in enumerate(dims)]
    lam = [np.exp(-np.arange(c) / max(1.0, c / 6.0)) for c in caps]
    lam = [x / np.linalg.norm(x) for x in lam]
    gates = [I.random_unitary(a * b, rng) for a, b in zip(dims, dims[1:])]
    op = rng.standard_normal((dims[bond], dims[bond]))
    got = []
    for fused in (0, -1):              # digits, the FP64 pipe
        sim = B.Tebd(len(dims), 2, 0, 10, 2, 9, d_site=dims, chi_bond=caps, fused=fused)
        try:
            sim.set_mps(gam, lam)
            sim.set_gates(bond % 2, gates)
            (sim.step_odd if bond % 2 else sim.step_even)()
            got.append((sim.get_lambda(bond), sim.discarded_weight()[0], sim.expect(bond, op)))
        finally:
            sim.close()
    (la, wa, ea), (lb, wb, eb) = got
    r = min(len(la), len(lb))
    assert np.abs(la[:r] - lb[:r]).max() <= 1e-11
    assert abs(wa - wb) <= 1e-12
    assert abs(ea - eb) <= 1e-10 * np.linalg.norm(op, 2)
