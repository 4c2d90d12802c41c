"""Few tall bases the Cholesky QR gives up (steep spectra: B^H, or a sketch,
singular to rounding): the QRs of the last basis and of B^H then take the
many-CTA Householder form, not one CTA per matrix.

In the mixed form the QR of B^H is the only one of these, so a plan with the
many-CTA QR chosen outright must give the same bits.  In the FP64 form the
bars against the FP64 pipe are those of two FP64 codes on the same Omega:
1e-12 s_1, 1e-10 of theta's norm, 1e-12 for w."""
import numpy as np
import pytest

from paper_1504_00992_gb300 import inputs as I
from tests.gpu_util import rrsvd_device, truncated

pytestmark = pytest.mark.gpu


def _theta(m, n, rate, batch, seed):
    sig = np.exp(-rate * np.arange(min(m, n)))
    return np.stack([I.synthetic_theta(m, n, sig, seed=seed + t) for t in range(batch)])


def _run(B, theta, k, p, q, prec, tuning=None, profile=False):
    batch, m, n = theta.shape
    plan = B.rrsvd_plan_create(m, n, k, p, q, batch, prec, 9)
    try:
        if tuning:
            B.rrsvd_plan_set_tuning(plan, tuning)
        out = rrsvd_device(B, plan, theta)
        if profile:
            B.tebd_profiler_enable(True)
            try:
                B.tebd_profiler_reset()
                rrsvd_device(B, plan, theta)
                prof = B.tebd_profiler_read()
                out["kernels"] = {name: rec[1] for name, rec in prof.items()}
                out["ms"] = {name: rec[0] for name, rec in prof.items()}
            finally:
                B.tebd_profiler_enable(False)
        return out
    finally:
        B.rrsvd_plan_destroy(plan)


@pytest.mark.parametrize("m,n,k,p,q,batch", [
    (260, 1024, 40, 8, 0, 1),     # the fewest rows, the narrowest sketch
    (300, 1057, 50, 13, 1, 3),    # odd rows and columns: ragged row blocks, chunks and panels
    (400, 1600, 118, 10, 0, 2),   # four row chunks, eight panels
])
def test_mixed_form_keeps_the_bits_of_the_many_cta_qr(lib, m, n, k, p, q, batch):
    from paper_1504_00992_gb300 import binding as B
    theta = _theta(m, n, 0.8, batch, 60)
    a = _run(B, theta, k, p, q, B.TEBD_PREC_TF32, profile=True)
    b = _run(B, theta, k, p, q, B.TEBD_PREC_TF32, {"qrbh": 2})
    assert "k_qr" not in a["kernels"] and a["kernels"].get("k_qr[multi]") == 1
    for name in ("sigma", "U", "Vh", "w", "rank"):
        assert np.array_equal(a[name], b[name]), name


@pytest.mark.parametrize("m,n,k,p,q,batch", [(1100, 1040, 40, 10, 1, 2), (1030, 2049, 60, 20, 2, 1)])
def test_fp64_form_agrees_with_the_fp64_pipe(lib, m, n, k, p, q, batch):
    from paper_1504_00992_gb300 import binding as B
    theta = _theta(m, n, 0.8, batch, 80)
    a = _run(B, theta, k, p, q, B.TEBD_PREC_FP64, profile=True)
    b = _run(B, theta, k, p, q, B.TEBD_PREC_FP64, {"tiles": [32] * 6})
    assert a["kernels"].get("k_qr[multi]") == 2  # the last basis and B^H
    # no first or middle basis is left to one CTA: M l^2 16 flop at 8 GFLOP/s
    # would be 5 ms or more each, an empty launch is a few microseconds
    assert a["ms"]["k_qr"] < 0.2 * a["kernels"]["k_qr"]
    for t in range(batch):
        s1, nrm = b["sigma"][t][0], np.linalg.norm(theta[t])
        assert np.abs(a["sigma"][t] - b["sigma"][t]).max() <= 1e-12 * s1
        d = truncated(a["U"][t], a["sigma"][t], a["Vh"][t]) - truncated(b["U"][t], b["sigma"][t], b["Vh"][t])
        assert np.linalg.norm(d) <= 1e-10 * nrm
        assert abs(a["w"][t] - b["w"][t]) <= 1e-12
