"""The contraction of a bond from digit splits does not depend on how a term's
size is shared between the two Gammas: with column g of Gamma_l multiplied by
2^t_g and row g of Gamma_r by 2^-t_g, theta is the same number by number (the
FP64 multiply-adds give the same bits), and so must be the sweep's result, bit
for bit, in every form and for both kinds of gates."""
import numpy as np
import pytest

pytestmark = pytest.mark.gpu


def _swept(B, prec, d, t):
    rng = np.random.default_rng(20 + d)
    dims, chi = [64, d, d, 64], [64, 64, 64]
    c = [1] + chi + [1]
    gam = [rng.standard_normal((dims[s], c[s], c[s + 1], 2)).view(np.complex128)[..., 0] / 8.0 for s in range(4)]
    lam = []
    for x in chi:
        v = np.exp(-np.arange(x) / 3.0)
        lam.append(v / np.linalg.norm(v))
    gam[1] = gam[1] * 2.0 ** t
    gam[2] = gam[2] * 2.0 ** -t[:, None]
    sim = B.Tebd(4, 2, 0, 10, 1, 0, d_site=dims, chi_bond=chi, precision=prec)
    try:
        sim.set_mps(gam, lam)
        sim.set_gates(1, [np.linalg.qr(rng.standard_normal((dims[b] * dims[b + 1],) * 2))[0].astype(complex)
                          for b in range(3)])
        sim.step_odd()
        g, l = sim.get_mps()
        return list(g) + list(l)
    finally:
        sim.close()


@pytest.mark.parametrize("form", ["fp64", "tf32", "bf16"])
@pytest.mark.parametrize("d", [3, 6])
@pytest.mark.parametrize("kind", ["random", "steep"])
def test_theta_does_not_depend_on_the_gauge(lib, form, d, kind):
    from paper_1504_00992_gb300 import binding as B
    prec = {"fp64": B.TEBD_PREC_FP64, "tf32": B.TEBD_PREC_TF32, "bf16": B.TEBD_PREC_BF16}[form]
    t = np.random.default_rng(d).integers(-20, 21, 64) if kind == "random" else np.arange(64) // 2
    a, b = _swept(B, prec, d, np.zeros(64)), _swept(B, prec, d, t)
    for i, (x, y) in enumerate(zip(a, b)):
        assert np.array_equal(x, y), i
