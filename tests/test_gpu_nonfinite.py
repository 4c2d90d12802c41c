"""A non-finite entry of a chain's state in a bond contracted on the tensor
cores from digit splits (m, n >= 128, chi_m >= 32): the sweep reports it, in
every form, for gates applied in place (d_l d_r < 32) and gates that are a
GEMM, as the contraction in FP64 multiply-adds does by carrying the NaN into
theta and its norm."""
import numpy as np
import pytest


pytestmark = pytest.mark.gpu


def _chain(d, rng):
    """Sites 64, d, d, 64 with bonds of 64: the middle bond is 64 d x 64 d."""
    dims, chi = [64, d, d, 64], [1, 64, 64, 64, 1]
    gam = [rng.standard_normal((dims[s], chi[s], chi[s + 1], 2)).view(np.complex128)[..., 0] / 8.0 for s in range(4)]
    lam = []
    for b in range(3):
        v = np.exp(-np.arange(chi[b + 1]) / 8.0)
        lam.append(v / np.linalg.norm(v))
    return dims, chi[1:-1], gam, lam


@pytest.mark.parametrize("form", ["fp64", "tf32", "bf16"])
@pytest.mark.parametrize("d", [3, 6])
@pytest.mark.parametrize("where", ["left", "right", "lambda", "inf", "none"])
def test_a_nonfinite_state_is_reported(lib, form, d, where):
    from paper_1504_00992_gb300 import binding as B
    prec = {"fp64": B.TEBD_PREC_FP64, "tf32": B.TEBD_PREC_TF32, "bf16": B.TEBD_PREC_BF16}[form]
    dims, chi, gam, lam = _chain(d, np.random.default_rng(d))
    if where == "left":
        gam[1][d - 1, 5, 17] = np.nan
    elif where == "right":
        gam[2][0, 33, 60] = complex(0.0, np.nan)
    elif where == "inf":
        gam[1][0, 63, 0] = np.inf
    elif where == "lambda":
        lam[1][40] = np.nan
    sim = B.Tebd(4, 2, 0, 10, 1, 0, d_site=dims, chi_bond=chi, precision=prec)
    try:
        sim.set_mps(gam, lam)
        eye = [np.eye(dims[b] * dims[b + 1], dtype=np.complex128) for b in range(3)]
        sim.set_gates(1, eye)
        sim.step_odd()
        op = np.eye(64)
        if where == "none":
            assert np.isfinite(sim.expect(0, op))
        else:
            with pytest.raises(B.TebdError) as e:
                sim.expect(0, op)
            assert e.value.code == B.TEBD_ENUMERIC
    finally:
        sim.close()
