"""FP64 handles whose large bonds run from digit splits on the tensor cores:
the autotuner's choices leave the bits of a sweep as they are."""
import numpy as np
import pytest

pytestmark = pytest.mark.gpu

DIMS, CHI = [64, 3, 3, 64], [64, 64, 64]   # the middle bond: 192 x 192, l = 74


def _state(rng):
    c = [1] + CHI + [1]
    gam = [rng.standard_normal((DIMS[s], c[s], c[s + 1], 2)).view(np.complex128)[..., 0] / 8.0 for s in range(4)]
    lam = []
    for x in CHI:
        v = np.exp(-np.arange(x) / 8.0)
        lam.append(v / np.linalg.norm(v))
    return gam, lam


def _swept(B, **kw):
    rng = np.random.default_rng(4)
    sim = B.Tebd(4, 2, 0, 10, 1, 0, d_site=DIMS, chi_bond=CHI, **kw)
    try:
        gam, lam = _state(rng)
        sim.set_mps(gam, lam)
        sim.set_gates(1, [np.linalg.qr(rng.standard_normal((DIMS[b] * DIMS[b + 1],) * 2))[0].astype(complex)
                          for b in range(3)])
        info = B.tebd_wave_info(sim.h, 1, 0)
        sim.step_odd()
        g, l = sim.get_mps()
        return info, g, l
    finally:
        sim.close()


def test_the_autotuner_does_not_choose_between_two_arithmetics(lib):
    from paper_1504_00992_gb300 import binding as B
    _, g0, l0 = _swept(B)
    info, g1, l1 = _swept(B, autotune=1)
    assert not info["fused"] and info["tune_ms"] == [0.0, 0.0]   # the two were not timed against each other
    for a, b in zip(list(g0) + list(l0), list(g1) + list(l1)):
        assert np.array_equal(a, b)
