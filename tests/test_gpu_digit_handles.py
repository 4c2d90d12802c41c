"""FP64 handles whose large bonds run from digit splits on the tensor cores:
the autotuner's choices leave the bits of a sweep as they are, and the reverse
pass recomputes a recorded sweep with the bits it had."""
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


def _gradient(B, fused):
    """Two recorded sweeps over a state whose middle Schmidt values lie in
    pairs with squares 1e-8 apart; the cotangents of the first sweep's gate."""
    rng = np.random.default_rng(8)

    def haar(m, n):
        return np.linalg.qr(rng.standard_normal((m, n, 2)).view(np.complex128)[..., 0])[0]

    lam = [np.exp(-np.arange(64) / 20.0) for _ in range(3)]
    lam[1] = np.repeat(np.exp(-np.arange(32) / 40.0), 2)
    lam = [x / np.linalg.norm(x) for x in lam]
    lam[1][1::2] = np.sqrt(lam[1][1::2] ** 2 - 1e-8)
    U, Vh = haar(192, 64).reshape(3, 64, 64), haar(192, 64).T.reshape(64, 3, 64).transpose(1, 0, 2)
    gam = [haar(64, 64)[:, None, :], U / lam[0][None, :, None], Vh / lam[2][None, None, :], haar(64, 64)[:, :, None]]
    sim = B.Tebd(4, 2, 0, 10, 1, 0, d_site=DIMS, chi_bond=CHI, fused=fused)
    try:
        sim.set_mps(gam, lam)
        gates = [haar(192, 192), np.kron(haar(3, 3), haar(3, 3)), haar(192, 192)]
        sim.set_gates(0, gates)
        sim.set_gates(1, gates)
        op = haar(3, 3)
        sim.record(True)
        sim.step_odd()
        sim.step_even()
        return sim.backward(1, op + op.conj().T)[1][1]
    finally:
        sim.close()


def test_the_reverse_pass_keeps_the_gauge_of_the_forward_sweep(lib):
    """A recomputation that differs from the forward sweep by rounding turns a
    pair's vectors by ~1e-16 / 1e-8, and the adjoint of the SVD divides that
    by 1e-8 again: an error of order one.  With the same bits 1e-16 / 1e-8
    remains, as on the FP64 pipe; the bar is 1e-5 of the largest cotangent."""
    from paper_1504_00992_gb300 import binding as B
    a, b = _gradient(B, 0), _gradient(B, -1)
    assert np.abs(a - b).max() <= 1e-5 * np.abs(b).max()
