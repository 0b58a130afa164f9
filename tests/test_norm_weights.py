"""CPU: the norm gain of one real-time line solve whose weights are rounded to float,
averaged over a smooth spectrum, in the three forms that real time runs in: the
folded Thomas sweeps, the centred TMA sweeps and the two-tail solve.  All three
move the norm by about 8e-7 kappa^2 (rms over kappa), of either sign, and which is
the better one at a given kappa is chance."""
import numpy as np


def _f32(z):
    return complex(np.float32(z.real), np.float32(z.imag))


THETA = np.linspace(-np.pi, np.pi, 2001)
WEIGHT = np.exp(-(THETA / 0.25) ** 2)
WEIGHT /= WEIGHT.sum()


def _gains(kappa):
    """Mean of |G(theta)|^2 - 1: folded, centred, two-tail (no rotation)."""
    left, right = np.exp(-1j * THETA), np.exp(1j * THETA)
    kap = 1j * kappa
    a0, off = 1 + 2 * kap, -kap
    m = 1 / a0
    for _ in range(300):
        m = 1 / (a0 - off * off * m)
    tail = -m * off                      # the multiplier of either recurrence
    al = be = _f32(tail)
    poles = (1 - al * left) * (1 - be * right)
    # psi'_p = x_p, x = d + be x_{p+1}, d = (1 + a0) psi + am psi_- + ap psi_+ + al d_-
    explicit = 1 + _f32(m * (1 - 2 * kap) - 1) + _f32(m * kap) * (left + right)
    folded = explicit / poles
    # psi' = 2 y - psi, the weight m2 - 2 rounded
    centred = (2 + _f32(2 * m - 2)) / poles - 1
    # psi' = psi + gc psi + g2 (f + b)
    g = 1 / (a0 - 2 * off * off * m)
    tails = al * left / (1 - al * left) + be * right / (1 - be * right)
    two = 1 + _f32(2 * g - 2) + _f32(2 * g) * tails
    return [float((WEIGHT * (np.abs(v) ** 2 - 1)).sum()) for v in (folded, centred, two)]


def test_rounded_weights_move_the_norm_alike():
    for lo, hi in ((0.001, 0.005), (0.008, 0.04), (0.04, 0.12)):
        kappa = np.exp(np.linspace(np.log(lo), np.log(hi), 200))
        gain = np.array([_gains(k) for k in kappa]) / kappa[:, None] ** 2
        rms = np.sqrt((gain**2).mean(0))
        assert (rms > 6e-7).all() and (rms < 1e-6).all(), rms
        assert (np.abs(gain).max(0) < 6.4e-6).all()
        # either sign, and neither of the Thomas forms always the better one
        assert (gain.min(0) < 0).all() and (gain.max(0) > 0).all()
        better = (np.abs(gain[:, 1]) < np.abs(gain[:, 0])).mean()
        assert 0.3 < better < 0.7, better
