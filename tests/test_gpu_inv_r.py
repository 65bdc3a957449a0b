"""1/r and r of the FP64 pair passes against exact values.  Two atoms at a
distance d along x that their coordinates hold exactly, f = 0, F = 0 and
phi(r) = r: the energy is r as the kernel has it and the force 1/r times d.
r^2 is rounded once (2^-53 relative, half of it in r); the series step adds
half a rounding of x y^2 (2^-54) and the final operation one (2^-53), so that r
is within 2^-52 of d, and 1/r likewise of 1/d; the force adds the rounding of
its product (2^-53).  2^-57 for the terms of higher order (the third-order
remainder is (5/16) e^3 at |e| < 2^-18)."""
import numpy as np
import pytest

from paper_2405_07898_gb300 import binding, inputs as I

pytestmark = pytest.mark.gpu

R_CUT = 4.0


def distances():
    rng = np.random.default_rng(36)
    d = [2.0**e * m for e in range(-18, 2) for m in (1.0, 1.0 + 2.0**-20, 1.5, 2.0 - 2.0**-20)]  # ends of binades
    d += [np.sqrt(2.0) * 2.0**e for e in range(-10, 2)]  # r^2 at the ends of its binades
    d += list(R_CUT - 2.0 ** -np.arange(3.0, 30.0))  # near the cutoff
    d += list(2.0 ** rng.uniform(-8.0, 2.0, 1200))
    d = np.round(np.array(d) * 2.0**48) / 2.0**48  # exact in the coordinates below
    return d[(d > 0) & (d < R_CUT)]


def test_r_and_its_reciprocal():
    line = I.Knots(0.0, R_CUT, np.array([0.0, R_CUT]), I.BC_CLAMPED, I.BC_CLAMPED, 1.0, 1.0)
    zero = I.Knots(0.0, R_CUT, np.zeros(2), I.BC_CLAMPED, I.BC_CLAMPED, 0.0, 0.0)
    pot = I.Potential(mass=np.array([1.0]), F=[zero], f=[zero], phi=[line], r_cut=R_CUT, skin=0.5)
    pos = np.array([[2.5, 4.0, 4.0], [3.5, 4.0, 4.0]])
    s = I.System(box=np.array([8.0, 8.0, 8.0]), pos=pos, vel=None, types=np.zeros(2, np.int32), pot=pot, open_axes=7)
    d = distances()
    r, f = np.empty_like(d), np.empty((len(d), 2, 3))
    with binding.MD(s, precision="fp64") as md:
        for k, x in enumerate(d):
            pos[1, 0] = pos[0, 0] + x
            assert pos[1, 0] - pos[0, 0] == x
            md.set_state(pos)
            r[k] = md.energy()[0]
            f[k] = md.forces()
    assert np.all(f[:, :, 1:] == 0.0) and np.all(f[:, 0, 0] == -f[:, 1, 0])
    assert np.abs(r / d - 1.0).max() <= 2.0**-52 * (1.0 + 2.0**-5) + 2.0**-53  # and the division here
    assert np.abs(f[:, 0, 0] - 1.0).max() <= 2.0**-52 + 2.0**-53 + 2.0**-57
