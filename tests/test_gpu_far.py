"""Atoms so far outside an open box that FP32 coordinates no longer tell
neighbours apart, while FP64 ones do: the FP32 screens of the list build and of
the FP64 passes must leave every such pair to FP64.  The gas lies across a
value where FP32 changes to the next number, as the list build sees it (x
itself) and as the passes do (less a cell's centre), so that close atoms round
to different numbers.  Lists are integers and equal the oracle's.  Forces:
coordinates relative to a cell's centre are rounded at the size of the
position, 2^-53 |x| an atom and axis or 2^-52 |x| a pair, and a force changes
by less than 10 times its size over an Angstrom (atoms of the gas are 1
Angstrom apart at least): 10 sqrt(2) 2^-52 2^30 = 3.4e-6 at the largest
distance that is tested, below the bound of 1e-5; a missed pair is an error of order 1."""
import numpy as np
import pytest

import oracle as O
from paper_2405_07898_gb300 import binding, inputs as I

pytestmark = pytest.mark.gpu

R_LIST = 4.8


def gas(e, n=500, seed=5):
    rng = np.random.default_rng(seed)
    box = R_LIST * 1.03 * np.array([3.0, 3.0, 3.0])
    keep = []
    while len(keep) < n:
        x = rng.random(3) * box
        if all(((x - y) ** 2).sum() > 1.0 for y in keep):
            keep.append(x)
    pos = np.array(keep)
    edge = 2.0**e + 2.0 ** (e - 24)  # half-way between two FP32 numbers
    pos[: n // 2, 0] += edge - 1.2
    pos[: n // 2, 1] -= edge + 6.0
    return I.System(box=box, pos=pos, vel=None, types=np.zeros(n, np.int32),
                    pot=I.johnson_potential(I.BCC_TA_LIKE, 200), open_axes=3)


@pytest.mark.parametrize("persistent", ["off", "on"])
@pytest.mark.parametrize("e", [23, 26, 28, 30, 39])
def test_lists_and_forces(e, persistent):
    s = gas(e)
    w = O.wrap(s.pos, s.box, s.open_axes)
    want_off, want_js = O.neighbors_cells(w, s.box, R_LIST, s.open_axes)
    for lanes in (1, 8):
        with binding.MD(s, precision="fp64", persistent=persistent, lanes_per_atom=lanes) as md:
            for again in range(2):
                off, js = md.neighbors()
                np.testing.assert_array_equal(off, want_off)
                np.testing.assert_array_equal(js, want_js)
                if e <= 30:
                    F = O.eam_eval(O.Potential(s.pot), w, s.box, s.types, open_axes=s.open_axes)[2]
                    f = md.forces()
                    assert np.linalg.norm(f - F) <= 1e-5 * np.linalg.norm(F)
                if not again:
                    md.set_state(s.pos)  # by the other form of the list build
    with binding.MD(s, precision="mixed", persistent=persistent) as md:
        off, js = md.neighbors()
        np.testing.assert_array_equal(off, want_off)
        np.testing.assert_array_equal(js, want_js)
