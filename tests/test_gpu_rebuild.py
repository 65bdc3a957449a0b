"""The list build against the oracle's exact lists, entry for entry, where its
runs of cells and groups of four candidates have edges: one to five cells on
an axis, periodic and open, a few atoms (groups that reach past the last
atom), crowded cells (runs longer than a mask), atoms at cell boundaries and
far outside an open box.  The lists are integers: equality, no tolerance."""
import numpy as np
import pytest

import oracle as O
from paper_2405_07898_gb300 import binding, inputs as I

pytestmark = pytest.mark.gpu

R_LIST = 4.8  # of the BCC potential


def gas(cells, open_axes, n, seed, far=0.0):
    rng = np.random.default_rng(seed)
    box = R_LIST * 1.03 * np.array(cells, dtype=np.float64)
    pos = rng.random((n, 3)) * box
    pos[: n // 8, 0] = np.round(pos[: n // 8, 0] / box[0] * cells[0]) * box[0] / cells[0]  # on cell boundaries
    if far:
        pos[: n // 2] += far * np.array([1.0, -1.0, 0.0])
    return I.System(box=box, pos=pos, vel=None, types=np.zeros(n, np.int32),
                    pot=I.johnson_potential(I.BCC_TA_LIKE, 200), open_axes=open_axes)


@pytest.mark.parametrize("precision", ["fp64", "mixed"])
@pytest.mark.parametrize("persistent", ["off", "on"])
@pytest.mark.parametrize("cells,open_axes,n", [
    ((3, 3, 3), 0, 1), ((3, 4, 5), 0, 3), ((3, 3, 3), 0, 257), ((5, 3, 4), 0, 1001),
    ((1, 3, 4), 1, 130), ((2, 1, 3), 3, 95), ((1, 1, 1), 7, 33), ((2, 5, 1), 5, 402), ((4, 2, 2), 6, 515),
    ((3, 3, 3), 0, 1900),  # about 70 atoms a cell: runs of more than 200 candidates
    ((40, 30, 33), 0, 40007),  # past the warp-per-atom build
])
def test_lists_equal_the_oracles(cells, open_axes, n, persistent, precision):
    s = gas(cells, open_axes, n, seed=n + open_axes)
    with binding.MD(s, precision=precision, persistent=persistent, lanes_per_atom=2) as md:
        check(md, s)
        if n > 200:  # again from the sorted order
            md.set_state(s.pos[::-1].copy())
            s.pos = s.pos[::-1].copy()
            check(md, s)


@pytest.mark.parametrize("far", [37.0, 5.0e4])
def test_far_outside_an_open_box(far):
    """FP64 lists stay exact however far outside an open box the atoms are."""
    s = gas((3, 3, 3), 3, 700, seed=5, far=far)
    with binding.MD(s, precision="fp64", persistent="off") as md:
        check(md, s)


def check(md, s):
    w = O.wrap(s.pos, s.box, s.open_axes)
    off, js = md.neighbors()
    want_off, want_js = O.neighbors_cells(w, s.box, R_LIST, s.open_axes)
    np.testing.assert_array_equal(off, want_off)
    np.testing.assert_array_equal(js, want_js)
    _, start, atoms = md.cells()
    _, want_start, want_atoms = O.cells(w, s.box, R_LIST, s.open_axes)
    np.testing.assert_array_equal(start, want_start)
    np.testing.assert_array_equal(atoms, want_atoms)
