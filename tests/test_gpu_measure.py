"""md_set_state of systems that are evaluated by the single launch (and, beyond
its size rule, by a launch per kernel): energies, virial, forces, lists and
cells against the oracle, a denser state that outgrows the list, a state that
is not finite and the next good one."""
import numpy as np
import pytest

import oracle as O
from paper_2405_07898_gb300 import binding, inputs as I
from bars import assert_forces

pytestmark = pytest.mark.gpu

TOL = {"fp64": 1e-10, "mixed": 2e-5}  # the bars of energies and virials in the other parity tests


def check(md, s, pos, precision):
    w = O.wrap(pos, s.box)
    _, _, F, E, W = O.eam_eval(O.Potential(s.pot), w, s.box, s.types)
    assert_forces(md.forces(), F, precision)
    assert abs(md.energy()[0] - E.sum()) <= TOL[precision] * abs(E.sum())
    assert np.linalg.norm(md.virial() - W) <= TOL[precision] * np.linalg.norm(W)
    off, js = md.neighbors()
    want_off, want_js = O.neighbors_cells(w, s.box, s.pot.r_list)
    np.testing.assert_array_equal(off, want_off)
    np.testing.assert_array_equal(js, want_js)


@pytest.mark.parametrize("precision", ["fp64", "mixed"])
@pytest.mark.parametrize("persistent", ["on", "off"])
@pytest.mark.parametrize("cells", [(5, 5, 5), (10, 11, 9), (13, 13, 13)])  # 250, 1,980, 4,394 atoms
def test_states_against_the_oracle(cells, persistent, precision):
    s = I.thermal_system(I.BCC_TA_LIKE, cells, 0.02, 300.0, 8)
    rng = np.random.default_rng(9)
    with binding.MD(s, precision=precision, persistent=persistent) as md:
        for sigma in (0.15, 0.3):
            pos = s.pos + rng.normal(0.0, sigma, s.pos.shape)  # also outside the box
            md.set_state(pos, s.vel, 3)
            check(md, s, pos, precision)
        _, vel, step = md.get_state()
        assert step == 3
        np.testing.assert_array_equal(vel, s.vel)
        cap = md.stats()["list_capacity"]
        dense = pos * np.array([0.45, 1.0, 1.0])  # half the box empty: longer lists
        md.set_state(dense, None)
        assert md.stats()["list_capacity"] > cap
        check(md, s, dense, precision)
        bad = pos.copy()
        bad[7, 1] = np.nan
        with pytest.raises(binding.MDError) as e:
            md.set_state(bad, s.vel)
        assert e.value.status == -5  # MD_ERR_NONFINITE
        md.set_state(pos, s.vel, 4)
        check(md, s, pos, precision)
        md.step(12, 2.0)
        p, _, step = md.get_state()
        assert step == 16
        assert_forces(md.forces(), O.eam_eval(O.Potential(s.pot), O.wrap(p, s.box), s.box, s.types)[2], precision)
