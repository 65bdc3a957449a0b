"""A single launch whose waits run out may end inside a list build, with the
cell counts of that build in place.  md_set_state has to start from none of
it: cells, lists and forces of the next state equal the oracle's.  Wait limits
from 1 us up, a build every step, so that launches end at every kind of
barrier; also through the state load of larger FP64 systems, which takes a
launch per kernel.  md_profile, which would build lists from the leftovers,
refuses before it queues anything."""
import numpy as np
import pytest

import oracle as O
from paper_2405_07898_gb300 import binding, inputs as I
from bars import assert_forces

pytestmark = pytest.mark.gpu

MD_ERR_TIMEOUT = -6


@pytest.mark.parametrize("cells,precision", [((10, 10, 10), "mixed"), ((10, 10, 10), "fp64"), ((14, 13, 15), "fp64")])
def test_state_set_after_launches_that_timed_out(cells, precision):
    s = I.thermal_system(I.BCC_TA_LIKE, cells, 0.05, 300.0, 31)
    _, _, F, _, _ = O.eam_eval(O.Potential(s.pot), O.wrap(s.pos, s.box), s.box, s.types)
    want_off, want_js = O.neighbors_cells(O.wrap(s.pos, s.box), s.box, s.pot.r_list)
    _, want_start, want_atoms = O.cells(O.wrap(s.pos, s.box), s.box, s.pot.r_list)
    ended = 0
    for limit in (1, 2, 3, 4, 5, 6, 8, 10, 15, 25, 40):
        with binding.MD(s, precision=precision, persistent="on", lanes_per_atom=2, rebuild_every=1,
                        wait_limit_us=limit) as md:
            for _ in range(3):
                md.step(40, 2.0)
                try:
                    md.sync()
                except binding.MDError as e:
                    assert e.status == MD_ERR_TIMEOUT
                    ended += 1
                    before = md.stats()["kernel_launches"]
                    with pytest.raises(binding.MDError) as p:
                        md.profile(2, 2.0)
                    assert p.value.status == MD_ERR_TIMEOUT
                    assert md.stats()["kernel_launches"] == before
                md.set_state(s.pos, s.vel, 0)
                _, start, atoms = md.cells()
                np.testing.assert_array_equal(start, want_start)
                np.testing.assert_array_equal(atoms, want_atoms)
                off, js = md.neighbors()
                np.testing.assert_array_equal(off, want_off)
                np.testing.assert_array_equal(js, want_js)
                assert_forces(md.forces(), F, precision, f"limit {limit} us")
    assert ended >= 3  # the limit of 1 us runs out every time
