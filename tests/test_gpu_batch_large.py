"""A batch whose largest replica is beyond the pinned staging buffer, beside
replicas within it: states equal the single contexts' bit for bit."""
import numpy as np
import pytest

from paper_2405_07898_gb300 import binding, inputs as I

pytestmark = pytest.mark.gpu


def test_states_beyond_the_staging_buffer():
    systems = [I.bcc_cube(7), I.bcc_cube(33), I.bcc_cube(32)]  # 686, 71,874 and 65,536 atoms
    with binding.MDBatch(systems, schedule=1) as b:
        b.step(12, 2.0)
        got = [b.get_state(r) for r in (1, 0, 2)]
    for r, state in zip((1, 0, 2), got):
        with binding.MD(systems[r], precision="mixed", lanes_per_atom=1, persistent="off") as md:
            md.step(12, 2.0)
            for a, x in zip(state, (*md.get_state()[:2], md.forces())):
                np.testing.assert_array_equal(a, x)
