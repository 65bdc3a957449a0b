"""md_force_match on a state in error answers with the error and queues no
kernel: what a timed-out or refused state left is not a list to follow."""
import numpy as np
import pytest

from paper_2405_07898_gb300 import binding, inputs as I

pytestmark = pytest.mark.gpu


def refused(md, s, status):
    before = md.stats()["kernel_launches"]
    with pytest.raises(binding.MDError) as e:
        md.force_match(np.zeros((s.n, 3)), 0.0, 0.1)
    assert e.value.status == status
    assert md.stats()["kernel_launches"] == before


def test_states_in_error():
    s = I.bcc_2000_fp64()
    s.pot = I.johnson_potential(I.BCC_TA_LIKE, 64)  # within the capacity of the gradient bins
    with binding.MD(s, precision="fp64", persistent="on", lanes_per_atom=2, wait_limit_us=1) as md:
        want = md.force_match(np.zeros((s.n, 3)), 0.0, 0.1)
        md.step(200, 2.0)
        refused(md, s, -6)  # MD_ERR_TIMEOUT, seen by this call first
        refused(md, s, -6)
        md.set_state(s.pos, s.vel, 0)
        bad = s.pos.copy()
        bad[3, 2] = np.inf
        with pytest.raises(binding.MDError):
            md.set_state(bad)
        refused(md, s, -5)  # MD_ERR_NONFINITE
        md.set_state(s.pos, s.vel, 0)
        got = md.force_match(np.zeros((s.n, 3)), 0.0, 0.1)
    assert got[0] == want[0]
    np.testing.assert_array_equal(got[1], want[1])
