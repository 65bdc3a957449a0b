"""One state, every way in: the evaluation of md_create, of md_set_state with
the same arrays and of md_set_potential with the same tables give the same
forces, energies and virial bit for bit, and runs from them the same
trajectories, whichever launches the schedules chose."""
import numpy as np
import pytest

from paper_2405_07898_gb300 import binding, inputs as I

pytestmark = pytest.mark.gpu

SYSTEMS = {
    "bcc_1024": lambda: I.bcc_cube(8, 1000.0),
    "bcc_2000": lambda: I.bcc_2000_fp64(),
    "bcc_6750": lambda: I.bcc_cube(15, 1000.0),
    "bcc_16000": lambda: I.bcc_cube(20, 1000.0),
    "fcc_5460": lambda: I.thermal_system(I.FCC_CU_LIKE, (13, 15, 7), 0.02, 300.0, 12),
    "bcc_43904": lambda: I.bcc_cube(28, 1000.0),
    "bcc_71874": lambda: I.bcc_cube(33, 300.0),
    "slab": lambda: I.bcc_slab_small(),
    "alloy": lambda: I.multi_type_system((9, 10, 11)),
}


def answers(md):
    return [md.forces(), np.array(md.energy()), md.virial()]


def equal(a, b, what):
    for x, y in zip(a, b):
        np.testing.assert_array_equal(x, y, err_msg=what)


@pytest.mark.parametrize("precision", ["mixed", "fp64"])
@pytest.mark.parametrize("persistent", ["auto", "off"])
@pytest.mark.parametrize("which", list(SYSTEMS))
def test_same_bits_by_every_way_in(which, persistent, precision):
    s = SYSTEMS[which]()
    with binding.MD(s, precision=precision, persistent=persistent) as md:
        first = answers(md)
        md.set_potential(s.pot)
        equal(first, answers(md), "md_set_potential after md_create")
        md.step(25, 2.0)
        run = list(md.get_state()[:2]) + answers(md)
        md.set_state(s.pos, s.vel, 0)
        equal(first, answers(md), "md_set_state")
        md.set_potential(s.pot)
        equal(first, answers(md), "md_set_potential after md_set_state")
        md.step(25, 2.0)
        equal(run, list(md.get_state()[:2]) + answers(md), "25 steps")


@pytest.mark.parametrize("cells,precision,one", [(10, "mixed", True), (10, "fp64", True), (13, "fp64", False),
                                                 (32, "mixed", True), (33, "mixed", False)])
def test_evaluated_by_one_launch_up_to_its_size(cells, precision, one):
    """The single launch evaluates a state up to 65,536 atoms (FP64: 4,096);
    larger systems that step by it are faster with a launch per kernel."""
    s = I.bcc_cube(cells)
    with binding.MD(s, precision=precision, persistent="on", lanes_per_atom=2) as md:
        before = md.stats()["kernel_launches"]
        md.set_state(s.pos, s.vel)
        assert (md.stats()["kernel_launches"] - before == 1) == one
