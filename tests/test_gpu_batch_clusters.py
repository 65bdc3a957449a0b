"""Each cluster shape of the batch launch (2, 4 and 8 blocks per replica),
chosen by hand: parts of a replica that are ragged or empty (1 atom, fewer
than 32 a block), list builds across blocks, the hand-over of the next replica
to the cluster's blocks (more replicas than clusters that can be resident).
States equal the single contexts' bit for bit."""
import numpy as np
import pytest

from paper_2405_07898_gb300 import binding, inputs as I
from test_gpu_batch_teams import SYSTEMS, gas

pytestmark = pytest.mark.gpu

MORE = {
    "below_32_a_block": lambda: [gas(n, n) for n in (2, 31, 63, 65, 127, 129, 250)],
    "queued": lambda: [gas(30 + k, 100 + k) for k in range(330)],
}
_single = {}


def single(which, systems):
    """The single contexts' states after 14 + 14 + 9 steps."""
    if which not in _single:
        _single[which] = []
        for s in systems:
            with binding.MD(s, precision="mixed", lanes_per_atom=1, persistent="off") as md:
                for n in (14, 14, 9):
                    md.step(n, 2.0)
                _single[which].append((*md.get_state()[:2], md.forces(), *md.energy()))
    return _single[which]


@pytest.mark.parametrize("schedule,blocks", [(6, 2), (7, 4), (8, 8)])
@pytest.mark.parametrize("which", list(SYSTEMS) + list(MORE))
def test_replicas_equal_single_contexts(which, schedule, blocks):
    systems = {**SYSTEMS, **MORE}[which]()
    with binding.MDBatch(systems, schedule=1) as b:
        assert b.info()["blocks_per_replica"] == 1
        b.step(14, 2.0)  # a graph of this length is kept, with one block per replica
        b.set_schedule(schedule)
        b.step(14, 2.0)
        b.step(9, 2.0)
        info = b.info()
        assert info["blocks_per_replica"] == blocks and info["blocks"] % blocks == 0
        assert info["rebuilds"] >= 3 * len(systems)
        pe, ke = b.energy()
        got = [b.get_state(r) for r in range(len(systems))]
    for r, want in enumerate(single(which, systems)):
        for a, x in zip(got[r], want[:3]):
            np.testing.assert_array_equal(a, x, err_msg=f"replica {r}")
        # sums over another partition of the atoms: FP32 partial sums of at
        # most 32 atoms a thread (2^-24 each) in FP64 totals
        assert abs(pe[r] - want[3]) <= 32 * 2.0**-24 * max(abs(want[3]), 1e-3)
        assert abs(ke[r] - want[4]) <= 32 * 2.0**-24 * max(abs(want[4]), 1e-9)


def test_shapes_that_do_not_exist_and_back_to_the_chosen_one():
    systems = [I.bcc_cube(6), I.bcc_cube(7)]
    with binding.MDBatch(systems) as b:
        chosen = b.info()
        for bad in (-1, 9):
            with pytest.raises(binding.MDError) as e:
                b.set_schedule(bad)
            assert e.value.status == -1
        b.set_schedule(8)
        assert b.info()["blocks"] == 16
        b.set_schedule(0)
        for k in ("blocks", "threads_per_block", "blocks_per_replica"):
            assert b.info()[k] == chosen[k]
