"""Batches against single contexts, bit for bit: a replica is advanced by the
per-atom functions of the single-system path (one lane per atom), by one block
or by a cluster of blocks (few replicas), so its state after steps with list
builds must equal the single context's exactly, whatever the split."""
import numpy as np
import pytest

from paper_2405_07898_gb300 import binding, inputs as I

pytestmark = pytest.mark.gpu


def gas(n, seed):
    rng = np.random.default_rng(seed)
    box = np.array([15.1, 21.0, 33.0])
    keep = [rng.random(3) * box]
    while len(keep) < n:
        x = rng.random(3) * box
        d = np.asarray(keep) - x
        d -= box * np.round(d / box)
        if (d * d).sum(1).min() > 1.6**2:
            keep.append(x)
    pos = np.asarray(keep)
    return I.System(box=box, pos=pos, vel=rng.normal(scale=0.002, size=pos.shape), types=np.zeros(n, np.int32),
                    pot=I.johnson_potential(I.BCC_TA_LIKE, 300))


SYSTEMS = {
    "one_atom": lambda: [gas(1, 1)],
    "ragged": lambda: [gas(33, 2), gas(257, 3), gas(1023, 4)],
    "one_crystal": lambda: [I.bcc_cube(12, 900.0)],
    "mixed": lambda: [I.thermal_system(I.FCC_CU_LIKE, (5, 6, 7), 0.02, 600.0, 5), gas(500, 6),
                      I.thermal_system(I.BCC_TA_LIKE, (9, 8, 11), 0.02, 1100.0, 7)],
    "many": lambda: [gas(40 + 7 * k, 10 + k) for k in range(45)],
}


@pytest.mark.parametrize("schedule", [0, 1, 3, 4])
@pytest.mark.parametrize("which", list(SYSTEMS))
def test_replicas_equal_single_contexts(which, schedule):
    systems = SYSTEMS[which]()
    with binding.MDBatch(systems, schedule=schedule) as b:
        b.step(14, 2.0)
        b.step(9, 2.0)
        pe, ke = b.energy()
        got = [b.get_state(r) for r in range(len(systems))]
    for r, s in enumerate(systems):
        with binding.MD(s, precision="mixed", lanes_per_atom=1, persistent="off") as md:
            md.step(14, 2.0)
            md.step(9, 2.0)
            pos, vel, _ = md.get_state()
            e = md.energy()
            for a, want in zip(got[r], (pos, vel, md.forces())):
                np.testing.assert_array_equal(a, want)
        # sums over another partition of the atoms: FP32 partial sums of at
        # most 32 atoms a thread (2^-24 each) in FP64 totals
        assert abs(pe[r] - e[0]) <= 32 * 2.0**-24 * max(abs(e[0]), 1e-3)
        assert abs(ke[r] - e[1]) <= 32 * 2.0**-24 * max(abs(e[1]), 1e-9)
