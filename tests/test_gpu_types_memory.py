"""Alloys with large tables: the rows per type pair, whose size grows with the
square of the types, are made only up to 256 MB; beyond, the general kernels
read the plain rows, and forces are right either way."""
import numpy as np
import pytest

import oracle as O
from paper_2405_07898_gb300 import binding, inputs as I
from bars import assert_forces
from test_gpu_types import alloy

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("n_knots,pair_rows", [(20_000, True), (150_000, False)])
def test_device_memory_of_the_tables(n_knots, pair_rows):
    import torch

    s = alloy(8, n_knots, cells=(5, 5, 5), n_knots=n_knots)
    asked = []

    def alloc(nbytes):
        asked.append(nbytes)
        return torch.cuda.caching_allocator_alloc(nbytes)

    with binding.MD(s, precision="mixed", persistent="off", lanes_per_atom=1,
                    allocator=(alloc, torch.cuda.caching_allocator_delete)) as md:
        f = md.forces()
        md.step(12, 2.0)
        pos = md.get_state()[0]
        late = md.forces()
    pot = O.Potential(s.pot)
    assert_forces(f, O.eam_eval(pot, O.wrap(s.pos, s.box), s.box, s.types)[2], "mixed")
    assert_forces(late, O.eam_eval(pot, O.wrap(pos, s.box), s.box, s.types)[2], "mixed")
    # a word is 4 bytes: F, f and phi rows of 4 words each, per pair 16 words and the f rows again
    plain, extra = (8 + 8 + 36) * 4 * 4 * n_knots, (36 * 16 + 8 * 4) * 4 * n_knots
    state = 64 << 20  # more than the state and the list of 250 atoms take
    assert sum(asked) < plain + (extra if pair_rows else 0) + state
    if pair_rows:
        assert sum(asked) > extra
