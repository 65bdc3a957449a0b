"""Batches of the same systems take the same launch shape in one process, so
that their energies, whose sums follow the shape, are the same bits."""
import numpy as np
import pytest

from paper_2405_07898_gb300 import binding, inputs as I

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("nrep", [1, 7, 40, 160])
def test_energies_do_not_depend_on_the_creation(nrep):
    systems = [I.thermal_system(I.BCC_TA_LIKE, (5 + k % 4, 6, 5 + k % 3), 0.02, 300.0, 40 + k) for k in range(nrep)]
    first = None
    for _ in range(6):
        with binding.MDBatch(systems) as b:
            b.step(12, 2.0)
            i = b.info()
            got = [i["blocks"], i["threads_per_block"], *b.energy()]
        if first is None:
            first = got
        for x, y in zip(first, got):
            np.testing.assert_array_equal(x, y)
