"""Forces of several atom types against the oracle, after steps with list
builds, for each kind of tables: all f and phi on one knot grid (rows per type
pair), a grid of its own for one of them (any tables), one type whose f and phi
differ in their grid; graphs and the single launch bit for bit."""
import dataclasses

import numpy as np
import pytest

import oracle as O
from paper_2405_07898_gb300 import binding, inputs as I
from bars import assert_forces

pytestmark = pytest.mark.gpu


def alloy(ntypes, knots_of_last_phi, cells=(5, 6, 7), n_knots=300):
    rng = np.random.default_rng(100 * ntypes + knots_of_last_phi)
    base = I.BCC_TA_LIKE
    ps = [dataclasses.replace(base, mass=base.mass * 0.85**t, re=base.re - 0.05 * t, E0=3.0 + 0.2 * t, fe=1.0 + 0.1 * t,
                              A=0.6 + 0.05 * t) for t in range(ntypes)]
    tabs = [I.johnson_knots(p, n_knots) for p in ps]
    phi = []
    for a in range(ntypes):
        for b in range(a, ntypes):
            n = knots_of_last_phi if a == b == ntypes - 1 else n_knots
            pa, pb = I.johnson_knots(ps[a], n)[2], I.johnson_knots(ps[b], n)[2]
            phi.append(I.Knots(pa.x0, pa.dx, 0.5 * (pa.y + pb.y), I.BC_CLAMPED, I.BC_NATURAL, 0.5 * (pa.d_lo + pb.d_lo)))
    pot = I.Potential(mass=np.array([p.mass for p in ps]), F=[t[0] for t in tabs], f=[t[1] for t in tabs], phi=phi,
                      r_cut=base.r_cut, skin=base.skin)
    pos, box = I.bcc_lattice(*cells, base.a)
    pos = I.displace(pos, box, 0.05, rng)
    types = rng.integers(0, ntypes, len(pos)).astype(np.int32)
    return I.System(box=box, pos=pos, vel=I.maxwell(len(pos), pot.mass[types], 500.0, rng), types=types, pot=pot)


@pytest.mark.parametrize("precision", ["fp64", "mixed"])
@pytest.mark.parametrize("lanes", [1, 4])
@pytest.mark.parametrize("ntypes,last", [(2, 300), (3, 300), (8, 300), (3, 211), (1, 211)])
def test_forces_of_each_kind_of_tables(ntypes, last, lanes, precision):
    s = alloy(ntypes, last)
    out = []
    for persistent in ("off", "on"):
        with binding.MD(s, precision=precision, lanes_per_atom=lanes, persistent=persistent) as md:
            pot = O.Potential(s.pot)
            assert_forces(md.forces(), O.eam_eval(pot, O.wrap(s.pos, s.box), s.box, s.types)[2], precision)
            md.step(23, 2.0)
            pos, vel, _ = md.get_state()
            f = md.forces()
            assert_forces(f, O.eam_eval(pot, O.wrap(pos, s.box), s.box, s.types)[2], precision)
            out.append((pos, vel, f))
    for a, b in zip(*out):
        np.testing.assert_array_equal(a, b)
    # the steps between used the same forces: FP64 trajectories of the oracle
    if precision == "fp64":
        ref = O.System(O.Potential(s.pot), s.box, s.pos, s.vel, s.types)
        ref.step(23, 2.0)
        d = out[0][0] - ref.state()["pos"]
        d -= s.box * np.round(d / s.box)
        assert np.abs(d).max() < 1e-9
