"""FP64 step against the oracle where its forms differ: relaxation times equal
to 1 (products with 1 left out) and not, with and without a body force, and
densities at both ends of the exponent range, where the common velocity's
quotients leave the shared-reciprocal path.  Bit-equal in every case."""
import numpy as np
import pytest

import oracle
import workloads as W

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("scale", [1.0, 1e-70, 1e70])
@pytest.mark.parametrize("tau", [(1.0, 1.0), (1.0, 0.9), (0.8, 1.0), (1.1, 0.7)])
@pytest.mark.parametrize("body", [(0.0, 0.0), (1e-5, -2e-5)])
def test_f64_forms_bit_equal(scale, tau, body):
    from paper_0807_0602_gb300.build import build
    build()
    from paper_0807_0602_gb300.lbm import Lattice
    geom = W.capillary_geometry(70, 21, 10, 60, 0, 17)
    nA, nB = W.random_fields(geom, 11, 0.2, 1.2)
    prm = W.params(0.9 / scale, *tau, -0.1, 0.07, body=body)
    ref = oracle.OracleLattice(geom, prm, nA * scale, nB * scale)
    ref.step(12)
    want = ref.populations()
    with Lattice(dict(geom=geom, params=prm, init=("fields", nA * scale, nB * scale)), precision="f64") as lat:
        for sched in ((128, 4, 6, 4), (64, 8, 9, 4), (128, 5, 4, 4)):
            lat.schedule = sched
            lat.step(4)
        got = lat.populations()
    assert np.all(np.isfinite(want)) and np.array_equal(got, want)


@pytest.mark.parametrize("tau", [(1.0, 1.0), (1.0, 1.3)])
@pytest.mark.parametrize("lo,hi", [(0.9, 1.1), (0.02, 2.0)])
def test_integer_forms_bit_equal_on_larger_grids(tau, lo, hi):
    """From 30 000 nodes on the brackets are formed on integers where u.u is
    below its bound (everywhere in the mild field, not so in the rough one)."""
    from paper_0807_0602_gb300.build import build
    build()
    from paper_0807_0602_gb300.lbm import Lattice
    geom = W.capillary_geometry(251, 130, 30, 220, 0, 117)
    nA, nB = W.random_fields(geom, 4, lo, hi)
    prm = W.params(0.9, *tau, -0.1, 0.07)
    ref = oracle.OracleLattice(geom, prm, nA, nB)
    ref.step(8)
    with Lattice(dict(geom=geom, params=prm, init=("fields", nA, nB)), precision="f64") as lat:
        lat.step(3)
        for sched in ((128, 4, 6, 4), (64, 8, 9, 4), (128, 5, 4, 4), (32, 6, 8, 4), (64, 6, 11, 4)):
            lat.schedule = sched
            lat.step(1)
        got = lat.populations()
    assert np.all(np.isfinite(got)) and np.array_equal(got, ref.populations())
