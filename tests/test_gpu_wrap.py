"""Bidirectional and chained tiles next to the periodic wrap: with nx = 62 k + 1
(W = 64) or 126 k + 1 (W = 128) the last strip is one column wide, and the
strip before it reads a column whose neighbour is column 0.  Plates that start
there must bounce its populations back (they used to be missed)."""
import numpy as np
import pytest

import oracle
import workloads as W

pytestmark = pytest.mark.gpu


def Lattice(*a, **k):
    from paper_0807_0602_gb300.build import build
    build()
    from paper_0807_0602_gb300 import lbm
    return lbm.Lattice(*a, **k)


def _run(nx, ny, x0, x1):
    geom = W.capillary_geometry(nx, ny, x0, x1, 2, ny - 3)
    nA, nB = W.random_fields(geom, 3, 0.2, 1.2)
    return dict(geom=geom, params=W.params(0.9, 1.0, 0.9, -0.1, 0.05), init=("fields", nA, nB))


# plates at column 0 only, over the whole width, and ending at the last column
GRIDS = [(125, 24, 0, 50), (187, 40, 0, 62), (187, 16, 0, 187), (187, 16, 100, 187), (253, 24, 0, 84),
         (379, 17, 0, 180)]


@pytest.mark.parametrize("nx,ny,x0,x1", GRIDS)
@pytest.mark.parametrize("kernel", [9, 11, 12, None])
def test_fp64_next_to_the_wrap_equals_the_oracle(nx, ny, x0, x1, kernel):
    run = _run(nx, ny, x0, x1)
    ref = oracle.OracleLattice(run["geom"], run["params"], run["init"][1], run["init"][2])
    ref.step(12)
    kw = {} if kernel is None else dict(tile=(64, 5), kernel=(kernel, 4))
    with Lattice(run, precision="f64", **kw) as lat:
        lat.step(5)
        lat.step(7)
        assert np.array_equal(lat.populations(), ref.populations())


@pytest.mark.parametrize("nx,ny,x0,x1", GRIDS)
@pytest.mark.parametrize("prec", ["f32", "f16s"])
@pytest.mark.parametrize("kernel", [9, 11])
@pytest.mark.parametrize("width", [64, 128])
def test_fp32_next_to_the_wrap_equals_the_staged_march(nx, ny, x0, x1, prec, kernel, width):
    run = _run(nx, ny, x0, x1)
    kw = dict(precision=prec, rho_ref=(1.0, 1.0))
    with Lattice(run, tile=(width, 5), kernel=(kernel, 4), **kw) as a, \
            Lattice(run, tile=(128, 4), kernel=(6, 4), **kw) as b:
        a.step(12)
        b.step(12)
        assert np.array_equal(a.populations().view(np.uint8), b.populations().view(np.uint8))


def test_a_batch_of_unlike_runs_next_to_the_wrap():
    runs = [_run(187, 40, 0, 62), _run(253, 24, 0, 84), _run(130, 24, 0, 40)]
    with Lattice(runs, precision="f32", tile=(64, 7), kernel=(9, 4)) as a, \
            Lattice(runs, precision="f32", tile=(128, 4), kernel=(6, 4)) as b:
        a.step(12)
        b.step(12)
        for r in range(3):
            assert np.array_equal(a.populations(r), b.populations(r))
