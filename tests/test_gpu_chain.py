"""Chained steps (many steps in one launch), the overlapping launches of the
node-tile and bidirectional kernels, and the schedules that handles start
with.  Every schedule gives the same bits, so each case compares populations
(both buffers show in the velocity) with the staged march or the oracle."""
import numpy as np
import pytest

import oracle
import workloads as W

pytestmark = pytest.mark.gpu
CHAIN = 12


def Lattice(*a, **k):
    from paper_0807_0602_gb300.build import build
    build()
    from paper_0807_0602_gb300 import lbm
    return lbm.Lattice(*a, **k)


def _run(nx, ny, kind, ratio=False, seed=5):
    if kind == "box":
        geom = W.periodic_box(nx, ny)
    elif kind == "mask":
        geom = W.periodic_box(nx, ny)
        m = np.zeros((ny, nx), np.uint8)
        m[0, : nx // 2] = 1
        m[ny // 2, nx // 3: nx // 2] = 1
        m[:, 0] |= np.arange(ny) % 5 == 0
        geom["mask"] = m
    else:
        geom = W.capillary_geometry(nx, ny, nx // 8, nx - nx // 8, 0, ny - 3)
    nA, nB = W.random_fields(geom, seed, 0.2, 1.2)
    prm = W.params(0.9, 1.0, 0.9, -0.1, 0.05)
    if ratio:
        prm.update(alpha=(4 / 9, 0.8), mass=(1.0, 25 / 9))
    return dict(geom=geom, params=prm, init=("fields", nA, nB))


# one column of tiles and less, tile edges in both directions, one row, masks
GRIDS = [(5, 4, "box"), (3, 1, "box"), (62, 8, "cap"), (63, 9, "cap"), (124, 7, "box"), (125, 33, "mask"),
         (300, 40, "cap")]


@pytest.mark.parametrize("nx,ny,kind", GRIDS)
@pytest.mark.parametrize("rows", [1, 2, 5, 16])
@pytest.mark.parametrize("ratio", [False, True])
def test_chained_steps_equal_the_oracle(nx, ny, kind, rows, ratio):
    run = _run(nx, ny, kind, ratio)
    ref = oracle.OracleLattice(run["geom"], run["params"], run["init"][1], run["init"][2])
    ref.step(41)
    with Lattice(run, precision="f64", tile=(64, rows), kernel=(CHAIN, 4)) as lat:
        lat.step(1)      # one step, an even and an odd number of chained ones
        lat.step(30)
        lat.step(7)
        lat.step(3)
        assert lat.status() == 0
        assert np.array_equal(lat.populations(), ref.populations())
        v, w = lat.velocity(), ref.velocity()
        assert np.array_equal(v[0], w[0]) and np.array_equal(v[1], w[1])


@pytest.mark.parametrize("chunk", [0, -1, 3])
def test_chained_batch_with_log_equals_single_steps(chunk):
    """Runs of uneven size share the chain; the log cuts it at its records."""
    runs = [_run(90, 14, "cap", seed=1), _run(200, 33, "cap", seed=2), _run(64, 50, "cap", seed=3)]
    kw = dict(precision="f64", log_every=10, log_capacity=16, graph_chunk=chunk)
    with Lattice(runs, tile=(64, 3), kernel=(CHAIN, 4), **kw) as a, Lattice(runs, tile=(128, 4), kernel=(6, 4), **kw) as b:
        for n in (4, 31, 25):
            a.step(n)
            b.step(n)
        for r in range(3):
            assert np.array_equal(a.populations(r), b.populations(r))
            assert np.array_equal(a.log(r), b.log(r))


def test_chain_is_refused_outside_fp64_and_its_tilings():
    from paper_0807_0602_gb300 import _lib as L
    with Lattice(_run(64, 18, "cap"), precision="f32") as lat:
        with pytest.raises(L.LbmError):
            lat.schedule = (64, 4, CHAIN, 4)
    with Lattice(_run(64, 18, "cap"), precision="f64") as lat:
        before = lat.schedule
        for bad in ((128, 4, CHAIN, 4), (64, 4, CHAIN, 3), (64, 0, CHAIN, 4)):
            with pytest.raises(L.LbmError):
                lat.schedule = bad
        assert lat.schedule == before


# grids on both sides of the sizes at which the starting schedule changes
@pytest.mark.parametrize("prec,nx,ny", [("f32", 33, 7), ("f32", 3, 5), ("f32", 300, 40), ("f32", 1300, 100),
                                        ("f32", 1301, 100), ("f32", 2500, 100),
                                        ("f32", 2501, 100), ("f32", 1300, 700), ("f16s", 300, 40),
                                        ("f16s", 2501, 100), ("f64", 100, 40), ("f64", 300, 99), ("f64", 300, 101)])
def test_starting_schedule_gives_the_same_bits(prec, nx, ny):
    run = _run(nx, ny, "cap" if nx > 8 else "box")
    kw = dict(precision=prec, rho_ref=(1.0, 1.0))
    with Lattice(run, **kw) as a, Lattice(run, tile=(128, 4), kernel=(6, 4), **kw) as b:
        for n in (1, 18, 5):
            a.step(n)
            b.step(n)
        assert np.array_equal(a.populations().view(np.uint8), b.populations().view(np.uint8))
        va, vb = a.velocity(), b.velocity()
        assert np.array_equal(va[0], vb[0]) and np.array_equal(va[1], vb[1])


def test_pair_kernel_tiles_give_the_whole_velocity():
    run = _run(300, 40, "cap")
    with Lattice(run, precision="f32") as a, Lattice(run, precision="f32", tile=(64, 8), kernel=(7, 4)) as b:
        a.step(6)
        b.step(6)
        for p, q in zip(a.velocity(), b.velocity()):
            assert np.array_equal(p, q)


def test_checkpoint_of_a_starting_schedule_loads(tmp_path):
    run = _run(300, 40, "cap")
    from paper_0807_0602_gb300.lbm import Lattice as Lat
    for prec in ("f32", "f64"):
        with Lattice(run, precision=prec) as a:
            a.step(9)
            a.save(str(tmp_path / prec))
            a.step(8)
            with Lat.load(str(tmp_path / prec)) as b:
                b.step(8)
                assert np.array_equal(a.populations(), b.populations())


# less than a tile, exact tiles, one column or row more, wraps on every side
@pytest.mark.parametrize("nx,ny,kind", [(4, 4, "box"), (26, 10, "box"), (27, 11, "cap"), (25, 9, "mask"),
                                        (53, 31, "mask"), (130, 20, "cap")])
@pytest.mark.parametrize("prec,ratio", [("f32", False), ("f32", True), ("f16s", False)])
def test_two_steps_per_launch_equal_single_steps(nx, ny, kind, prec, ratio):
    run = _run(nx, ny, kind, ratio)
    kw = dict(precision=prec, rho_ref=(1.0, 1.0), log_every=11, log_capacity=8)
    with Lattice(run, tile=(32, 6), kernel=(13, 4), **kw) as a, Lattice(run, tile=(128, 4), kernel=(6, 4), **kw) as b:
        for n in (1, 4, 5, 6, 9, 20):     # both parities at the start, whole log intervals and parts
            a.step(n)
            b.step(n)
            assert np.array_equal(a.populations().view(np.uint8), b.populations().view(np.uint8))
            for p, q in zip(a.velocity(), b.velocity()):   # reads the state of the step before
                assert np.array_equal(p, q)
        assert np.array_equal(a.log(), b.log(), equal_nan=True)


def test_two_step_tilings_are_validated():
    from paper_0807_0602_gb300 import _lib as L
    with Lattice(_run(64, 18, "cap"), precision="f32") as lat:
        before = lat.schedule
        for bad in ((64, 6, 13, 4), (32, 14, 13, 4), (32, 6, 13, 3)):
            with pytest.raises(L.LbmError):
                lat.schedule = bad
        assert lat.schedule == before
    with Lattice(_run(64, 3, "box"), precision="f32") as lat:   # fewer than four rows
        with pytest.raises(L.LbmError):
            lat.schedule = (32, 6, 13, 4)


@pytest.mark.parametrize("chunk", [0, -1, 70])
def test_steps_of_several_chained_launches(chunk):
    """800 000 nodes: at most 41 steps to a launch, within the log's graph, too."""
    run = dict(_run(2000, 400, "cap"), params=W.params(1.0, 1.0, 1.0, -0.2), init=("slab", 0, 700))
    for every in (0, 100):
        kw = dict(precision="f64", graph_chunk=chunk, log_every=every, log_capacity=8 if every else 0)
        with Lattice(run, tile=(64, 16), kernel=(CHAIN, 4), **kw) as a, Lattice(run, tile=(64, 16), kernel=(9, 4), **kw) as b:
            for n in (1, 130, 269):
                a.step(n)
                b.step(n)
                assert a.status() == 0 and a.t == b.t
            for p, q in zip(a.densities(), b.densities()):
                assert np.array_equal(p, q)
            for p, q in zip(a.velocity(), b.velocity()):   # reads the state of the step before
                assert np.array_equal(p, q)
            if every:
                assert np.array_equal(a.log(), b.log())
