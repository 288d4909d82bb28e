"""Changing a handle's schedule: what happens when memory runs out, that
the autotuner can stay with the schedule it starts from, and that checkpoints
keep a schedule somebody chose."""
import numpy as np
import pytest

import workloads as W

pytestmark = pytest.mark.gpu


def _run(nx, ny):
    geom = W.capillary_geometry(nx, ny, nx // 8, nx - nx // 8, 0, ny - 3)
    nA, nB = W.random_fields(geom, 5, 0.2, 1.2)
    return dict(geom=geom, params=W.params(0.9, 1.0, 0.9, -0.1, 0.05), init=("fields", nA, nB))


# (precision, grid, schedule before, schedules whose tables need memory beyond
# the starting schedule's: kernel 9 with two rows, kernel 8)
@pytest.mark.parametrize("prec,grid,before,wanted", [
    ("f64", (300, 60), (64, 16, 9, 4), [(64, 16, 12, 4), (64, 1, 9, 4), (64, 1, 12, 4)]),
    ("f64", (300, 60), (64, 16, 12, 4), [(64, 1, 12, 4), (64, 1, 9, 4), (128, 1, 6, 4)]),
    ("f32", (700, 200), (128, 16, 6, 4), [(32, 6, 13, 4), (128, 4, 10, 4), (64, 1, 9, 4)]),
])
def test_a_schedule_that_does_not_fit_in_memory_leaves_the_old_one(monkeypatch, prec, grid, before, wanted):
    """The old schedule stays and works (kernels 12 and 13 used to be selected
    without their tables, which the next step would have read)."""
    from paper_0807_0602_gb300 import _lib as L
    from paper_0807_0602_gb300 import lbm
    from paper_0807_0602_gb300.build import build
    build()
    deny = []

    class Denying(lbm._TorchAllocator):
        def _alloc(self, ctx, nbytes, stream):
            return None if deny else super()._alloc(ctx, nbytes, stream)

    monkeypatch.setattr(lbm, "_TorchAllocator", Denying)
    run = _run(*grid)
    with lbm.Lattice(run, precision=prec, tile=before[:2], kernel=before[2:]) as a, \
            lbm.Lattice(run, precision=prec, tile=(128, 4), kernel=(6, 4)) as b:
        a.step(3)
        for s in wanted:
            deny.append(1)
            with pytest.raises(L.LbmError) as e:
                a.schedule = s
            assert e.value.code == L.LBM_ENOMEM
            deny.clear()
            assert a.schedule == before and a.status() == L.LBM_OK
            a.step(6)
        a.schedule = wanted[0]
        a.step(5)
        b.step(3 + 6 * len(wanted) + 5)
        assert a.schedule == wanted[0]
        assert np.array_equal(a.populations(), b.populations())


def test_the_autotuner_times_the_starting_schedule():
    """1024 x 66 FP32 starts with two steps per launch (3.0 us per step), a
    quarter faster than every other kernel: it has to be among the finalists."""
    from paper_0807_0602_gb300 import lbm
    from paper_0807_0602_gb300.build import build
    build()
    run = _run(1024, 66)
    run.update(params=W.params(1.0, 1.0, 1.0, -0.2), init=("slab", 0, 400))
    with lbm.Lattice(run, precision="f32", autotune=True) as a, lbm.Lattice(run, precision="f32") as b:
        start = a.schedule
        assert start == (32, 6, 13, 4) and start == b.schedule
        a.step(3000)
        b.step(3000)
        assert start in [s for s, _ in a.tuning()]
        assert a.schedule == min(a.tuning(), key=lambda c: c[1])[0]
        assert np.array_equal(a.populations(), b.populations())


@pytest.mark.parametrize("prec,schedule", [
    ("f32", (64, 5, 9, 4)), ("f32", (32, 14, 8, 4)), ("f32", (128, 4, 10, 3)), ("f16s", (256, 7, 2, 6)),
    ("f64", (64, 3, 12, 4)), ("f64", (256, 100000, 0, 4)), ("f32", (64, 6, 11, 4)), ("f32", None), ("f64", None)])
def test_checkpoints_keep_a_chosen_schedule(tmp_path, prec, schedule):
    from paper_0807_0602_gb300 import lbm
    from paper_0807_0602_gb300.build import build
    build()
    path = str(tmp_path / "state")
    with lbm.Lattice(_run(300, 40), precision=prec) as a:
        first = a.schedule
        if schedule is not None:
            a.schedule = schedule
        a.step(9)
        a.save(path)
        a.step(8)
        with lbm.Lattice.load(path) as b:
            assert b.schedule == (schedule or first)
            b.step(8)
            assert np.array_equal(a.populations().view(np.uint8), b.populations().view(np.uint8))


def test_checkpoints_keep_a_chosen_tiling(tmp_path):
    from paper_0807_0602_gb300 import lbm
    from paper_0807_0602_gb300.build import build
    build()
    path = str(tmp_path / "state")
    with lbm.Lattice(_run(300, 40), precision="f32") as a:
        a.tiling = (128, 16)
        a.step(9)
        a.save(path)
        with lbm.Lattice.load(path) as b:
            assert b.tiling == (128, 16) and b.schedule == a.schedule


@pytest.mark.parametrize("prec", ["f64", "f32", "f16s"])
def test_tilings_of_the_marches_equal_each_other(prec):
    """Tiles of one row up to more rows than the run has, strips of each width,
    with and without graphs.  (A tile given at creation without a kernel changes
    nothing: the library chooses the schedule.)"""
    from paper_0807_0602_gb300 import lbm
    from paper_0807_0602_gb300.build import build
    build()
    geom = W.capillary_geometry(333, 37, 50, 300, 2, 30)
    run = dict(geom=geom, params=W.params(1.2, 1.0, 0.9, -0.1, 0.05), init=("slab", 0, 120))
    kw = dict(precision=prec, rho_ref=(1.0, 1.0))
    with lbm.Lattice(run, **kw) as lat, lbm.Lattice(run, tile=(64, 3), **kw) as given:
        assert lat.schedule == given.schedule
        lat.step(23)
        want = lat.populations().view(np.uint8)
    for tile, chunk in (((128, 16), 0), ((64, 1), -1), ((64, 3), 5), ((256, 37), 0), ((128, 100), 7)):
        kernels = {6, 0} if prec != "f64" or tile[0] < 256 else {0}
        for kernel in kernels:
            with lbm.Lattice(run, graph_chunk=chunk, tile=tile, kernel=(kernel, 4), **kw) as lat:
                assert lat.schedule == (*tile, kernel, 4)
                lat.step(23)
                assert np.array_equal(lat.populations().view(np.uint8), want)


def test_batched_runs_of_the_marches_equal_solo_runs():
    from paper_0807_0602_gb300 import lbm
    from paper_0807_0602_gb300.build import build
    build()
    runs = [W.capillary_run(L, H, 1.0 + 0.05 * j, 1.0, 0.8 + 0.1 * j, -0.1 * j)
            for j, (L, H) in enumerate(((40, 6), (100, 13), (65, 30), (7, 3)))]
    for kernel in (6, 0):
        with lbm.Lattice(runs, precision="f32", tile=(64, 8), kernel=(kernel, 4)) as bat:
            bat.step(40)
            for r, run in enumerate(runs):
                with lbm.Lattice(run, precision="f32", tile=(128, 16), kernel=(kernel, 4)) as solo:
                    solo.step(40)
                    assert np.array_equal(solo.populations(), bat.populations(r))
                    assert np.array_equal(solo.interface(), bat.interface(r))
                    assert np.array_equal(solo.mass(), bat.mass(r))
