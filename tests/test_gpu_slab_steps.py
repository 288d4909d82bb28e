"""Steps of GPU slabs by one library call against the general exchange
(get_columns / set_columns after every step): equal bits for every precision,
slab count down to the smallest slab, and slabs that step different kernels;
slabs that cannot share a launch take the general exchange."""
import numpy as np
import pytest

import workloads as W

pytestmark = pytest.mark.gpu


def _slabs(nx, ny, parts, seed=9, **kw):
    from paper_0807_0602_gb300.build import build
    build()
    from paper_0807_0602_gb300 import slab as SL
    geom = W.capillary_geometry(nx, ny, nx // 8, nx - 3, 0, ny - 1)
    nA, nB = W.random_fields(geom, seed, 0.2, 1.2)
    run = dict(geom=geom, params=W.params(1.2, 1.0, 0.9, -0.1, 0.05), init=("fields", nA, nB))
    return [SL.Slab(run, a, b, nA, nB, **kw) for a, b in SL.slab_bounds(nx, parts)]


def _general(slabs, n):
    from paper_0807_0602_gb300 import slab as SL
    for _ in range(n):
        for s in slabs:
            s.step()
        SL.exchange_local(slabs)


def _all(slabs):
    return np.concatenate([s.lat.populations() for s in slabs], axis=-1)


@pytest.mark.parametrize("prec", ["f32", "f16s", "f64"])
@pytest.mark.parametrize("nx,ny,parts", [(300, 41, 1), (300, 41, 3), (16, 5, 4), (133, 67, 32)])
def test_native_steps_equal_the_general_exchange(prec, nx, ny, parts):
    from paper_0807_0602_gb300 import slab as SL
    kw = dict(precision=prec, rho_ref=(1.0, 1.0))
    a, b = _slabs(nx, ny, parts, **kw), _slabs(nx, ny, parts, **kw)
    for n in (1, 6, 2):
        assert SL._step_native(a, n)
        _general(b, n)
    assert all(s.lat.t == 9 and s.lat.status() == 0 for s in a)
    assert np.array_equal(_all(a).view(np.uint8), _all(b).view(np.uint8))


def test_other_slabs_take_the_general_exchange():
    import torch
    from paper_0807_0602_gb300 import slab as SL
    a, b = _slabs(120, 20, 2), _slabs(120, 20, 2)
    other = torch.cuda.Stream()
    with torch.cuda.stream(other):
        c = _slabs(120, 20, 2)
    mixed = [a[0], c[1]]
    assert not SL._step_native(mixed, 1) and not SL._step_native([a[0], a[0]], 1)
    assert not SL._step_native(a + _slabs(120, 21, 2), 1)
    a[1].lat.schedule = (64, 5, 9, 4)      # different kernels in one ring
    SL.step_local(a, 5)
    _general(b, 5)
    assert np.array_equal(_all(a), _all(b))


@pytest.mark.parametrize("prec", ["f32", "f64"])
@pytest.mark.parametrize("cuts", [(0, 2, 40), (0, 3, 5, 40), (0, 37, 40)])
def test_slabs_of_two_or_three_columns_step(prec, cuts):
    """Slabs built by hand may be narrower than the library's call takes: they
    go through the general exchange and still equal the undivided run."""
    from paper_0807_0602_gb300 import slab as SL
    from paper_0807_0602_gb300.lbm import Lattice
    geom = W.capillary_geometry(40, 12, 5, 37, 0, 11)
    nA, nB = W.random_fields(geom, 4, 0.2, 1.2)
    run = dict(geom=geom, params=W.params(1.2, 1.0, 0.9, -0.1, 0.05), init=("fields", nA, nB))
    _slabs(40, 12, 1)   # (builds the library)
    slabs = [SL.Slab(run, a, b, nA, nB, precision=prec) for a, b in zip(cuts, cuts[1:])]
    with Lattice(run, precision=prec) as whole:
        SL.step_local(slabs, 7)
        whole.step(7)
        got = np.concatenate([s.owned(s.lat.populations()) for s in slabs], axis=-1)
        assert np.array_equal(got, whole.populations())
