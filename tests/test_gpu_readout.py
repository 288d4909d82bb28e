"""Field readouts and column copies: densities of FP32 and FP16-shifted
populations equal the FP64 sum of the stored values bit for bit, whatever
their range, signs and finiteness; column windows of every alignment equal
the populations they come from; log records equal the separate readouts."""
import numpy as np
import pytest

import workloads as W

pytestmark = pytest.mark.gpu


def Lattice(*a, **k):
    from paper_0807_0602_gb300.build import build
    build()
    from paper_0807_0602_gb300 import lbm
    return lbm.Lattice(*a, **k)


def _box(nx, ny, prec, **kw):
    geom = W.periodic_box(nx, ny)
    nA, nB = W.random_fields(geom, 2, 0.2, 1.2)
    return Lattice(dict(geom=geom, params=W.params(0.9, 1.0, 1.0), init=("fields", nA, nB)), precision=prec, **kw)


def _values(kind, shape, rng):
    v = rng.uniform(0.01, 1.0, shape)
    if kind == "signs":            # sums of mixed signs, some cancelling far
        v *= rng.choice([-1.0, 1.0], shape)
        v[:, 1] = -v[:, 0] * (1 + 2.0 ** -rng.integers(1, 24, v[:, 0].shape))
    elif kind == "wide":           # magnitudes over the whole FP32 range
        v = np.ldexp(v, rng.integers(-140, 120, shape))
    elif kind == "edge":           # sums just around powers of two, spans around 2^16
        v = np.ldexp(1.0 + 2.0 ** -23 * rng.integers(-2, 3, shape), rng.integers(-17, 1, shape))
        v[:, 0] = 2.0 - v[:, 1]
    elif kind == "special":
        v[rng.random(shape) < 0.1] = 0.0
        v[rng.random(shape) < 0.05] = np.nan
        v[rng.random(shape) < 0.05] = np.inf
    return v


@pytest.mark.parametrize("prec", ["f32", "f16s", "f64"])
@pytest.mark.parametrize("kind", ["plain", "signs", "wide", "edge", "special"])
def test_densities_are_the_fp64_sums(prec, kind):
    import torch
    nx, ny = 200, 33
    rng = np.random.default_rng(9)
    dt = {"f32": np.float32, "f16s": np.float16, "f64": np.float64}[prec]
    with np.errstate(over="ignore"):
        f = _values(kind, (2, 9, ny, nx), rng).astype(dt)
    with _box(nx, ny, prec) as lat:     # rho_ref = 0: stored values are the populations
        lat.set_columns(0, torch.as_tensor(f, device="cuda"))
        got = np.stack(lat.densities())
    want = np.zeros((2, ny, nx))
    with np.errstate(invalid="ignore"):
        for i in range(9):
            want = want + f[:, i].astype(np.float64)
    assert np.array_equal(np.isnan(got), np.isnan(want))
    ok = ~np.isnan(want)
    assert np.array_equal(got[ok], want[ok])


@pytest.mark.parametrize("prec", ["f32", "f16s", "f64"])
@pytest.mark.parametrize("x0,n", [(0, 64), (0, 1), (1, 2), (3, 61), (8, 56), (8, 8), (60, 4), (62, 2), (16, 5)])
def test_column_windows(prec, x0, n):
    import torch
    with _box(64, 11, prec) as lat:
        lat.step(3)
        pops = lat.populations()
        cols = lat.get_columns(x0, n)
        assert np.array_equal(cols.cpu().numpy(), pops[..., x0:x0 + n])
        store = torch.zeros(cols.numel() + 1, dtype=cols.dtype, device="cuda")   # a buffer off 16 bytes
        odd = store[1:].view(cols.shape)
        assert np.array_equal(lat.get_columns(x0, n, out=odd).cpu().numpy(), pops[..., x0:x0 + n])
        new = torch.as_tensor(np.flip(pops[..., x0:x0 + n], axis=2).copy(), device="cuda")
        lat.set_columns(x0, new)
        want = pops.copy()
        want[..., x0:x0 + n] = new.cpu().numpy()
        assert np.array_equal(lat.populations(), want)


@pytest.mark.parametrize("prec", ["f32", "f16s", "f64"])
def test_log_records_equal_the_separate_readouts(prec):
    geoms = [W.capillary_geometry(90, 14, 10, 80, 0, 12), W.capillary_geometry(400, 21, 40, 390, 1, 19),
             W.periodic_box(64, 9)]
    runs = []
    for g in geoms:
        nA, nB = W.slab_fields(g, 0, g["nx"] // 3)
        runs.append(dict(geom=g, params=W.params(1.0, 1.0, 1.0, -0.2), init=("fields", nA, nB)))
    with Lattice(runs, precision=prec, log_every=7, log_capacity=8, rho_ref=(0.04, 2.0)) as lat:
        for k in range(1, 4):
            lat.step(7)
            for r in range(3):
                rec = lat.log(r)[k]
                assert rec[0] == 7 * k
                assert np.array_equal(rec[4:], lat.mass(r))
                if geoms[r]["y_top"] >= 0:
                    assert np.array_equal(rec[1:4], lat.interface(r))
                else:
                    assert np.all(np.isnan(rec[1:4]))


@pytest.mark.parametrize("prec", ["f32", "f16s", "f64"])
@pytest.mark.parametrize("kernel", [None, (128, 4, 2, 4), (64, 8, 7, 4)])
def test_memory_off_16_bytes(monkeypatch, prec, kernel):
    """A caller's allocator may return memory on 8-byte boundaries only; column
    windows and the bulk-copy kernels read 16 bytes at a time."""
    from paper_0807_0602_gb300 import lbm
    from paper_0807_0602_gb300.build import build
    build()
    given, wrong, off = {}, [], 8

    class Off8(lbm._TorchAllocator):
        def _alloc(self, ctx, nbytes, stream):
            p = super()._alloc(ctx, nbytes + off, stream)
            if p is not None:
                given[p + off] = nbytes
                return p + off

        def _free(self, ctx, ptr, nbytes, stream):
            if given.pop(int(ptr), None) != nbytes:
                wrong.append((ptr, nbytes))
            super()._free(ctx, int(ptr) - off, nbytes + off, stream)

    with _box(64, 24, prec) as lat:
        lat.step(5)
        want = lat.populations()
    monkeypatch.setattr(lbm, "_TorchAllocator", Off8)
    kw = {} if kernel is None else dict(tile=kernel[:2], kernel=kernel[2:])
    with _box(64, 24, prec, **kw) as lat:
        info = lat.run_info()
        assert (info.base[0] | info.base[1]) % 16 == 0
        lat.step(5)
        assert np.array_equal(lat.get_columns(0, 64).cpu().numpy(), want)
        assert np.array_equal(lat.get_columns(8, 16).cpu().numpy(), want[..., 8:24])
    assert not given and not wrong   # every allocation given back as it was
