"""Mass and entropy of the diagnostics (fixed-point sums of csrc/entropy.cuh) against sums in
extended precision, on populations of every magnitude, sign and kind the kernels tell apart."""
import numpy as np
import pytest
import torch

pytestmark = pytest.mark.gpu


@pytest.fixture(scope="module")
def E():
    from paper_2605_01774_gb300 import elbm
    elbm.lib()
    return elbm


def _weights(d):
    c = np.array(np.meshgrid(*[[-1, 0, 1]] * d, indexing="ij")).reshape(d, -1)
    m = (c != 0).sum(0).astype(np.longdouble)
    return (np.longdouble(2) / 3) ** (d - m) * (np.longdouble(1) / 6) ** m


def _values(kind, shape, dtype, seed):
    """Populations [Q, N]; `kind` says which part of the range they test."""
    g = np.random.default_rng(seed)
    w = _weights(2 if shape[0] == 9 else 3).astype(np.float64)[:, None]
    if kind == "near_equilibrium":                    # v close to W: the logarithm is near zero
        v = w * (1 + 1e-3 * g.standard_normal(shape))
    elif kind == "weights":                           # the same few values everywhere
        v = np.broadcast_to(w, shape).copy()
    elif kind == "spread":                            # neighbours of very different size, some negative or zero
        big = 30 if dtype == np.float32 else 250
        v = 10.0 ** g.uniform(-big, big, shape) * np.where(g.random(shape) < 0.2, -1, 1)
        v[g.random(shape) < 0.05] = 0
    elif kind == "powers":                            # mantissas at both ends of their range
        v = 2.0 ** g.integers(-20, 20, shape)
        v = np.where(g.random(shape) < 0.5, v, np.nextafter(v.astype(dtype), dtype(0)))
    elif kind == "tiny":                              # below the range of a scaled sum (FP64) or of normal values
        v = w * (1e-37 if dtype == np.float32 else 1e-306) * (1 + g.random(shape))
    else:                                             # "negative": no population is positive
        v = -w * g.random(shape)
    return v.astype(dtype)


def _reference(v):
    if v.dtype == np.float32:                         # FP32 arithmetic flushes subnormals to zero
        v = np.where(np.abs(v) < np.finfo(np.float32).tiny, np.float32(0), v)
    x, w = v.astype(np.longdouble), _weights(2 if v.shape[0] == 9 else 3)[:, None]
    safe = np.where(x > 0, x, 1)
    t = np.where(x > 0, x * np.log(safe / w), 0)
    # the terms' own size bounds the rounding: 2^-53 each for a value and its logarithm, doubled
    # for the additions of a thread's and a block's nodes
    size = np.where(x > 0, x * (1 + np.abs(np.log(safe / w))), 0).sum()
    return x.sum(), t.sum(), 4 * 2.0 ** -53 * np.abs(x).sum(), 4 * 2.0 ** -53 * size


@pytest.mark.parametrize("kind", ["near_equilibrium", "weights", "spread", "powers", "tiny", "negative"])
@pytest.mark.parametrize("prec", ["f32", "f64"])
@pytest.mark.parametrize("dims", [(3, 1, 1), (33, 20, 13)])
def test_sums_3d(E, dims, prec, kind):
    dtype = np.float32 if prec == "f32" else np.float64
    n = int(np.prod(dims))
    v = _values(kind, (27, n), dtype, 7)
    lat = E.Lattice(dims, prec)
    E.elbm_write_populations(lat.h, v)
    d = E.elbm_reduce(lat.h)
    lat.close()
    mass, ent, em, ee = _reference(v)
    assert abs(np.longdouble(d["mass"]) - mass) <= em
    assert abs(np.longdouble(d["entropy"]) - ent) <= ee
    flushed = np.where(np.abs(v) < np.finfo(np.float32).tiny, 0, v) if prec == "f32" else v
    assert d["gmin"] == float(flushed.min())


@pytest.mark.parametrize("kind", ["near_equilibrium", "spread", "powers"])
@pytest.mark.parametrize("prec", ["f32", "f64"])
@pytest.mark.parametrize("dims", [(5, 3), (700, 500), (1200, 700)])
def test_sums_2d(E, dims, prec, kind):
    """Fewer nodes than a block, one node per thread, and the three-nodes-at-once loop with its rest."""
    dtype = np.float32 if prec == "f32" else np.float64
    v = _values(kind, (9, dims[0] * dims[1]), dtype, 9)
    lat = E.Lattice2D(dims, prec)
    E.elbm2d_write_populations(lat.h, v)
    d = E.elbm2d_reduce(lat.h)
    mass, ent, em, ee = _reference(v)
    assert abs(np.longdouble(d["mass"]) - mass) <= em
    assert abs(np.longdouble(d["entropy"]) - ent) <= ee
    assert d["gmin"] == float(v.min())


@pytest.mark.parametrize("prec", ["f32", "f64"])
def test_faces_and_source(E, prec):
    """The pulled form: Dirichlet faces, and a source half-step in the state."""
    dims, n = (13, 6, 5), 13 * 6 * 5
    v = _values("near_equilibrium", (27, n), np.float64, 3)
    src = np.random.default_rng(4).random(n).astype(np.float32) * np.float32(1e-3)
    for source in (None, src):
        lat = E.Lattice(dims, prec, bc=(1.3, 0.8))
        if source is not None:
            E.elbm_set_source(lat.h, source)
        E.elbm_write_populations(lat.h, v)
        d = E.elbm_reduce(lat.h)
        back = np.empty((27, n))
        E.elbm_read_populations(lat.h, back)
        lat.close()
        mass, ent, em, ee = _reference(back)
        # an FP32 state with a source is read back rounded to FP32, and summed unrounded
        rough = 2.0 ** -24 * np.abs(back).sum() if prec == "f32" and source is not None else 0.0
        assert abs(np.longdouble(d["mass"]) - mass) <= em + rough
        assert abs(np.longdouble(d["entropy"]) - ent) <= ee + 4 * rough


def test_non_finite_values_are_counted_and_left_out(E):
    v = _values("near_equilibrium", (27, 64), np.float32, 5)
    bad = v.copy()
    bad[3, 7], bad[20, 7], bad[13, 40] = np.nan, np.inf, -np.inf
    lat = E.Lattice((8, 8, 1), "f32")
    E.elbm_write_populations(lat.h, bad)
    d = E.elbm_reduce(lat.h, allow_nonfinite=True)
    lat.close()
    assert d["status"] == 6
    ok = np.isfinite(bad)
    mass, ent, em, ee = _reference(np.where(ok, bad, 0).astype(np.float32))
    assert abs(np.longdouble(d["mass"]) - mass) <= em
    assert abs(np.longdouble(d["entropy"]) - ent) <= ee
    assert d["gmin"] == float(bad[ok].min())
