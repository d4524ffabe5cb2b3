"""The FP64 transform (64-bit block fixed-point passes) against the direct sum of
Eq. 7 in extended precision: tile edges, ragged and elongated grids, the largest
column length, fields of a wide range of magnitudes, and NaN / infinity / zero."""
import math

import numpy as np
import pytest

pytestmark = pytest.mark.gpu


def field(kind, ny, nx, seed):
    r = np.random.Generator(np.random.PCG64(seed))
    if kind == "noise":
        return r.standard_normal((ny, nx))
    if kind == "checker":  # no mean: the low frequencies hold only rounding errors of the rest
        return r.random((ny, nx)) * (1.0 - 2.0 * (np.add.outer(np.arange(ny), np.arange(nx)) % 2))
    if kind == "rows":  # row magnitudes over 40 decades
        return r.standard_normal((ny, nx)) * 10.0 ** (-40.0 * r.random((ny, 1)))
    if kind == "tiny":  # few values, near the bottom of the normal range
        return 1e-290 * r.standard_normal((ny, nx)) * (r.random((ny, nx)) < 0.05)
    p = np.zeros((ny, nx))
    p[ny // 2, nx // 3] = 1.0
    return p


@pytest.mark.parametrize("nx,ny,k", [(2, 2, 0.5), (17, 16, -0.4), (33, 64, 0.0), (100, 257, 0.6), (513, 40, -0.6),
                                     (24, 2049, 0.3), (1025, 31, -0.8)])
@pytest.mark.parametrize("kind", ["noise", "checker", "rows", "tiny", "delta"])
def test_transform_vs_direct_sum(bem_mod, cuda_ok, nx, ny, k, kind):
    p = field(kind, ny, nx, 11)
    scale = np.longdouble(1e290) if kind == "tiny" else np.longdouble(1)
    with bem_mod.Handle(nx, ny, 1.0 / nx, 1.0 / nx, k, 0.3) as h:
        inf = h.info()
        K = h.influence_table().astype(np.longdouble)
        u = h.convolve(p, precision="fp64")
    r = np.random.Generator(np.random.PCG64(5))
    pts = [(int(r.integers(ny)), int(r.integers(nx))) for _ in range(24)]
    ps = p.astype(np.longdouble) * scale
    ref = np.array([(K[np.abs(np.arange(ny) - y)][:, np.abs(np.arange(nx) - x)] * ps).sum()
                    for y, x in pts]) * np.longdouble(inf.compliance)
    got = np.array([u[y, x] for y, x in pts]).astype(np.longdouble) * scale
    # an FFT's error is relative to the whole field, of the order of eps log2(points); steep
    # spectra (k < 0) amplify what rounding leaves at the low frequencies of a field without mean
    bound = 2.0 ** -52 * math.log2(inf.Px * inf.Py) * max(1.0, min(nx, ny) ** -k)
    peak = max(float(np.abs(ref).max()), float(K[0, 0] * np.abs(ps).max() * np.longdouble(inf.compliance)))
    assert float(np.abs(got - ref).max()) <= bound * peak


@pytest.mark.parametrize("bad", [math.nan, math.inf, -math.inf])
def test_nonfinite_input_reaches_every_output(bem_mod, cuda_ok, bad):
    p = field("noise", 50, 40, 3)
    p[49, 39] = bad
    with bem_mod.Handle(40, 50, 0.02, 0.02, 0.2, 0.3) as h:
        u = h.convolve(p, precision="fp64")
        assert not np.isfinite(u).any()
        assert np.array_equal(h.convolve(np.zeros((50, 40)), precision="fp64"), np.zeros((50, 40)))
        assert np.isfinite(h.convolve(field("noise", 50, 40, 3), precision="fp64")).all()
