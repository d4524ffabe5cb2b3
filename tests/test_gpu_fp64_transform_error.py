"""The FP64 transform's error against an extended-precision FFT of the same
influence table, over the whole field.

On steep operators (k < 0) the root-mean-square error may be no larger than that of
the same transform by FP64 butterflies, which the integer passes replaced: the
bounds are that transform's errors, measured on the same fields.  Over every column
length the error stays within eps log2(points) of the field's largest value, the
growth of an FFT's rounding errors, with no allowance for steep operators on fields
that have a mean."""
import math

import numpy as np
import pytest
import scipy.fft as sf

pytestmark = pytest.mark.gpu


def dome(ny, nx):
    """A contact pressure: a rough dome on part of the grid, zero elsewhere."""
    r = np.random.Generator(np.random.PCG64(9))
    x, y = (np.arange(nx) + 0.5) / nx - 0.43, (np.arange(ny) + 0.5) / ny - 0.55
    return np.sqrt(np.maximum(0.0, 1.0 - (x[None, :] ** 2 + y[:, None] ** 2) / 0.09)) * (0.75 + 0.5 * r.random((ny, nx)))


def difference(bem_mod, nx, ny, k, p):
    """(transform - extended-precision transform, the latter), as long doubles."""
    dx = 1.0 / max(nx, ny)
    with bem_mod.Handle(nx, ny, dx, dx, k, 0.3) as h:
        T = h.influence_table().astype(np.longdouble)
        A = np.longdouble(h.info().compliance)
        u = h.convolve(p, precision="fp64").astype(np.longdouble)
    Q, P = 2 * (T.shape[0] - 1), 2 * (T.shape[1] - 1)
    iy, ix = np.minimum(np.arange(Q), Q - np.arange(Q)), np.minimum(np.arange(P), P - np.arange(P))
    hat = sf.rfft2(T[iy][:, ix], workers=8).real
    ref = sf.irfft2(sf.rfft2(p.astype(np.longdouble), s=(Q, P), workers=8) * hat, s=(Q, P), workers=8)[:ny, :nx] * A
    return u - ref, ref


@pytest.mark.parametrize("ny", [16, 32, 64, 100, 200, 400, 600, 1500, 4000])  # columns of 32 to 8192 points
@pytest.mark.parametrize("nx,k", [(24, -0.5), (70, 0.6), (300, -0.8)])
def test_error_over_column_lengths(bem_mod, cuda_ok, nx, ny, k):
    p = dome(ny, nx)
    d, ref = difference(bem_mod, nx, ny, k, p)
    assert float(np.abs(d).max()) <= 2.0 ** -52 * math.log2(16.0 * nx * ny) * float(np.abs(ref).max())


# nx, ny, k: root-mean-square error, relative to the field's, of the transform by FP64 butterflies (GB300)
BUTTERFLIES = [(64, 64, -0.5, 1.628e-16), (1501, 1100, -0.5, 2.077e-16), (1501, 1100, -0.2, 2.199e-16),
               (2048, 2048, -0.5, 2.329e-16), (2048, 2048, -0.35, 2.272e-16)]


@pytest.mark.parametrize("nx,ny,k,bound", BUTTERFLIES)
def test_error_on_steep_operators(bem_mod, cuda_ok, nx, ny, k, bound):
    d, ref = difference(bem_mod, nx, ny, k, dome(ny, nx))
    assert float(np.sqrt((d * d).sum() / (ref * ref).sum())) <= bound


@pytest.mark.parametrize("nx,ny", [(16, 16), (64, 32), (128, 256), (500, 500), (1024, 100), (40, 2000)])
@pytest.mark.parametrize("kind", ["ones", "square"])
def test_largest_growth(bem_mod, cuda_ok, nx, ny, kind):
    """Inputs of full magnitude throughout, in phase with a stage's butterflies: the integers come
    nearest to the ends of their range, and one that left it would be far off."""
    if kind == "ones":
        fields = [np.ones((ny, nx))]
    else:
        x, y = np.arange(nx)[None, :], np.arange(ny)[:, None]
        fields = [np.where(np.cos(2 * np.pi * (x * fx / 16.0 + y * fy / 16.0) + ph) >= 0, 1.0, -1.0)
                  for fx, fy, ph in ((1, 2, 0.4), (3, 1, 0.1), (2, 0, 0.8), (0, 3, 0.3), (7, 5, 0.2))]
    for p in fields:
        d, ref = difference(bem_mod, nx, ny, 0.3, p)
        assert float(np.abs(d).max()) <= 2.0 ** -52 * math.log2(16.0 * nx * ny) * float(np.abs(ref).max())
