"""The multipole moments by axis-wise Cartesian sums (moments.cuh) where the split into rows, groups of 16 cells and warps can
go wrong: rows shorter than a group, ragged rows, unaligned rows, more and fewer row groups than warps, a shifted
origin, zeros between sources, and every order.

The reference evaluates every cell's harmonics in extended precision (numpy longdouble: 64 or 113 bits) from the
coordinates origin + (i + 1/2) h.  Tolerance: the kernel rounds a handful of times per group of 16 cells and once at the
end, so it may be off by a few 2^-53 of sum |rho| h^3 |r^l Y_lm| <= sum |rho| h^3 rmax^l, taken as 16."""
from math import factorial

import numpy as np
import pytest

from paper_1602_05700_gb300 import inputs as I

pytestmark = pytest.mark.gpu

torch = pytest.importorskip("torch")
if not torch.cuda.is_available():  # pragma: no cover
    pytest.skip("needs a CUDA device", allow_module_level=True)

import paper_1602_05700_gb300 as hg  # noqa: E402

LD = np.longdouble
SHAPES = [((1, 1, 1), 0.3), ((5, 3, 2), 0.0), ((16, 33, 4), 0.0), ((17, 8, 70), 0.1), ((50, 40, 31), 0.0),
          ((36, 65, 12), -0.2)]


def moments_longdouble(rho, h, origin, lmax):
    """sum rho h^3 r^l Y_lm by the upward recurrences of the solid harmonics (real, orthonormal, Condon-Shortley)."""
    nz, ny, nx = rho.shape
    X = [LD(o) + (np.arange(n).astype(LD) + LD(0.5)) * LD(h) for o, n in zip(origin, (nx, ny, nz))]
    x, y, z = np.broadcast_arrays(X[0][None, None, :], X[1][None, :, None], X[2][:, None, None])
    r2 = x * x + y * y + z * z
    C, S = rho.astype(LD), np.zeros(rho.shape, LD)
    pi = LD("3.14159265358979323846264338327950288")
    Q = np.zeros((lmax + 1) ** 2, LD)
    for m in range(lmax + 1):
        if m:
            C, S = x * C - y * S, x * S + y * C
        df = LD(1)
        for k in range(1, m + 1):
            df *= -(2 * k - 1)
        q0 = q1 = None
        for l in range(m, lmax + 1):
            if l == m:
                q = np.full(rho.shape, df)
            elif l == m + 1:
                q = (2 * m + 1) * z * df
            else:
                q = ((2 * l - 1) * z * q1 - (l + m - 1) * r2 * q0) / (l - m)
            q0, q1 = q1, q
            K = np.sqrt((2 if m else 1) * LD(2 * l + 1) / (4 * pi) * LD(factorial(l - m)) / LD(factorial(l + m)))
            Q[l * l + l + m] = (q * C).sum() * K * LD(h) ** 3
            if m:
                Q[l * l + l - m] = (q * S).sum() * K * LD(h) ** 3
    return Q


@pytest.mark.parametrize("shape,shift", SHAPES)
@pytest.mark.parametrize("lmax", [0, 1, 2, 3, 4, 5, 6, 7, 8])
@pytest.mark.parametrize("dtype", [np.float32, np.float64])
def test_moments_against_extended_precision(dtype, lmax, shape, shift):
    nx, ny, nz = shape
    h = 1.0 / 48
    origin = (-0.5 * nx * h + shift, -0.5 * ny * h - 0.5 * shift, -0.5 * nz * h + 0.25 * shift)
    rho = I.noise(shape[::-1], 401, -1.0, 2.0).astype(dtype)
    rho[:, 1::3] = 0.0  # whole rows of vacuum
    g = hg.Grid(nx, ny, nz, h, origin, 1.0, 1.0, 0.25 * h, "f64", "multipole", lmax)
    g.set_density(torch.from_numpy(rho).cuda())
    Q = g.moments()
    g.free()
    Qx = moments_longdouble(rho, h, origin, lmax)
    rmax = np.sqrt(sum(max(abs(o), abs(o + n * h)) ** 2 for o, n in zip(origin, shape)))
    for l in range(lmax + 1):
        bound = 16 * 2.0 ** -53 * np.abs(rho.astype(np.float64)).sum() * h ** 3 * rmax ** l
        sl = slice(l * l, (l + 1) ** 2)
        err = float(np.abs(Q[sl].astype(LD) - Qx[sl]).max())
        assert err <= bound, (l, err / bound)
