"""Multipole moments of compact sources about an expansion origin far from the centre of the grid, and on boxes with one long
axis (several stretches of the power table in moments.cuh, powers beyond 2^53).

The rounding error has to scale with the source's own extent about the origin, not with the box: the bound takes
|x| + h/2, |y| + h/2, |z| + h/2 (the kernel counts half cells from the one nearest the origin) in the absolute value of
every term of r^l Y_lm.  Roundings per term, each 2^-53 of it: the power (1), the product and the sum of four cells (4), the
normalisation (2), the result (1); everything else is carried in pairs: 8 in all."""
from concurrent.futures import ThreadPoolExecutor
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
PI = LD("3.14159265358979323846264338327950288")


def norm(l, m):
    return np.sqrt((2 if m else 1) * LD(2 * l + 1) / (4 * PI) * LD(factorial(l - m)) / LD(factorial(l + m)))


def moments(w, x, y, z, lmax):
    """sum w r^l Y_lm over single cells, in extended precision (solid harmonics by their recurrences)."""
    r2 = x * x + y * y + z * z
    C, S = w.copy(), np.zeros_like(w)
    Q = np.zeros((lmax + 1) ** 2, LD)
    df = LD(1)
    for m in range(lmax + 1):
        if m:
            C, S = x * C - y * S, x * S + y * C
            df *= -(2 * m - 1)
        q0 = q1 = None
        for l in range(m, lmax + 1):
            q = (np.full_like(w, df) if l == m else (2 * m + 1) * z * df if l == m + 1
                 else ((2 * l - 1) * z * q1 - (l + m - 1) * r2 * q0) / (l - m))
            q0, q1 = q1, q
            Q[l * l + l + m] = (q * C).sum() * norm(l, m)
            if m:
                Q[l * l + l - m] = (q * S).sum() * norm(l, m)
    return Q


def term_sizes(w, x, y, z, lmax):
    """sum |w| over the absolute values of the terms of r^l Y_lm (Legendre's expansion in z and r^2, (x + i y)^m)."""
    r2 = x * x + y * y + z * z
    A = np.zeros((lmax + 1) ** 2)
    for l in range(lmax + 1):
        for m in range(l + 1):
            s = sum(factorial(2 * l - 2 * k) / (factorial(k) * factorial(l - k) * factorial(l - 2 * k - m))
                    * z ** (l - 2 * k - m) * r2 ** k for k in range((l - m) // 2 + 1))
            a = float((np.abs(w) * s * (x + y) ** m).sum()) * 2.0 ** -l * float(norm(l, m))
            A[l * l + l + m] = A[l * l + l - m] = a
    return A


def check(rho, h, origin, lmax, dtype):
    nz, ny, nx = rho.shape
    rho = rho.astype(dtype)
    g = hg.Grid(nx, ny, nz, h, origin, 1.0, 1.0, 0.25 * h, "f64", "multipole", lmax)
    g.set_density(torch.from_numpy(rho).cuda())
    Q = g.moments()
    g.free()
    k, j, i = np.nonzero(rho)
    w = rho[k, j, i].astype(LD) * LD(h) ** 3
    xyz = [LD(o) + (n.astype(LD) + LD(0.5)) * LD(h) for o, n in zip(origin, (i, j, k))]
    ref = moments(w, *xyz, lmax)
    bound = 8 * 2.0 ** -53 * term_sizes(w.astype(np.float64), *(np.abs(v).astype(np.float64) + 0.5 * h for v in xyz), lmax)
    err = np.abs(Q.astype(LD) - ref).astype(np.float64)
    assert (err <= bound).all(), [(q, float(err[q] / bound[q])) for q in np.nonzero(err > bound)[0]]


@pytest.mark.parametrize("at", [(0.5, 0.5, 0.5), (0.75, 0.4, 0.5), (0.9, 0.1, 0.2), (0.3, 0.95, 0.9)])
@pytest.mark.parametrize("n,h", [(64, 1.0 / 64), (75, 0.013)])
@pytest.mark.parametrize("lmax", [1, 4, 8])
@pytest.mark.parametrize("dtype", [np.float32, np.float64])
def test_compact_source_away_from_the_centre(dtype, lmax, n, h, at):
    origin = tuple(-f * n * h for f in at)
    x, y, z = (o + (np.arange(n) + 0.5) * h for o in origin)
    inside = x[None, None, :] ** 2 + y[None, :, None] ** 2 + z[:, None, None] ** 2 < (3.2 * h) ** 2
    check(np.where(inside, I.noise((n, n, n), 411, 0.5, 1.5), 0.0), h, origin, lmax, dtype)


@pytest.mark.parametrize("shape", [(300, 5, 4), (5, 300, 4), (4, 5, 300), (2100, 3, 2), (513, 2, 33)])
@pytest.mark.parametrize("lmax", [0, 4, 6, 8])
def test_boxes_with_a_long_axis(lmax, shape):
    h = 1.0 / 48
    origin = tuple(-0.6 * n * h for n in shape)
    check(I.noise(shape[::-1], 412, 0.5, 1.5), h, origin, lmax, np.float64)


@pytest.mark.parametrize("shape", [(140, 20, 7), (300, 40, 3), (520, 16, 5), (270, 1, 40), (129, 3, 23), (40, 31, 5)])
@pytest.mark.parametrize("lmax", [0, 1, 4, 8])
@pytest.mark.parametrize("dtype", [np.float32, np.float64])
def test_thin_boxes(dtype, lmax, shape):
    """Several planes of few rows in one task, and rows cut into segments where there are fewer tasks than warps."""
    h = 1.0 / 32
    check(I.noise(shape[::-1], 413, 0.5, 1.5), h, tuple(-0.45 * n * h for n in shape), lmax, dtype)


def test_threads_with_rows_of_different_lengths():
    """The table of powers takes shared memory by the row's length; grids of short and long rows share the kernel."""
    def moments_of(nx, times):
        g = hg.Grid(nx, 3, 2, 1.0 / 32, (-1.0, 0.0, 0.0), 1.0, 1.0, 1.0 / 128, "f64", "multipole", 8)
        rho = torch.from_numpy(I.noise((2, 3, nx), 414, 0.5, 1.5)).cuda()
        out = []
        for _ in range(times):
            g.set_density(rho)
            out.append(g.moments())
        g.free()
        return np.array(out)

    lengths = [2000, 320, 900, 2100]
    alone = {nx: moments_of(nx, 1)[0] for nx in lengths}
    with ThreadPoolExecutor(len(lengths)) as ex:
        for nx, out in zip(lengths, ex.map(lambda nx: moments_of(nx, 40), lengths)):
            assert (out == alone[nx]).all()
