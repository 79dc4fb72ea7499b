"""The FP64 stage's integer comparisons (limiter, wave speeds, floors) on values where a comparison can go wrong: zeros of
both signs, equal neighbours, infinities, NaN, subnormal differences, vacuum and negative pressure -- the same cells as
the oracle's plain comparisons, bit for bit, with NaN in the same places."""
import numpy as np
import pytest

import oracle as O
from paper_1602_05700_gb300 import inputs as I

pytestmark = pytest.mark.gpu

torch = pytest.importorskip("torch")
if not torch.cuda.is_available():  # pragma: no cover
    pytest.skip("needs a CUDA device", allow_module_level=True)

import paper_1602_05700_gb300 as hg  # noqa: E402


@pytest.mark.parametrize("floors", [(0.0, 0.0), (1e-3, 1e-4)])
@pytest.mark.parametrize("special", [0.0, -0.0, np.inf, -np.inf, np.nan, 5e-324, -1.0, 1e300])
def test_fp64_stage_with_special_values(special, floors):
    shape = (6, 11, 37)
    nz, ny, nx = shape
    W = I.hydro_noise(shape, 71)
    W[:, :, :, 10:14] = W[:, :1, :1, 10:11]      # a uniform slab: every difference zero
    W[1:4, :, :, 20] *= -1.0                      # sign changes
    rng = np.random.default_rng(72)
    for q in range(5):                            # the special value in a few cells of every field
        for _ in range(3):
            W[q, rng.integers(nz), rng.integers(ny), rng.integers(nx)] = special
    h, gamma = 1.0 / nx, 5.0 / 3.0
    H = hg.Hydro(nx, ny, nz, h, gamma, *floors, dtype="f64")
    hgo = O.HydroGrid(nx, ny, nz, h, gamma, *floors)
    with np.errstate(all="ignore"):
        H.set_primitive(W)
        U = O.hydro_cons(hgo, W)
        for _ in range(2):
            H.step(1e-4)
            O.hydro_step(hgo, U, 1e-4)
    got = H.state("cpu").numpy()
    assert np.array_equal(got, U, equal_nan=True)
