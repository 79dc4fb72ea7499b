"""Calls that leave the flat sweep at 11.5 million float cells, at their true size: the batch's class of large float grids (TMA-staged
entries with their tensor maps in the table, on the second stream, beside flat entries of both precisions) and the
adjoint's reverse sub-step with its running sum as a pass of its own."""
import numpy as np
import pytest

pytestmark = pytest.mark.gpu

torch = pytest.importorskip("torch")
if not torch.cuda.is_available():  # pragma: no cover
    pytest.skip("needs a CUDA device", allow_module_level=True)

import paper_1602_05700_gb300 as hg  # noqa: E402
from tests.test_gpu_parity import robin_cfl  # noqa: E402

LARGE = 11500000


def rand(shape, seed, lo, hi):
    gen = torch.Generator(device="cuda").manual_seed(seed)
    return torch.empty(shape, dtype=torch.float64, device="cuda").uniform_(lo, hi, generator=gen)


def grid(shape, prec, bc, seed=None, lmax=0):
    nx, ny, nz = shape
    h = 1.0 / max(shape)
    dt = (robin_cfl(nx, ny, nz, h) if bc == "robin" else 0.5) * h / np.sqrt(3.0)
    g = hg.Grid(nx, ny, nz, h, (-0.5 * nx * h, -0.5 * ny * h, -0.5 * nz * h), 1.0, 1.0, dt, prec, bc, lmax)
    if seed is not None:
        phi = rand(shape[::-1], seed, -1.0, -0.5)
        g.set_density(rand(shape[::-1], seed + 1, 0.0, 2.0))
        g.set_phi(phi, phi + 1e-3 * rand(shape[::-1], seed + 2, -1.0, 1.0))
    return g


def blob(g):
    return g.save_state(torch.empty(g.state_bytes(), dtype=torch.uint8, device="cuda"))


BIG = [((227, 226, 225), "f32k", "robin"), ((232, 224, 224), "f32k", "periodic"), ((256, 225, 200), "f32k", "dirichlet")]
SMALL = [((48, 40, 33), "f64", "robin"), ((64, 64, 64), "f32k", "periodic"), ((101, 77, 78), "f64", "periodic"),
         ((33, 47, 50), "f32k", "robin")]


@pytest.mark.parametrize("split", [None, False, True])
@pytest.mark.parametrize("specs", [SMALL + BIG, BIG[:1], SMALL[:1] + BIG[1:2], SMALL[1:2] + BIG[2:]],
                         ids=["mixed", "large alone", "large and f64", "large and flat float"])
def test_batch_with_large_grids_equals_individual_steps(specs, split):
    assert all(np.prod(s[0]) > LARGE for s in BIG)
    a, b = ([grid(*s, seed=10 * i) for i, s in enumerate(specs)] for _ in range(2))
    batch = hg.Batch(a)
    batch.set_split(split)
    batch.step(27)  # autotunes on its first sub-steps
    batch.step(4)   # replays a graph from the other parity
    for g in b:
        g.step(31)
    for ga, gb in zip(a, b):
        assert torch.equal(blob(ga), blob(gb)), (ga.nx, ga.ny, ga.nz)
    batch.free()
    for g in a + b:
        g.free()


@pytest.mark.parametrize("bc", ["dirichlet", "periodic"])
def test_large_adjoint_sums_the_levels_of_the_reverse_run(bc):
    """The reverse recursion of a terminal loss is the sub-step itself with no source, from lambda^T = v and lambda^{T+1} = 0:
    a second grid gives its levels, added here in FP64.  The float pair that holds the sum rounds near 2^-46."""
    shape, T = BIG[1][0], 6
    v = rand(shape[::-1], 71, -1.0, 1.0).float().double()
    g = grid(shape, "f32k", bc)
    got = g.adjoint(v, T)
    lam = grid(shape, "f32k", bc)
    lam.set_density(torch.zeros_like(v))
    lam.set_phi(v, torch.zeros_like(v))
    total = torch.zeros_like(v)
    for m in range(T):
        total += lam.phi(torch.float64)
        lam.step(1)
    want = -(g.dt * g.dt) * 4.0 * np.pi * total
    if bc == "periodic":
        want -= want.mean()
    assert (got - want).abs().max().item() <= T * 2.0 ** -44 * want.abs().max().item()
    g.free()
    lam.free()


def test_large_robin_adjoint_is_linear():
    """Doubling the injection doubles the gradient exactly (a power of two commutes with every rounding)."""
    shape = BIG[0][0]
    v = rand(shape[::-1], 72, -1.0, 1.0).float().double()
    g = grid(shape, "f32k", "robin")
    a, b = g.adjoint(v, 7), g.adjoint(2.0 * v, 7)
    assert torch.equal(2.0 * a, b) and a.abs().max().item() > 0.0
    g.free()
