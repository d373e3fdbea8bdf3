"""The predictor and faces computed by teams of warps (32 zones a block): zone counts around one block, every order,
form, solver and physics, against the oracle; and converged predictors, whose zones stop after different iterations
while their team goes on.

Bars: FP64 1e-12, FP32 1e-5 relative L1 after one step.  The nodal fourth-order formulas amplify the rounding of a
node about 20 times and a step adds some tens of roundings: 20 x 50 x 1.1e-16 = 1e-13 in FP64, and 20 x 6e-8 = 1.2e-6
times the CFL number's share of a flux in FP32.
"""
import itertools

import numpy as np
import pytest

from gpu_util import ensure_built, rel_l1, to_dev, to_host
from oracle import scheme
from paper_1006_2146_gb300 import inputs

pytestmark = pytest.mark.gpu
SHAPES = [(1, 1, 31), (2, 4, 4), (3, 1, 11), (3, 5, 7)]          # 31, 32, 33 and 105 zones


@pytest.fixture(scope="module")
def ader():
    torch = pytest.importorskip("torch")
    if not torch.cuda.is_available():
        pytest.skip("no CUDA device")
    ensure_built()
    import paper_1006_2146_gb300 as p
    return p


def _state(shape, mhd, seed=5):
    nz, ny, nx = shape
    U = inputs.random_smooth(shape, seed=seed, amp=0.2, kmax=2)
    if not mhd:
        return U, None
    rng = np.random.default_rng(seed)
    A = rng.normal(size=(3,) + shape) * 0.05
    up = lambda a, d: np.roll(a, -1, 2 - d) - a
    B = np.stack([up(A[2], 1) * ny - up(A[1], 2) * nz, up(A[0], 2) * nz - up(A[2], 0) * nx,
                  up(A[1], 0) * nx - up(A[0], 1) * ny]) / max(shape) + 0.7
    return inputs.with_field(U, B)


@pytest.mark.parametrize("mhd,fp32", [(False, False), (True, False), (False, True), (True, True)])
@pytest.mark.parametrize("order,form", list(itertools.product((2, 3, 4), ("modal", "nodal"))))
def test_block_remainders(ader, order, form, mhd, fp32):
    for n, shape in enumerate(SHAPES):
        solver = ("hll", "linearized")[n % 2]
        U, B = _state(shape, mhd)
        dx = tuple(1.0 / m for m in shape[::-1])
        dt = 0.5 * scheme.max_dt(U, dx, 0.4, Bface=B)
        want = scheme.ader_step(U, dx, dt, order, form, solver, Bface=B)
        s = ader.Solver(shape, order=order, form=form, solver=solver, fp32=fp32, mhd=mhd)
        d, b = to_dev(U), None if B is None else to_dev(B)
        s.step(d, dt, Bface=b)
        assert s.status() == 0
        bar = 1e-5 if fp32 else 1e-12
        assert rel_l1(to_host(d), want[0] if mhd else want) <= bar, (shape, solver)
        if mhd:
            assert rel_l1(to_host(b), want[1]) <= bar, (shape, solver)
        s.close()


@pytest.mark.parametrize("order,form", list(itertools.product((2, 3, 4), ("modal", "nodal"))))
def test_converged_zones_of_one_team(ader, order, form):
    """Uniform zones converge at once, perturbed ones beside them take more iterations."""
    shape = (3, 5, 7)
    U, _ = _state(shape, False)
    U[:, 0] = U[:, :1, :1, :1].mean(axis=(1, 2, 3))[:, None, None]
    dx = tuple(1.0 / m for m in shape[::-1])
    dt = 0.5 * scheme.max_dt(U, dx, 0.4)
    want, iters = scheme.ader_step(U, dx, dt, order, form, "hll", tol=1e-10, return_iters=True)
    s = ader.Solver(shape, order=order, form=form)
    s.set_predictor(1e-10, 50)
    d = to_dev(U)
    s.step(d, dt)
    assert s.status() == 0
    assert rel_l1(to_host(d), want) <= 1e-12
    total, largest, capped = s.predictor_stats()
    assert iters.min() < iters.max() or order == 2
    # a change within an ulp of the tolerance may go either way in a zone or two
    assert capped == 0 and abs(total - int(iters.sum())) <= 2 and abs(largest - int(iters.max())) <= 1
    s.close()
