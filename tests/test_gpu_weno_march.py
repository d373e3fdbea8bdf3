"""FP64 reconstruction tiles that march through full chunks of planes: the same bits as the per-zone kernels, and the
oracle's step.

A block marches through eight planes where the grid has enough of them (tiles x nz >= 16 SMs), sliding its columns and
loading a plane ahead; smaller grids take fewer planes a block or the per-zone kernels.  Every test asserts through
ader_weno_tile_planes that its grid takes the tiles with eight planes."""
import numpy as np
import pytest

from gpu_util import ensure_built, rel_l1, to_dev, to_host
from oracle import scheme
from paper_1006_2146_gb300 import _lib, inputs

pytestmark = pytest.mark.gpu

# (nz, ny, nx): several full chunks; a last chunk of three planes; half a tile wide and half a tile deep, whose halos wrap
# more than once around the grid
SHAPES = [(96, 64, 128), (91, 64, 128), (99, 256, 16), (99, 4, 1024)]


@pytest.fixture(scope="module")
def ader():
    torch = pytest.importorskip("torch")
    if not torch.cuda.is_available():
        pytest.skip("no CUDA device")
    ensure_built()
    import paper_1006_2146_gb300 as p
    return p


def _field(shape):
    nz, ny, nx = shape
    rng = np.random.default_rng(93)
    A = rng.normal(size=(3,) + shape) * 0.01
    up = lambda a, d: np.roll(a, -1, 2 - d) - a
    B = np.stack([up(A[2], 1) * ny - up(A[1], 2) * nz, up(A[0], 2) * nz - up(A[2], 0) * nx,
                  up(A[1], 0) * nx - up(A[0], 1) * ny])
    return B / np.abs(B).max() * 0.1 + 0.5


def _step(ader, shape, U, dt, tiled, B=None, rk=False, tol=0.0, **kw):
    s = ader.Solver(shape, mhd=B is not None, **kw)
    s.set_tiled(tiled)
    assert _lib.ader_weno_tile_planes(s.h) == (8 if tiled else 0)
    if tol:
        s.set_predictor(tol, 30)
    d, b = to_dev(U), None if B is None else to_dev(B)
    (s.rk_step if rk else s.step)(d, dt, Bface=b)
    assert s.status() == 0
    s.close()
    return to_host(d), None if b is None else to_host(b)


@pytest.mark.parametrize("mhd", [False, True])
@pytest.mark.parametrize("order,form", [(2, "nodal"), (3, "modal"), (3, "nodal")])
@pytest.mark.parametrize("shape", SHAPES)
def test_marching_tiles_equal_per_zone_kernels(ader, shape, order, form, mhd):
    U, B = inputs.random_smooth(shape, seed=94 + order, amp=0.3), None
    if mhd:
        U, B = inputs.with_field(U, _field(shape))
    a, b = (_step(ader, shape, U, 2e-4, tiled, B, order=order, form=form) for tiled in (True, False))
    assert np.array_equal(a[0], b[0])
    if mhd:
        assert np.array_equal(a[1], b[1])


def test_marching_tiles_with_converged_predictor_and_rk(ader):
    shape = SHAPES[1]
    U = inputs.random_smooth(shape, seed=95, amp=0.3)
    for kw in (dict(tol=1e-13, order=3, form="nodal"), dict(rk=True, order=3, form="modal", solver="linearized"),
               dict(rk=True, order=2, form="modal")):
        a, b = (_step(ader, shape, U, 2e-4, tiled, **kw) for tiled in (True, False))
        assert np.array_equal(a[0], b[0])


def test_marching_tiles_match_the_oracle(ader):
    shape = SHAPES[2]
    U = inputs.random_smooth(shape, seed=96, amp=0.3)
    dx = tuple(1.0 / m for m in shape[::-1])
    dt = 0.5 * scheme.max_dt(U, dx, 0.4)
    want = scheme.ader_step(U, dx, dt, 3, "modal", "hll")
    assert rel_l1(_step(ader, shape, U, dt, True, order=3, form="modal")[0], want) <= 1e-12
