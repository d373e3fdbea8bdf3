"""FP64 reconstruction tiles on grids that are no multiple of a tile: the same bits as the per-zone kernels.

The tiles take any grid with enough columns to fill them (a block's columns past the grid's end only serve as
halos), so ragged x and y sides, sides shorter than a tile, and every count of planes per block are compared with
ader_set_tiled(0), which takes the per-zone kernels."""
import numpy as np
import pytest

from gpu_util import ensure_built, to_dev, to_host
from oracle import scheme
from paper_1006_2146_gb300 import inputs

pytestmark = pytest.mark.gpu


@pytest.fixture(scope="module")
def ader():
    torch = pytest.importorskip("torch")
    if not torch.cuda.is_available():
        pytest.skip("no CUDA device")
    ensure_built()
    import paper_1006_2146_gb300 as p
    return p


# (nz, ny, nx): one plane over a block's last column and row, one short of them, one tile wide, a thin slab
SHAPES = [(90, 33, 65), (120, 31, 63), (160, 16, 24), (2, 250, 255)]


@pytest.mark.parametrize("mhd", [False, True])
@pytest.mark.parametrize("order", [2, 3])
@pytest.mark.parametrize("shape", SHAPES)
def test_ragged_tiles_equal_per_zone_kernels(ader, shape, order, mhd):
    nz, ny, nx = shape
    U = inputs.random_smooth(shape, seed=90 + order, amp=0.3)
    B = None
    if mhd:
        rng = np.random.default_rng(91)
        A = rng.normal(size=(3,) + shape) * 0.02
        up = lambda a, d: np.roll(a, -1, 2 - d) - a
        B = np.stack([up(A[2], 1) * ny - up(A[1], 2) * nz, up(A[0], 2) * nz - up(A[2], 0) * nx,
                      up(A[1], 0) * nx - up(A[0], 1) * ny]) + 0.5
        U, B = inputs.with_field(U, B)
    dt = 0.5 * scheme.max_dt(U, (1 / nx, 1 / ny, 1 / nz), 0.4, Bface=B)
    out = []
    for tiled in (True, False):
        s = ader.Solver(shape, order=order, form="modal", mhd=mhd)
        s.set_tiled(tiled)
        d, b = to_dev(U), None if B is None else to_dev(B)
        s.step(d, dt, Bface=b)
        out.append((to_host(d), None if b is None else to_host(b)))
        s.close()
    assert np.array_equal(out[0][0], out[1][0])
    if mhd:
        assert np.array_equal(out[0][1], out[1][1])
