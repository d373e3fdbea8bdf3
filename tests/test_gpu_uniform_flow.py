"""A uniform oblique flow is a fixed point of the predictor at orders 2 and 3: the space-time polynomial of a step is the
same at its end as at its start, exactly: in FP64, and in FP32 for the nodal forms (whose flux differences are
subtractions of rounded values), for Euler and MHD, by teams of warps and by one thread."""
import numpy as np
import pytest

from gpu_util import ensure_built, to_dev, to_host

pytestmark = pytest.mark.gpu
STATE = (1.1, 0.37, -0.53, 0.71, 2.6, 0.9, -0.4, 0.7)


@pytest.fixture(scope="module")
def ader():
    torch = pytest.importorskip("torch")
    if not torch.cuda.is_available():
        pytest.skip("no CUDA device")
    ensure_built()
    import paper_1006_2146_gb300 as p
    return p


# (form, mhd, fp32, tiled); the FP32 modal differences may be contracted with a product, to a last place of a flux
CASES = [(form, mhd, fp32, tiled) for form in ("modal", "nodal") for mhd, fp32, tiled in
         ((False, False, True), (True, False, True), (False, True, True), (False, True, False), (True, True, True))
         if form == "nodal" or not fp32]


@pytest.mark.parametrize("form,mhd,fp32,tiled", CASES)
@pytest.mark.parametrize("order", [2, 3])
def test_uniform_flow_has_no_time_modes(ader, order, form, mhd, fp32, tiled):
    import torch
    shape, nv = (4, 5, 33), 8 if mhd else 5
    full = lambda values: np.stack([np.full(shape, v) for v in values])
    U, B = full(STATE[:5]), full(STATE[5:]) if mhd else None
    s = ader.Solver(shape, order=order, form=form, fp32=fp32, mhd=mhd)
    s.set_tiled(tiled)
    s.set_dense_output(True)
    s.step(to_dev(U), 0.01, Bface=None if B is None else to_dev(B))
    ends = []
    for tau in (0.0, 1.0):
        o = torch.empty(({2: 4, 3: 10}[order], nv) + shape, dtype=torch.float64, device="cuda")
        s.dense_output(tau, o)
        ends.append(to_host(o))
    assert s.status() == 0
    s.close()
    assert np.array_equal(ends[0], ends[1])
    assert np.all(ends[0][1:] == 0.0)
