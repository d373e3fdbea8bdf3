"""Tuned launch shapes of a batch: phases whose kernel has one shape (predictors by teams of warps) are not listed, the
others of every group are, and a tuned batch steps as its problems do."""
import pytest

from gpu_util import ensure_built, to_dev, to_host
from paper_1006_2146_gb300 import _lib, inputs

pytestmark = pytest.mark.gpu
PREDICT = 5               # BatchPhase PH_PREDICT

# (order, nodal, team of warps) of Euler groups; FP32
GROUPS = [(2, 0, False), (3, 1, False), (4, 0, True), (4, 1, False)]


@pytest.fixture(scope="module")
def ader():
    torch = pytest.importorskip("torch")
    if not torch.cuda.is_available():
        pytest.skip("no CUDA device")
    ensure_built()
    import paper_1006_2146_gb300 as p
    return p


def test_one_shape_predictors_are_not_tuned(ader):
    import torch
    n = 12
    grid = (n, n, n, 1 / n, 1 / n, 1 / n)
    U = inputs.random_smooth((n, n, n), seed=40, amp=0.2)
    flags = [_lib.ADER_FP32_BULK | (_lib.ADER_NODAL if nodal else 0) for _, nodal, _ in GROUPS]
    orders = [o for o, _, _ in GROUPS]
    b = _lib.ader_batch_create([grid] * 4, orders, [1.4] * 4, [_lib.ADER_HLL] * 4, flags)
    Us = [to_dev(U) for _ in GROUPS]
    _lib.ader_batch_tune(b, Us, [None] * 4)
    chosen = _lib.ader_batch_tuning(b)
    listed = {g for g, phase, _, _ in chosen if phase == PREDICT}
    assert listed == {g for g, (_, _, team) in enumerate(GROUPS) if not team}
    assert {g for g, _, _, _ in chosen} == {0, 1, 2, 3}
    _lib.ader_batch_step(b, Us, [None] * 4, torch.full((4,), 1e-3, dtype=torch.float64, device="cuda"))
    rc, _ = _lib.ader_batch_status(b, 4)
    assert rc == 0
    for (order, nodal, _), u in zip(GROUPS, Us):
        s = ader.Solver((n, n, n), order=order, form="nodal" if nodal else "modal", fp32=True)
        d = to_dev(U)
        s.step(d, 1e-3)
        assert s.status() == 0
        assert abs(to_host(d) - to_host(u)).max() <= 1e-6 * abs(U).max()
        s.close()
    _lib.ader_batch_destroy(b)
