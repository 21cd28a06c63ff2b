"""Device memory of fixed-order summation: the element-result scratch exists for
the levels whose applies can write it (2-D orders up to 16, 3-D up to 8, fewer
than 1024 elements along an axis) and for no other."""
import ctypes

import pytest

torch = pytest.importorskip("torch")

from paper_2504_10710_gb300 import glls, inputs  # noqa: E402

CASES = [((2, 3), 17, glls.SMOOTHER_GLL), ((1, 2), 36, glls.SMOOTHER_GLL), ((2, 3), 16, glls.SMOOTHER_GLL),
         ((2, 1, 2), 9, glls.SMOOTHER_GLL), ((2, 2, 3), 8, glls.SMOOTHER_GLL), ((1030, 2), 2, glls.SMOOTHER_FEM)]

IDS = lambda v: "x".join(map(str, v)) if isinstance(v, tuple) else str(v)  # noqa: E731


def _orders(nelem, p):
    """Orders of the levels: halved down to 1, or 2 where an axis has one element
    (p = 1 then has no interior unknown)."""
    last = 1 if min(nelem) > 1 else 2
    orders = [p]
    while orders[-1] > last:
        orders.append(max(last, orders[-1] // 2))
    return orders


def _scratch_bytes(nelem, p):
    """Element results of the levels in both precisions."""
    if max(nelem) >= 1024:
        return 0
    elements = 1
    for n in nelem:
        elements *= n
    limit = 16 if len(nelem) == 2 else 8
    return sum(12 * elements * (q + 1) ** len(nelem) for q in _orders(nelem, p) if q <= limit)


@pytest.mark.gpu
@pytest.mark.parametrize("nelem,p,smoother", CASES, ids=IDS)
def test_allocated(nelem, p, smoother):
    mk = inputs.random2d if len(nelem) == 2 else inputs.random3d
    wl = mk(nelem, p, amp=0.05, seed=1)
    held = []
    for s in (glls.SUM_COLORED, glls.SUM_ATOMIC):
        prob, _ = glls.problem_for(wl, smoother, summation=s)
        clone = prob.clone(nrhs=3)
        held.append((prob.info.instance_bytes, clone.info.instance_bytes))
        levels = prob.levels
        clone.close()
        prob.close()
    want = _scratch_bytes(nelem, p)
    assert levels == len(_orders(nelem, p))
    assert held[0][0] - held[1][0] == want
    assert held[0][1] - held[1][1] == 3 * want


@pytest.mark.parametrize("nelem,p,smoother", CASES, ids=IDS)
def test_estimated(nelem, p, smoother):
    out = []
    for s in (glls.SUM_COLORED, glls.SUM_ATOMIC):
        mk = inputs.random2d if len(nelem) == 2 else inputs.random3d
        wl = mk(nelem, p, amp=0.0, seed=1)
        xi, _ = glls.gll(p)
        desc, keep = glls.mesh_desc(len(nelem), nelem, p, wl.coords(xi), smoother, summation=s)
        n = ctypes.c_size_t()
        assert glls.lib().glls_estimate_bytes(ctypes.byref(desc), ctypes.byref(n)) == glls.OK
        out.append(n.value)
    assert abs((out[0] - out[1]) - _scratch_bytes(nelem, p)) <= 2     # the two totals are truncated to bytes
