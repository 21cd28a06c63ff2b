"""3-D transfers at both sides of the slowest-axis kernel's window of 32 values:
the restriction from order 11 spans 32 (the kernel's widest form), from orders
12 and 16 35 and 47 (the row-per-thread kernel).  Tolerance: the transfer tests'
times (p / 8)^2, the growth of the derivative entries in the residual."""
import numpy as np
import pytest

pytestmark = pytest.mark.gpu
torch = pytest.importorskip("torch")

from oracle import gll as ogll  # noqa: E402
from oracle.discretize import Level  # noqa: E402
from oracle.multigrid import Hierarchy  # noqa: E402
from paper_2504_10710_gb300 import glls, inputs  # noqa: E402


@pytest.mark.parametrize("restriction", ["transpose", "interp"])
@pytest.mark.parametrize("nelem,p", [((2, 2, 3), 11), ((2, 2, 3), 12), ((1, 2, 3), 16)],
                         ids=lambda v: "x".join(map(str, v)) if isinstance(v, tuple) else f"p{v}")
def test_restrict_and_prolong(nelem, p, restriction):
    wl = inputs.random3d(nelem, p, amp=0.05, seed=62)
    prob, _ = glls.problem_for(wl, glls.SMOOTHER_FEM, glls.RESTRICT_INTERP if restriction == "interp"
                               else glls.RESTRICT_TRANSPOSE)
    xi, _ = ogll.gll(p)
    lv = Level(3, nelem, p, wl.coords(xi))
    h = Hierarchy(lv, smoother="fem", restriction=restriction)
    top = prob.levels - 1
    rng = np.random.default_rng(3)
    r, x = (np.where(lv.interior, rng.standard_normal(lv.shape), 0.0) for _ in range(2))
    lc = h.levels[top - 1]
    e = np.where(lc.interior, rng.standard_normal(lc.shape), 0.0)
    rc_ref, x_ref = h.restrict(top, r - lv.apply(x)), x + h.prolong(top, e)
    for dtype, tol in ((torch.float64, 1e-11), (torch.float32, 5e-4)):
        tol *= (p / 8) ** 2
        rd, xd, ed = (torch.from_numpy(v).to("cuda", dtype) for v in (r, x, e))
        rc = torch.full(lc.shape, 3.0, dtype=dtype, device="cuda")
        prob.restrict(top, rd, xd, rc)
        assert np.abs(rc.double().cpu().numpy() - rc_ref).max() <= tol * np.abs(rc_ref).max(), dtype
        prob.prolong_add(top, ed, xd)
        assert np.abs(xd.double().cpu().numpy() - x_ref).max() <= tol * np.abs(x_ref).max(), dtype
    prob.close()
