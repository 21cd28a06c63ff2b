"""Line-block solves whose segment operators do not fit in shared memory beside
the line's values (the run-time-order kernel then reads them from global
memory), and the sizes just inside the limit: with one line per CTA the limit of
200 KB lies between orders 38 and 39 in FP64 and 54 and 55 in FP32 on lines of
one or two elements, and at order 16 between 96 and 97 elements in FP64.

Tolerance: as in the other line-form tests (ten times 1e-12 in FP64 and 5e-5 in
FP32 relative to the largest entry, or 8 kappa eps of the line), the first of
the two times (p / 8)^2: the set-up's geometry, which the two sides round
separately, is built from derivative entries that grow with p^2."""
import numpy as np
import pytest

pytestmark = pytest.mark.gpu
torch = pytest.importorskip("torch")

from oracle import gll as ogll  # noqa: E402
from oracle.discretize import Level  # noqa: E402
from oracle.lines import BlockLineSmoother, line_block_bands  # noqa: E402
from paper_2504_10710_gb300 import glls, inputs  # noqa: E402


@pytest.fixture(scope="module", autouse=True)
def _built():
    import __graft_entry__
    __graft_entry__.build()


def _condition(ab):
    """Condition number of each banded line matrix."""
    nl, w1, n = ab.shape
    T = np.zeros((nl, n, n))
    for o in range(w1):
        for j in range(o, n):
            T[:, j - o, j] = T[:, j, j - o] = ab[:, w1 - 1 - o, j]
    return np.linalg.cond(T)


@pytest.mark.parametrize("nelem,p", [((1, 2), 38), ((2, 1), 39), ((2, 1), 54), ((1, 2), 55), ((96, 1), 16),
                                     ((1, 97), 16)],
                         ids=lambda v: "x".join(map(str, v)) if isinstance(v, tuple) else f"p{v}")
def test_solve_and_update(nelem, p):
    wl = inputs.random2d(nelem, p, amp=0.05, seed=33)
    prob, _ = glls.problem_for(wl)
    xi, _ = ogll.gll(p)
    lv = Level(2, nelem, p, wl.coords(xi))
    Ae = lv.element_matrices()
    top = prob.levels - 1
    rng = np.random.default_rng(6)
    r, y, x = (np.where(lv.interior, rng.standard_normal(lv.shape), 0.0) for _ in range(3))
    for s in range(2):
        ab, _ = line_block_bands(lv, s, Ae=Ae)
        sm = BlockLineSmoother(lv, s, Ae=Ae)
        kappa = _condition(ab)
        for dtype, eps in ((torch.float64, 2.0 ** -53), (torch.float32, 2.0 ** -24)):
            rd, yd, xd = (torch.from_numpy(v).to("cuda", dtype) for v in (r, y, x))
            got = torch.full_like(xd, float("nan"))
            prob.line_solve(top, s, rd, got)
            pairs = [(got.double().cpu().numpy(), sm.apply_inverse(rd.double().cpu().numpy()))]
            g, x0 = (rd.double() - yd.double()).cpu().numpy(), xd.double().cpu().numpy()
            prob.line_update(top, s, 0.5, rd, yd, xd)
            pairs.append((xd.double().cpu().numpy() - x0, 0.5 * sm.apply_inverse(g)))
            for a, b in pairs:
                a, b = a.ravel()[sm.lin], b.ravel()[sm.lin]
                floor = (1e-11 if dtype == torch.float64 else 5e-4) * (p / 8) ** 2 * np.abs(b).max()
                bound = np.maximum(8 * kappa * eps * np.abs(b).max(1), floor)
                assert np.all(np.abs(a - b).max(1) <= bound), (s, dtype, (np.abs(a - b).max(1) / bound).max())
            seam = np.any([i % p == 0 for i in np.indices(lv.shape)], axis=0) & lv.interior
            assert np.all(yd.cpu().numpy()[seam] == 0.0)
    prob.close()
