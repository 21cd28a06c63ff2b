"""Line-block solves at the sizes where their forms change: one segment per
line, vertex systems that fill their lane groups exactly or by one more (16,
32, 64 vertices), lines per CTA that do not divide the line count, the largest
compile-time order and the run-time order.

Tolerance: the parity tests' for the same call (ten times 1e-12 in FP64 and
5e-5 in FP32, relative to the largest entry; it covers the rounding of the
set-up's geometry, which the two sides do not share), or 8 kappa eps per line
where a stretched line's condition number kappa makes that more."""
import numpy as np
import pytest

pytestmark = pytest.mark.gpu
torch = pytest.importorskip("torch")

from oracle.discretize import Level  # noqa: E402
from oracle.lines import BlockLineSmoother, line_block_bands  # noqa: E402
from oracle import gll as ogll  # noqa: E402
from paper_2504_10710_gb300 import glls, inputs  # noqa: E402

GRIDS = [((2, 16), 2), ((17, 3), 5), ((33, 2), 2), ((34, 2), 3), ((65, 2), 2), ((3, 33), 8), ((2, 66), 4),
         ((1, 4), 7), ((5, 4), 12), ((3, 5), 9), ((2, 3), 13), ((3, 16, 2), 3), ((17, 2, 2), 2), ((2, 3, 9), 6)]


def _condition(ab):
    """Condition number of each banded line matrix."""
    nl, w1, n = ab.shape
    T = np.zeros((nl, n, n))
    for o in range(w1):
        for j in range(o, n):
            T[:, j - o, j] = T[:, j, j - o] = ab[:, w1 - 1 - o, j]
    return np.linalg.cond(T)


@pytest.mark.parametrize("nelem,p", GRIDS, ids=["x".join(map(str, g)) + f"_p{p}" for g, p in GRIDS])
def test_line_update_and_solve(nelem, p):
    wl = inputs.random2d(nelem, p, amp=0.1, seed=31) if len(nelem) == 2 else inputs.random3d(nelem, p, amp=0.1, seed=32)
    prob, _ = glls.problem_for(wl)
    xi, _ = ogll.gll(p)
    lv = Level(len(nelem), nelem, p, wl.coords(xi))
    top = prob.levels - 1
    rng = np.random.default_rng(5)
    field = lambda: np.where(lv.interior, rng.standard_normal(lv.shape), 0.0)  # noqa: E731
    for s in range(lv.dim):
        ab, _ = line_block_bands(lv, s, Ae=lv.element_matrices())
        sm = BlockLineSmoother(lv, s, Ae=lv.element_matrices())
        kappa = _condition(ab)
        r, y, x = field(), field(), field()
        for dtype, eps in ((torch.float64, 2.0 ** -53), (torch.float32, 2.0 ** -24)):
            rd, yd, xd = (torch.from_numpy(v).to("cuda", dtype) for v in (r, y, x))
            g = (rd.double() - yd.double()).cpu().numpy()
            ref = sm.apply_inverse(g)
            got = torch.zeros_like(xd)
            prob.line_solve(top, s, rd, got)
            pairs = [(got.double().cpu().numpy(), sm.apply_inverse(rd.double().cpu().numpy()), 1.0)]
            x0 = xd.double().cpu().numpy()
            prob.line_update(top, s, 0.5, rd, yd, xd)
            pairs.append((xd.double().cpu().numpy() - x0, 0.5 * ref, 0.5))
            for a, b, scale in pairs:
                a, b = a.ravel()[sm.lin], b.ravel()[sm.lin]
                floor = (1e-11 if dtype == torch.float64 else 5e-4) * np.abs(b).max()
                bound = np.maximum(8 * kappa * eps * np.abs(b).max(1), floor)
                assert np.all(np.abs(a - b).max(1) <= bound), (s, dtype, scale, (np.abs(a - b).max(1) / bound).max())
            # the update resets y on element-boundary nodes and leaves the others
            idx = np.indices(lv.shape)[::-1]
            seam = np.any([i % p == 0 for i in idx], axis=0)
            left = yd.double().cpu().numpy()
            assert np.all(left[seam & lv.interior] == 0.0)
            kept = ~seam & lv.interior
            assert np.array_equal(left[kept], torch.from_numpy(y).to(dtype).double().numpy()[kept])
    prob.close()
