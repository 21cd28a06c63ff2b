"""The packed FP32 3-D apply (p = 1..8) where its pairing changes: element
counts that leave an unpaired last element, one element pair, and right-hand
side counts of one, two and three (elements paired for the odd counts, right-
hand sides for the even one), against the oracle's operator at the parity
tolerance of the FP32 apply."""
import numpy as np
import pytest

pytestmark = pytest.mark.gpu
torch = pytest.importorskip("torch")

from oracle import gll as ogll  # noqa: E402
from oracle.discretize import Level  # noqa: E402
from paper_2504_10710_gb300 import glls, inputs  # noqa: E402


@pytest.mark.parametrize("p", [1, 2, 3, 4, 5, 6, 7, 8])
@pytest.mark.parametrize("nelem", [(3, 3, 3), (1, 2, 1), (5, 1, 3)], ids=lambda g: "x".join(map(str, g)))
def test_pairs(nelem, p):
    if p == 1 and min(nelem) < 2:
        pytest.skip("order 1 needs two elements along every axis")
    wl = inputs.random3d(nelem, p, amp=0.1, seed=41)
    prob, _ = glls.problem_for(wl)
    xi, _ = ogll.gll(p)
    lv = Level(3, nelem, p, wl.coords(xi))
    rng = np.random.default_rng(p)
    for nrhs in (1, 2, 3):
        x = np.where(lv.interior, rng.standard_normal((nrhs,) + lv.shape), 0.0).astype(np.float32)
        y = torch.full((nrhs, lv.N), 7.0, dtype=torch.float32, device="cuda")
        prob.apply_multi(prob.levels - 1, torch.from_numpy(x).cuda(), y, nrhs)
        got = y.double().cpu().numpy()
        for j in range(nrhs):
            ref = lv.apply(x[j].astype(np.float64)).ravel()
            assert np.abs(got[j] - ref).max() < 5e-5 * np.abs(ref).max(), (nrhs, j)
    prob.close()
