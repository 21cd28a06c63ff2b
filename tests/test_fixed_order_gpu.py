"""Fixed-order summation through the element-result scratch (the smoothing step
and the restriction run it), at orders of every apply kernel and outside their
range: repeats give the same bits, and the values agree with the atomic sums
(the two differ in summation order only) at the parity tolerances."""
import pytest

pytestmark = pytest.mark.gpu
torch = pytest.importorskip("torch")

import numpy as np  # noqa: E402

from paper_2504_10710_gb300 import glls, inputs  # noqa: E402

GRIDS = [((3, 2), 2), ((1, 4), 5), ((4, 3), 16), ((2, 2), 17), ((2, 3, 2), 3), ((2, 1, 2), 4), ((3, 3, 3), 6),
         ((2, 2, 3), 7), ((2, 2, 2), 9)]


@pytest.mark.parametrize("dtype", [torch.float64, torch.float32], ids=["f64", "f32"])
@pytest.mark.parametrize("nelem,p", GRIDS, ids=["x".join(map(str, g)) + f"_p{p}" for g, p in GRIDS])
def test_smooth_and_restrict(nelem, p, dtype):
    mk = inputs.random2d if len(nelem) == 2 else inputs.random3d
    wl = mk(nelem, p, amp=0.1, seed=51)
    fixed, _ = glls.problem_for(wl, summation=glls.SUM_COLORED)
    atomic, _ = glls.problem_for(wl)
    top = fixed.levels - 1
    shape = fixed.level_shape(top)
    inner = tuple(slice(1, -1) for _ in shape)
    rng = np.random.default_rng(7)
    r, x = np.zeros(shape), np.zeros(shape)
    r[inner], x[inner] = (rng.standard_normal(r[inner].shape) for _ in range(2))
    r, x = (torch.from_numpy(v).to("cuda", dtype) for v in (r, x))
    tol = 1e-11 if dtype == torch.float64 else 5e-4

    def results(prob):
        out = []
        for s in range(prob.dim):
            v = x.clone()
            prob.smooth(top, s, 0.6, r, v)
            out.append(v)
        rc = torch.zeros(prob.level_shape(top - 1), dtype=dtype, device="cuda")
        prob.restrict(top, r, x, rc)
        return out + [rc]

    a, b, c = results(fixed), results(fixed), results(atomic)
    for u, v, w in zip(a, b, c):
        assert torch.equal(u, v)
        assert (u - w).abs().max() <= tol * w.abs().max()
    fixed.close()
    atomic.close()
