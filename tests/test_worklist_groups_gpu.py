"""Work-list batches whose problems of one order chain fill several groups."""
import numpy as np
import pytest

torch = pytest.importorskip("torch")
pytestmark = pytest.mark.gpu

from paper_2504_10710_gb300 import glls, inputs  # noqa: E402


@pytest.fixture(scope="module", autouse=True)
def _built():
    import __graft_entry__
    __graft_entry__.build()


# (elements, order) of the problems: a chain of 0.93 M nodes (two groups, the
# largest problem not the first), one of 0.90 M in two groups of unequal size
# with a small problem of its own chain between them
GROUPS = {
    "p4_two_groups": [((9, 7), 4), ((110, 130), 4), ((127, 110), 4), ((120, 120), 4), ((125, 121), 4)],
    "p9_and_p5": [((64, 63), 9), ((4, 5), 5), ((61, 64), 9), ((5, 3), 9), ((50, 62), 9)],
}


@pytest.mark.parametrize("name", GROUPS)
def test_split_chain_equals_single_solves(name):
    """Each problem gets its own single-solve result.  Both are mixed solves to
    1e-10: the tolerance is that of the work-list batch's other mixed test."""
    o = glls.opts(tol=1e-10, gamma=1, alpha=2.0 / 3.0, precision=glls.PREC_MIXED)
    probs, alone = [], []
    for k, (ne, p) in enumerate(GROUPS[name]):
        wl = inputs.random2d(ne, p, amp=0.1, seed=90 + k)
        prob, coords = glls.problem_for(wl, glls.SMOOTHER_GLL)
        prob.set_rhs(wl.sample_rhs(coords)[0])
        prob.set_dirichlet(wl.sample_dirichlet(coords))
        u = np.zeros(prob.N)
        alone.append((u, prob.solve(u, o).iterations))
        probs.append(prob)
    for rep in range(2):
        outs = [np.full(p.N, np.nan) for p in probs]
        stats = glls.solve_batch(probs, outs, o, worklist=True)
        for (u, its), out, st in zip(alone, outs, stats):
            assert st.status == glls.OK and st.rel_residual <= 1e-10
            assert abs(st.iterations - its) <= 1
            assert np.linalg.norm(out - u) / np.linalg.norm(u) < 1e-8
    for p in probs:
        p.close()
