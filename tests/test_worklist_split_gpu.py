"""A chain of orders that fills two groups of a work list: that it is split, and
the FP64 form of the split plan."""
import numpy as np
import pytest

torch = pytest.importorskip("torch")
pytestmark = pytest.mark.gpu

from paper_2504_10710_gb300 import glls, inputs  # noqa: E402

# order 4, 0.93 M nodes: with 400,000 nodes a group two groups, dealt out largest
# first (A: 243 k and 224 k nodes; B: 231 k, 230 k and 1 k)
A, B = [(125, 121), (127, 110)], [(9, 7), (110, 130), (120, 120)]


@pytest.fixture(scope="module")
def problems():
    import __graft_entry__
    __graft_entry__.build()
    out = {}
    for k, ne in enumerate(A + B):
        wl = inputs.random2d(ne, 4, amp=0.1, seed=190 + k)
        prob, coords = glls.problem_for(wl)
        prob.set_rhs(wl.sample_rhs(coords)[0])
        prob.set_dirichlet(wl.sample_dirichlet(coords))
        out[ne] = prob
    yield out
    for p in out.values():
        p.close()


def _kernels(probs, o):
    outs = [np.zeros(p.N) for p in probs]
    return glls.solve_batch(probs, outs, o, worklist=True, raise_on_error=False)[0].kernels


@pytest.mark.parametrize("prec", [glls.PREC_MIXED, glls.PREC_FP64], ids=["mixed", "fp64"])
def test_split_into_two_groups(problems, prec):
    """Two passes of every loop: the batch launches the kernels of A alone and of
    B alone, not those of one loop over both."""
    o = glls.opts(tol=1e-10, gamma=1, alpha=2.0 / 3.0, precision=prec, max_iter=2)
    a, b = [problems[n] for n in A], [problems[n] for n in B]
    both = [problems[n] for n in (B[0], B[1], A[1], B[2], A[0])]
    assert _kernels(both, o) == _kernels(a, o) + _kernels(b, o)


def test_split_plan_in_fp64(problems):
    """Each problem gets its own single-solve result (FP64 tolerance of the
    other work-list test)."""
    o = glls.opts(tol=1e-10, gamma=1, alpha=2.0 / 3.0, precision=glls.PREC_FP64)
    probs = [problems[n] for n in (B[0], B[1], A[1], B[2], A[0])]
    alone = []
    for p in probs:
        u = np.zeros(p.N)
        alone.append((u, p.solve(u, o).iterations))
    outs = [np.full(p.N, np.nan) for p in probs]
    for (u, its), out, st in zip(alone, outs, glls.solve_batch(probs, outs, o, worklist=True)):
        assert st.status == glls.OK and st.iterations == its
        assert np.linalg.norm(out - u) / np.linalg.norm(u) < 1e-12
