"""Problems of a work list that have stopped: they move no mesh data while the
others of their group go on, and a stopped problem runs again in the next
solve."""
import time

import numpy as np
import pytest

torch = pytest.importorskip("torch")
pytestmark = pytest.mark.gpu

from paper_2504_10710_gb300 import glls, inputs  # noqa: E402


@pytest.fixture(scope="module", autouse=True)
def _built():
    import __graft_entry__
    __graft_entry__.build()


def _problem(n, p, amp, seed):
    wl = inputs.random2d((n, n), p, amp=amp, seed=seed)
    prob, coords = glls.problem_for(wl)
    return prob, wl.sample_rhs(coords)[0], wl.sample_dirichlet(coords)


def _set(prob, f, g, live):
    prob.set_rhs(f if live else 0.0 * f)
    prob.set_dirichlet(g if live else 0.0 * g)


def _ms(problems, o):
    outs = [torch.zeros(p.N, dtype=torch.float64, device="cuda") for p in problems]
    best = float("inf")
    for _ in range(8):
        torch.cuda.synchronize()
        t = time.perf_counter()
        for _ in range(5):
            st = glls.solve_batch(problems, outs, o, worklist=True)
        torch.cuda.synchronize()
        best = min(best, (time.perf_counter() - t) / 5 * 1e3)
    return best, [s.iterations for s in st]


def test_stopped_problems_move_no_mesh_data():
    """Two large problems beside a small one: with zero data they stop before
    the first pass, and then add to the small one's solve less than a third of
    what they add when they iterate (about the same number of passes).  Measured:
    0.21; 0.47 when their CTAs loaded operators before looking at the flag."""
    o = glls.opts(tol=1e-10, gamma=1, alpha=2.0 / 3.0, precision=glls.PREC_MIXED)
    small, f, g = _problem(6, 16, 0.2, 3)
    _set(small, f, g, True)
    alone, _ = _ms([small], o)
    large = [_problem(32, 16, 0.1, 4 + k) for k in range(2)]
    batch = [small] + [p for p, _, _ in large]
    for p, fk, gk in large:
        _set(p, fk, gk, False)
    stopped, its = _ms(batch, o)
    assert its[1:] == [0, 0] and its[0] > 5
    for p, fk, gk in large:
        _set(p, fk, gk, True)
    live, _ = _ms(batch, o)
    assert stopped - alone < (live - alone) / 3, (alone, stopped, live)
    for p in batch:
        p.close()


@pytest.mark.parametrize("prec", [glls.PREC_MIXED, glls.PREC_FP64], ids=["mixed", "fp64"])
def test_stopped_problem_runs_in_the_next_solve(prec):
    """The same plan with the live and the zero problems exchanged from solve to
    solve: each solve gives the live ones their single-solve result.  The
    coarsest grids differ, so that some steps hold only part of the problems."""
    o = glls.opts(tol=1e-10, gamma=1, alpha=2.0 / 3.0, precision=prec)
    items = [_problem(n, 5, 0.1, 60 + n) for n in (5, 33, 9, 20)]
    alone = []
    for p, f, g in items:
        _set(p, f, g, True)
        u = np.zeros(p.N)
        p.solve(u, o)
        alone.append(u)
    for mask in (0b0101, 0b1010, 0b1111, 0b0100, 0b0011):
        for k, (p, f, g) in enumerate(items):
            _set(p, f, g, bool(mask >> k & 1))
        outs = [np.full(p.N, np.nan) for p, _, _ in items]
        stats = glls.solve_batch([p for p, _, _ in items], outs, o, worklist=True)
        for k, (u, out, st) in enumerate(zip(alone, outs, stats)):
            assert st.status == glls.OK
            if mask >> k & 1:
                assert np.linalg.norm(out - u) / np.linalg.norm(u) < (1e-8 if prec == glls.PREC_MIXED else 1e-12)
            else:
                assert st.iterations == 0 and not out.any()
    for p, _, _ in items:
        p.close()
