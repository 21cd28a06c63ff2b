"""Fixed-order summation with an odd number of right-hand sides on an odd number
of 3-D elements: the element-pair FP32 apply and the FP64 even-odd apply with
its p.(A p) partials write the scratch of every right-hand side."""
import numpy as np
import pytest

torch = pytest.importorskip("torch")
pytestmark = pytest.mark.gpu

from paper_2504_10710_gb300 import glls, inputs  # noqa: E402


@pytest.mark.parametrize("prec", [glls.PREC_FP64, glls.PREC_MIXED], ids=["fp64", "mixed"])
@pytest.mark.parametrize("nelem,p,nrhs", [((3, 1, 3), 7, 3), ((3, 3, 1), 6, 3), ((1, 3, 3), 8, 2)],
                         ids=lambda v: "x".join(map(str, v)) if isinstance(v, tuple) else str(v))
def test_each_right_hand_side_has_its_single_solve_bits(nelem, p, nrhs, prec):
    wl = inputs.random3d(nelem, p, amp=0.1, seed=98, nrhs=nrhs)
    multi, coords = glls.problem_for(wl, nrhs=nrhs, summation=glls.SUM_COLORED)
    single, _ = glls.problem_for(wl, summation=glls.SUM_COLORED)
    F = np.ascontiguousarray(wl.sample_rhs(coords).reshape(nrhs, -1))
    g = wl.sample_dirichlet(coords).ravel()
    o = glls.opts(tol=1e-10, gamma=1, alpha=2.0 / 3.0, precision=prec)
    multi.set_rhs(F)
    multi.set_dirichlet(g)
    single.set_dirichlet(g)
    U = np.zeros((nrhs, multi.N))
    stats = multi.solve(U, o)
    for j in range(nrhs):
        single.set_rhs(F[j])
        u = np.zeros(multi.N)
        assert single.solve(u, o).iterations == stats[j].iterations
        assert np.array_equal(U[j], u), j
    multi.close()
    single.close()
