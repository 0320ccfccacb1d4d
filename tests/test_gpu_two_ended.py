"""Elimination from both ends of the slab: every split of the rows into the two
chains and the middle row (odd and even heights, no upper chain, no chain at
all), grids from one small leaf to several recursion levels, channel subsets
with different input and output counts, through the single elimination and
the conventional adjoint method, against the oracle.  Tolerances: the stated
ones of the two precisions (relative Frobenius and largest element)."""
import numpy as np
import pytest

import oracle as O
from paper_2306_09257_gb300 import workloads as W

pytestmark = pytest.mark.gpu

TOL = {"fp64": (1e-10, 1e-10), "mixed": (1e-6, 1e-5)}
ORDERS = [-1, 0, 1]
# nx, wavelength, slab rows, inputs, outputs (None: all propagating orders)
CASES = [(8, 6.0, 1, None, None), (8, 6.0, 2, [0], [-1, 0, 1]), (16, 7.0, 3, None, None), (32, 9.0, 4, [-2, 1], None),
         (64, 10.0, 2, None, [0]), (64, 10.0, 5, None, None), (128, 13.0, 4, [-4, 0, 3], [-2, -1, 0, 1, 5]),
         (256, 21.0, 3, None, None), (256, 21.0, 6, [0, 1], None), (512, 40.0, 2, None, None)]


def close(got, ref, tol):
    got, ref = np.asarray(got), np.asarray(ref)
    assert np.linalg.norm(got - ref) <= tol * np.linalg.norm(ref)
    assert np.max(np.abs(got - ref)) <= tol * np.max(np.abs(ref))


@pytest.mark.parametrize("prec", ["fp64", "mixed"])
@pytest.mark.parametrize("case", range(len(CASES)))
def test_against_oracle(case, prec):
    from paper_2306_09257_gb300 import apf
    nx, lam, h, m_in, m_out = CASES[case]
    w = W.small_workload(nx, 34 + h, 12, lam, h)
    eps = W.iid_eps(h, nx, 40 + case, 1.0, 2.5)
    kw = {k: np.array(v) for k, v in (("m_in", m_in), ("m_out", m_out)) if v is not None}
    sol, f_ref, _, g_ref = O.f_and_grad(O.problem_from_workload(w, eps, **kw), "splitter", ORDERS, 0.3)
    s = apf.solver_for_workload(w, eps, precision=prec, m_in=m_in, m_out=m_out)
    ts, tg = TOL[prec]
    for solve in (s.solve_S_grad, s.solve_S_grad_adjoint):
        S, f, g = solve("splitter", ORDERS, 0.3)
        close(S, sol.S, ts)
        close(g, g_ref, tg)
        assert abs(f - f_ref) <= 10 * ts * abs(f_ref)
