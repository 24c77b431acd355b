"""The FP32 mean rounds of a dense matrix (write rounds and product rounds in turn on padded arrays)
against the dense FP64 solution.

Sizes around their threshold (255 rows run the row-CSR rounds) and around the row groups, the padding
and the CTAs' row ranges; caps of 2, 3 and 5 rounds per inner solve, so that solves end in rounds of
either kind; kept and recomputed precisions, precision-only and joint starts, the host-driven loop, the
convergence fix's loaded matrix.

Tolerance: the solves end at a relative residual of 1e-11 on matrices whose diagonal is 1.3 times the
row's absolute sum, so |x - x*|_inf <= |r|_inf / (0.3 / 1.3 min A_ii), below 1e-9 |x|_inf here.
"""
import numpy as np
import pytest

import synth

pytestmark = pytest.mark.gpu

torch = pytest.importorskip("torch")


@pytest.fixture(scope="module")
def gb():
    import __graft_entry__

    __graft_entry__.build()
    import paper_0811_2518_gb300 as m

    return m


def _solve_and_check(gb, A, solver, seeds, tol=1e-11):
    for seed in seeds:
        b = synth.rhs(A.shape[0], seed)
        x, st, it, rel = solver.solve(torch.from_numpy(b).cuda(), tol=tol, max_iter=20000)
        assert st == gb.GABP_OK and rel <= tol
        ref = np.linalg.solve(A, b)
        assert np.max(np.abs(x.cpu().numpy() - ref)) <= 1e-9 * np.max(np.abs(ref))


@pytest.mark.parametrize("n", [255, 256, 257, 301, 608, 1217, 2600])
@pytest.mark.parametrize("opts", [{}, {"reuse_precisions": 0}, {"overlap_precision": 0}, {"device_loop": 0},
                                  {"device_loop": 0, "reuse_precisions": 0}, {"graphs": 0},
                                  {"inner_max_iter": 2, "max_refine": 200}, {"inner_max_iter": 3, "max_refine": 200},
                                  {"inner_max_iter": 5, "max_refine": 200, "overlap_precision": 0},
                                  {"gamma_mode": 1, "gamma": 0.1, "max_refine": 200}],
                         ids=lambda o: "-".join(f"{k}{v}" for k, v in o.items()) or "default")
def test_dense_rounds_reach_the_dense_solution(gb, n, opts):
    A = synth.dense_dd(n, 1.3, n)
    s = gb.Solver.from_dense(A, precision=gb.GABP_PREC_FP32_REFINE, **opts)
    _solve_and_check(gb, A, s, (1, 2))
    s.close()


def test_dense_handle_changes_path_and_values(gb):
    """New values, a batched solve, a serial solve and a pinned shape between dense solves on one handle."""
    n = 611
    A, A2 = synth.dense_dd(n, 1.3, 1), synth.dense_dd(n, 1.3, 2)
    s = gb.Solver.from_dense(A, precision=gb.GABP_PREC_FP32_REFINE)
    _solve_and_check(gb, A, s, (1,))
    s.set_values(synth.from_dense(A2).val)
    _solve_and_check(gb, A2, s, (1, 2))
    B = np.stack([synth.rhs(n, q) for q in (3, 4, 5)])
    X, st, _, _ = s.solve_batched(torch.from_numpy(B).cuda(), tol=1e-11)
    ref = np.linalg.solve(A2, B.T).T
    assert st == gb.GABP_OK and np.max(np.abs(X.cpu().numpy() - ref)) <= 1e-9 * np.max(np.abs(ref))
    _solve_and_check(gb, A2, s, (3,))
    s.set_options(lanes=8)
    _solve_and_check(gb, A2, s, (4,))
    s.set_options(lanes=0, reuse_precisions=0)
    X, st, _, _ = s.solve_batched(torch.from_numpy(B).cuda(), tol=1e-11)
    assert st == gb.GABP_OK and np.max(np.abs(X.cpu().numpy() - ref)) <= 1e-9 * np.max(np.abs(ref))
    s.set_options(reuse_precisions=1)
    _solve_and_check(gb, A2, s, (5,))
    x, st, _, _, _ = s.solve_systems(torch.from_numpy(B[0]).cuda(), np.array([0, n]), tol=1e-11)
    assert st == gb.GABP_OK and np.max(np.abs(x.cpu().numpy() - ref[0])) <= 1e-9 * np.max(np.abs(ref[0]))
    _solve_and_check(gb, A2, s, (6,))
    s.close()
