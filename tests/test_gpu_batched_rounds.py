"""The batched mean rounds that store every second round's messages, and the two-colour serial
sweeps that store one direction of every edge, against the dense FP64 solution.

Graphs with rows of no, one and odd numbers of edges, of two colours (a tree, a bipartite graph) and
of more; 1 to 130 columns (one, two and four columns a lane, and two chunks); caps of 2, 3 and 5
rounds per inner solve (a first round without messages, a second that writes the store, a third that
gathers), which the refinement loop has to turn into a converged answer all the same: in exact
arithmetic the error shrinks by 0.45 or more a step (a cap of 1 does not converge on the tree).

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


def _matrix(kind):
    rng = np.random.default_rng(11)
    n = 203
    A = np.zeros((n, n))
    if kind == "tree":
        for i in range(1, n - 2):  # the last two rows have no edge
            A[rng.integers(0, i), i] = rng.uniform(-1, 1)
    elif kind == "bipartite":
        A[:90, 90:] = rng.uniform(-1, 1, (90, n - 90)) * (rng.random((90, n - 90)) < 0.05)
    else:
        A = np.triu(rng.uniform(-1, 1, (n, n)) * (rng.random((n, n)) < 0.04), 1)
    A = A + A.T
    s = np.abs(A).sum(1)
    A[np.diag_indices(n)] = np.where(s > 0, 1.3 * s, 1.0)
    return A


@pytest.mark.parametrize("cap", [400, 2, 3, 5])
@pytest.mark.parametrize("R", [1, 33, 64, 130])
@pytest.mark.parametrize("schedule", [0, 1])
@pytest.mark.parametrize("kind", ["tree", "bipartite", "random"])
def test_batched_rounds_reach_the_dense_solution(gb, kind, schedule, R, cap):
    A = _matrix(kind)
    n = A.shape[0]
    B = np.random.default_rng(R).standard_normal((R, n))
    s = gb.Solver.from_csr(synth.from_dense(A), schedule=schedule, inner_max_iter=cap, max_refine=200)
    if schedule:
        assert (s.serial_colours()[1] == 2) == (kind != "random")
    for _ in range(2):  # the second call starts from the first one's stores
        X, st, it, rel = s.solve_batched(torch.from_numpy(B).cuda(), tol=1e-11, max_iter=20000)
        assert st == gb.GABP_OK and rel.max() <= 1e-11
        ref = np.linalg.solve(A, B.T).T
        assert np.max(np.abs(X.cpu().numpy() - ref)) <= 1e-9 * np.max(np.abs(ref))
    s.close()


@pytest.mark.parametrize("R", [1, 32, 40])
@pytest.mark.parametrize("kind", ["tree", "random", "dense rows"])
def test_few_rows_and_many_rows_give_the_same_bits(gb, kind, R):
    """A graph alone (rounds as long as their longest row: eight slots of a row together) and in 250 copies (rounds
    bound by their bytes: two slots) after equal rounds: rows of none to 29 slots, every remainder."""
    if kind == "dense rows":
        n = 203
        A = np.triu(np.random.default_rng(2).uniform(-1, 1, (n, n)), 1)
        A *= (np.arange(n)[:, None] + np.arange(n)[None, :]) % 7 == 0
        A[:46, :46] = A[46:92, :46] = A[:46, 46:92] = 0.0
        A = A + A.T
        A[np.diag_indices(n)] = 1.3 * np.maximum(np.abs(A).sum(1), 1.0)
    else:
        A = _matrix(kind)
    m = synth.from_dense(A)
    n = m.n
    B = np.random.default_rng(R).standard_normal((R, n))
    out = []
    for copies in (1, 250):
        big = synth.block_diag([m] * copies)
        s = gb.Solver.from_csr(big, lanes=4, inner_max_iter=9, inner_tol=1e-30, max_refine=2)
        X = s.solve_batched(torch.from_numpy(np.tile(B, (1, copies))).cuda(), tol=0.0, max_iter=1000, check=False)[0]
        out.append(X.cpu().numpy()[:, :n])
        s.close()
    assert np.any(out[0]) and np.array_equal(out[0], out[1])
