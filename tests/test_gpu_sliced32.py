"""The FP32 rounds on the sliced layout (rows by degree in windows of 4096, 32 a slice) against a sparse
direct solution.

Graphs of about two entries a row, the smallest that run on the layout: whole windows, one row more, one
row short of a slice, rows without entries, and a row of 96 and of 97 entries (the widest slice of the
layout, and one too wide for it).  Kept and recomputed precisions, precision-only and joint starts, the
host-driven loop, inner solves that end early, the convergence fix's loaded matrix.

Tolerance: weights in [0.5, 1] and a diagonal of 1.3 times the row's sum leave every row an excess of at
least 0.3 * 0.5, so a relative residual of 1e-11 means |x - x*|_2 <= 1e-11 |b|_2 / 0.15.
"""
import numpy as np
import pytest

import synth

pytestmark = pytest.mark.gpu

torch = pytest.importorskip("torch")
sp = pytest.importorskip("scipy.sparse")
import scipy.sparse.linalg as spla  # noqa: E402


@pytest.fixture(scope="module")
def gb():
    import __graft_entry__

    __graft_entry__.build()
    import paper_0811_2518_gb300 as m

    return m


def _graph(n, hub, seed):
    """0.95 n random edges, every 50th row without any, and a row of ``hub`` entries."""
    rng = np.random.default_rng(seed)
    live = np.setdiff1d(np.arange(n), np.append(np.arange(0, n, 50), 7))
    u, v = rng.choice(live, (2, int(0.95 * n)))
    far = rng.choice(live, hub, replace=False)
    i, j = np.concatenate([u, np.full(hub, 7)]), np.concatenate([v, far])
    key = np.unique((np.minimum(i, j) * n + np.maximum(i, j))[i != j])
    iu, ju = key // n, key % n
    w = rng.uniform(0.5, 1.0, key.size) * np.where(rng.random(key.size) < 0.5, 1.0, -1.0)
    off = sp.coo_matrix((np.concatenate([w, w]), (np.concatenate([iu, ju]), np.concatenate([ju, iu]))), (n, n)).tocsr()
    d = 1.3 * np.asarray(abs(off).sum(1)).ravel()
    d[d == 0.0] = 1.0
    a = (off + sp.diags(d)).tocsr()
    a.sort_indices()
    assert off.nnz <= 2.0 * n
    return a


def _check(gb, a, solver, seed, direct=None):
    b = synth.rhs(a.shape[0], seed)
    x, st, it, rel = solver.solve(torch.from_numpy(b).cuda(), tol=1e-11, max_iter=20000)
    assert st == gb.GABP_OK and rel <= 1e-11
    ref = (direct or spla.splu(a.tocsc()).solve)(b)
    assert np.linalg.norm(x.cpu().numpy() - ref) <= 1e-11 / 0.15 * np.linalg.norm(b)


def _solver(gb, a, **opts):
    return gb.Solver(a.shape[0], a.indptr.astype(np.int32), a.indices.astype(np.int32), a.data,
                     precision=gb.GABP_PREC_FP32_REFINE, **opts)


@pytest.mark.parametrize("n", [24576, 24577, 26655])
@pytest.mark.parametrize("opts", [{}, {"reuse_precisions": 0}, {"overlap_precision": 0}, {"device_loop": 0},
                                  {"device_loop": 0, "reuse_precisions": 0}, {"graphs": 0},
                                  {"inner_max_iter": 2, "max_refine": 200}, {"inner_max_iter": 3, "max_refine": 200},
                                  {"gamma_mode": 1, "gamma": 0.1, "max_refine": 200}],
                         ids=lambda o: "-".join(f"{k}{v}" for k, v in o.items()) or "default")
def test_sliced_rounds_reach_the_direct_solution(gb, n, opts):
    a = _graph(n, 40, n)
    s = _solver(gb, a, **opts)
    direct = spla.splu(a.tocsc()).solve
    for seed in (1, 2):
        _check(gb, a, s, seed, direct)
    assert s.tuned()["mean32"] == (0, 0)  # the row kernels, which are tuned, did not run
    s.close()


@pytest.mark.parametrize("hub,sliced", [(96, True), (97, False)])
def test_widest_slice(gb, hub, sliced):
    a = _graph(25000, hub, 3)
    s = _solver(gb, a)
    _check(gb, a, s, 1)
    assert (s.tuned()["mean32"] == (0, 0)) == sliced
    s.close()


def test_handle_moves_between_the_orders(gb):
    """Kept coefficients pass between the sliced rounds and the paths in CSR order (batched, pinned shapes, the
    serial schedule), both ways, and new values reach all of them."""
    n = 25003
    a = _graph(n, 40, 5)
    s = _solver(gb, a)
    p = None
    for scale in (1.0, 2.0):
        m = a * scale
        if scale != 1.0:
            s.set_values(m.data)
        direct = spla.splu(m.tocsc()).solve
        bs = synth.rhs_batch(n, 3, 9)
        for opts in ({}, {"lanes": 4}, {"lanes": 0}, {"schedule": 1}, {"schedule": 0}, {"overlap_precision": 0}, {}):
            s.set_options(**opts)
            _check(gb, m, s, 1, direct)
            q = s.marginal_precisions().cpu().numpy()
            p = q if p is None else p
            np.testing.assert_allclose(q, scale * p, rtol=1e-3)  # FP32 stationarity (2^-16 a round)
            x = s.solve_batched(torch.from_numpy(bs).cuda(), tol=1e-11, max_iter=20000)[0].cpu().numpy()
            for c in range(3):
                assert np.linalg.norm(x[c] - direct(bs[c])) <= 1e-11 / 0.15 * np.linalg.norm(bs[c])
        s.set_options(overlap_precision=1)
    s.close()


def test_no_room_reserved_where_the_layout_cannot_be(gb):
    """A graph of long rows (500 entries, 2 x 10^8 in all) takes the memory of the row kernels alone: per entry four
    message chains, a coefficient pair and the FP32 value, 28 bytes, per row 25 words.  Allocations are rounded to 2
    MB and graphs take some memory: 50 MB, half of 3 % of the four chains."""
    _check(gb, _graph(25000, 40, 3), _solver(gb, _graph(25000, 40, 3)), 1)  # kernels are loaded
    n, half = 400000, 250
    d = torch.cat([torch.arange(-half, 0, device="cuda"), torch.arange(0, half + 1, device="cuda")])
    col = (torch.arange(n, device="cuda")[:, None] + d[None, :]).remainder(n).int().sort(dim=1)[0]
    val = torch.where(col == torch.arange(n, device="cuda", dtype=torch.int32)[:, None], 2.0 * 600, -1.0).double()
    rowptr = torch.arange(n + 1, device="cuda", dtype=torch.int32) * (2 * half + 1)
    s = gb.Solver(n, rowptr, col.reshape(-1), val.reshape(-1), precision=gb.GABP_PREC_FP32_REFINE, lanes=8)
    del col, val
    b = torch.ones(n, dtype=torch.float64, device="cuda")
    x = torch.empty_like(b)
    torch.cuda.synchronize()
    torch.cuda.empty_cache()
    free = torch.cuda.mem_get_info()[0]
    assert s.solve(b, tol=1e-8, x=x)[1] == gb.GABP_OK
    assert free - torch.cuda.mem_get_info()[0] <= 28 * 500 * n + 100 * n + (50 << 20)
    s.close()
    assert float((x - 1.0 / 700).abs().max()) <= 1e-9
