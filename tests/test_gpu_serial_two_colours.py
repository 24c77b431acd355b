"""FP64 serial sweeps of two-colour graphs above the one-cluster sizes (two fused passes a sweep, the
residual of a sweep completed by the next one's first pass) against the oracle's serial schedule.

An odd grid, a tree and a bipartite graph with rows of no, few and hundreds of neighbours: x, every message
and the marginal precisions after fixed sweeps, equal sweep counts at convergence, max_iter, the status
of a zero right-hand side, repeated solves, new values, the freeze.  Bounds as tests/test_gpu_serial.py: 1e-12
of the messages' scale, amplified in x by the cancellation of its sums.
"""
import numpy as np
import pytest

import oracle
import synth

pytestmark = pytest.mark.gpu

torch = pytest.importorskip("torch")


@pytest.fixture(scope="module")
def gb():
    import __graft_entry__

    __graft_entry__.build()
    import paper_0811_2518_gb300 as m

    return m


def _bipartite(n0=2200, n1=3100, seed=9):
    rng = np.random.default_rng(seed)
    a, c = [], []
    for q in range(n0 - 5):  # the last five rows of one side have no edge
        k = 300 if q < 3 else int(rng.integers(1, 6))
        a += [q] * k
        c += list(n0 + rng.choice(n1 - 9, size=k, replace=False))
    a, c = np.array(a), np.array(c)  # one side first: the index-order colouring needs two colours
    w = -rng.uniform(0.1, 1.0, a.size)
    n = n0 + n1
    s = np.bincount(a, np.abs(w), minlength=n) + np.bincount(c, np.abs(w), minlength=n)
    d = np.where(s > 0, 1.2 * s, 1.0)
    return synth.from_coo(n, np.concatenate([a, c, np.arange(n)]), np.concatenate([c, a, np.arange(n)]),
                          np.concatenate([w, w, d]))


MATS = {
    "grid": lambda: synth.grid3d(17, 1.05, 3),
    "tree": lambda: synth.random_tree(6001, 3, dd=True),
    "bipartite": _bipartite,
}


def _check(m, b, r, x, P, hm, Pi):
    rows = np.repeat(np.arange(m.n), np.diff(m.rowptr))
    off = rows != m.col
    assert np.allclose(P[off], r["Pmsg"][off], rtol=1e-12, atol=0)
    assert not np.any(P[~off]) and not np.any(hm[~off])
    hm_ref = r["Pmsg"] * r["mumsg"]
    assert np.max(np.abs(hm[off] - hm_ref[off])) <= 1e-12 * np.max(np.abs(hm_ref[off]))
    absP = np.bincount(rows, np.abs(np.where(off, r["Pmsg"], m.val)), minlength=m.n)
    absh = np.abs(b) + np.bincount(rows[off], np.abs(hm_ref[off]), minlength=m.n)
    assert np.all(np.abs(x - r["x"]) <= 1e-12 * (absP * np.abs(r["x"]) + absh) / np.abs(r["P"]) + 1e-300)
    assert np.all(np.abs(Pi - r["P"]) <= 1e-12 * absP)


@pytest.mark.parametrize("name", list(MATS))
def test_sweeps_match_oracle(gb, name):
    m = MATS[name]()
    b = synth.rhs(m.n, 7)
    s = gb.Solver.from_csr(m, schedule=1)
    assert s.serial_colours()[1] == 2
    for sweeps in (1, 2, 3, 8):
        x, st, it, rel = s.solve(torch.from_numpy(b).cuda(), tol=0.0, max_iter=sweeps)
        r = oracle.gabp_serial(m, b, max_iter=sweeps, tol=0.0, messages=True)
        assert st == gb.GABP_NOT_CONVERGED and it == r["iters"] == s.stats()["rounds"] == sweeps
        res = b - (np.bincount(np.repeat(np.arange(m.n), np.diff(m.rowptr)), m.val * r["x"][m.col], minlength=m.n))
        assert abs(rel - np.linalg.norm(res) / np.linalg.norm(b)) <= 1e-9 * rel + 1e-12
        P, hm = s.messages()
        _check(m, b, r, x.cpu().numpy(), P.cpu().numpy(), hm.cpu().numpy(), s.marginal_precisions().cpu().numpy())
    s.close()


@pytest.mark.parametrize("name", list(MATS))
@pytest.mark.parametrize("every", [1, 16])
def test_converged_equal_sweeps_and_handle_reuse(gb, name, every):
    m = MATS[name]()
    s = gb.Solver.from_csr(m, schedule=1, check_every=every)
    for seed in (3, 4):
        b = synth.rhs(m.n, seed)
        x, st, it, rel = s.solve(torch.from_numpy(b).cuda(), tol=1e-11, max_iter=5000)
        r = oracle.gabp_serial(m, b, max_iter=5000, tol=1e-11)
        assert st == gb.GABP_OK and it == r["iters"] and rel <= 1e-11
        assert np.linalg.norm(x.cpu().numpy() - r["x"]) <= 1e-11 * np.linalg.norm(r["x"])
    z, st, it, rel = s.solve(torch.zeros(m.n, dtype=torch.float64, device="cuda"), tol=1e-12)
    assert st == gb.GABP_OK and it == 0 and rel == 0.0 and not torch.any(z)
    assert not bool(s.messages()[0].any())
    m.val = np.where(np.repeat(np.arange(m.n), np.diff(m.rowptr)) == m.col, 1.5 * m.val, m.val)
    s.set_values(m.val)
    x, st, it, rel = s.solve(torch.from_numpy(b).cuda(), tol=1e-11, max_iter=5000)
    r = oracle.gabp_serial(m, b, max_iter=5000, tol=1e-11)
    assert st == gb.GABP_OK and it == r["iters"]
    assert np.linalg.norm(x.cpu().numpy() - r["x"]) <= 1e-11 * np.linalg.norm(r["x"])
    s.close()


@pytest.mark.parametrize("name", list(MATS))
def test_freeze_is_the_plain_run_up_to_its_sweep(gb, name):
    m = MATS[name]()
    b = torch.from_numpy(synth.rhs(m.n, 5)).cuda()
    f = gb.Solver.from_csr(m, schedule=1, freeze_precisions=1)
    p = gb.Solver.from_csr(m, schedule=1)
    f.solve(b, tol=0.0, max_iter=40)
    F = f.stats()["freeze_round"]
    assert 0 < F < 40
    for t in sorted({1, 2, F - 1, F}):
        xf, xp = f.solve(b, tol=0.0, max_iter=t)[0], p.solve(b, tol=0.0, max_iter=t)[0]
        assert torch.equal(xf, xp)
        assert all(torch.equal(u, v) for u, v in zip(f.messages(), p.messages()))
    xf, xp = f.solve(b, tol=0.0, max_iter=F + 9)[0], p.solve(b, tol=0.0, max_iter=F + 9)[0]
    assert torch.allclose(xf, xp, rtol=1e-12, atol=1e-13 * float(xp.abs().max()))
    f.close()
    p.close()


def test_breakdown(gb):
    """A zero cavity precision in the middle of a large chain is reported as the oracle reports it."""
    n = 5001
    d = np.full(n, 3.0)
    w = np.ones(n - 1)
    d[2000], d[2001] = 1.0, 1.0  # neighbours whose cavities cancel: 1 - 1/1
    w[1999] = w[2001] = 1e-300
    i = np.arange(n - 1)
    m = synth.from_coo(n, np.concatenate([i, i + 1, np.arange(n)]), np.concatenate([i + 1, i, np.arange(n)]),
                       np.concatenate([w, w, d]))
    b = np.ones(n)
    r = oracle.gabp_serial(m, b, max_iter=50, tol=1e-12)
    s = gb.Solver.from_csr(m, schedule=1)
    x, st, it, rel = s.solve(torch.from_numpy(b).cuda(), tol=1e-12, max_iter=50)
    s.close()
    assert st == r["status"]
    if r["status"] == oracle.BREAKDOWN:
        assert it == r["iters"]


def test_no_room_for_the_two_colour_layout(gb):
    """Where the device has room for the general passes only (about 130 MB here, the two-colour layout and state
    360 MB), they run, with the same sweeps."""
    m = synth.grid3d(96, 1.05, 3)
    b = torch.from_numpy(synth.rhs(m.n, 7)).cuda()
    s = gb.Solver.from_csr(m, schedule=1)
    ref, st, sweeps, _ = s.solve(b, tol=1e-10, max_iter=500)
    assert st == gb.GABP_OK
    s.close()
    s = gb.Solver.from_csr(m, schedule=1)
    s.serial_colours()
    torch.cuda.synchronize()
    torch.cuda.empty_cache()
    keep = torch.empty(torch.cuda.mem_get_info()[0] - (250 << 20), dtype=torch.uint8, device="cuda")
    try:
        x, st, it, _ = s.solve(b, tol=1e-10, max_iter=500, x=torch.empty_like(b))
    finally:
        del keep
        torch.cuda.empty_cache()
    assert st == gb.GABP_OK and it == sweeps
    assert torch.allclose(x, ref, rtol=0, atol=1e-10 * float(ref.abs().max()))
    s.close()


def _regular(side, deg):
    """A bipartite graph of two sides, every row with ``deg`` neighbours around its place on the other side."""
    i = np.repeat(np.arange(side), deg)
    j = side + (i + np.tile(np.arange(deg), side)) % side
    w = -np.random.default_rng(1).uniform(0.1, 1.0, i.size)
    d = 1.2 * (np.bincount(i, -w, minlength=2 * side) + np.bincount(j, -w, minlength=2 * side))
    a = np.arange(2 * side)
    return synth.from_coo(2 * side, np.concatenate([i, j, a]), np.concatenate([j, i, a]), np.concatenate([w, w, d]))


@pytest.mark.parametrize("side,deg,freeze,two", [(6000, 50, 0, False), (6000, 50, 1, False), (40000, 30, 0, True),
                                                 (24000, 20, 0, True), (24000, 20, 1, False), (50000, 12, 1, True)])
def test_long_rows_run_the_general_passes(gb, side, deg, freeze, two):
    """Rows long for a lane each, and few of them, run the general passes: seen by the memory of their state (16
    bytes a slot, 24 with the freeze, where the two-colour layout and state take 52 and 60)."""
    m = _regular(side, deg)
    b = synth.rhs(m.n, 7)
    s = gb.Solver.from_csr(m, schedule=1, freeze_precisions=freeze)
    assert s.serial_colours()[1] == 2
    tb, x = torch.from_numpy(b).cuda(), torch.empty(m.n, dtype=torch.float64, device="cuda")
    torch.cuda.synchronize()
    free = torch.cuda.mem_get_info()[0]
    st, it = s.solve(tb, tol=1e-11, max_iter=3000, x=x)[1:3]
    taken = free - torch.cuda.mem_get_info()[0]
    assert (taken > 40 * 2 * side * deg) == two
    r = oracle.gabp_serial(m, b, max_iter=3000, tol=1e-11)
    assert st == gb.GABP_OK and it == r["iters"]
    assert np.linalg.norm(x.cpu().numpy() - r["x"]) <= 1e-11 * np.linalg.norm(r["x"])
    s.close()
