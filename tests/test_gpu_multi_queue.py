"""Independent systems solved by one SM each from a queue, alone and beside larger systems on the
grid-persistent kernel, against the dense FP64 solution and the oracle.

Batches that the choice of kernels gives to the queue: hundreds of small systems, among them rows without
edges, single rows, dense rows wider than a chunk of four lines, sizes around a slice (31 to 33 rows) and
around the 16 warps' slices; a broken system among good ones; zero right-hand sides; caps on rounds and
steps; new values and other offsets on one handle.  Solutions to 1e-9 of the dense ones (residual 1e-11,
diagonal 1.2 times the row's absolute sum or more).
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


def _small(n, seed, density=None):
    rng = np.random.default_rng(seed)
    A = np.triu(rng.uniform(-1, 1, (n, n)) * (rng.random((n, n)) < (density or min(1.0, 5.0 / n))), 1)
    A = A + A.T
    s = np.abs(A).sum(1)
    A[np.diag_indices(n)] = np.where(s > 0, 1.2 * s, 1.0)
    return A


def _batch():
    sizes = [1, 2, 31, 32, 33, 64, 65, 511, 512, 513, 700] + [17 + 3 * q for q in range(150)]
    mats = [_small(n, q) for q, n in enumerate(sizes)]
    mats += [_small(90, 500, 0.4), _small(60, 501, 1.0), _small(200, 502, 0.1)]  # rows of up to 59 slots
    return mats


def _solve(gb, s, mats, b, off, **kw):
    x, st, sts, its, rel = s.solve_systems(torch.from_numpy(b).cuda(), off, **kw)
    return x.cpu().numpy(), st, sts, its, rel


def _check(gb, mats, b, off, x, sts, rel, tol=1e-11):
    for k, A in enumerate(mats):
        sl = slice(off[k], off[k + 1])
        assert sts[k] == gb.GABP_OK and rel[k] <= tol, k
        ref = np.linalg.solve(A, b[sl])
        assert np.max(np.abs(x[sl] - ref)) <= 1e-9 * max(np.max(np.abs(ref)), 1e-300), k


def test_many_small_systems(gb):
    mats = _batch()
    big = synth.block_diag([synth.from_dense(A) for A in mats])
    off = big.meta["offsets"]
    b = synth.rhs(big.n, 3)
    b[off[20]:off[21]] = 0.0
    s = gb.Solver.from_csr(big)
    for _ in range(2):
        x, st, sts, its, rel = _solve(gb, s, mats, b, off, tol=1e-11)
        assert st == gb.GABP_OK and not np.any(x[off[20]:off[21]]) and its[0] <= its.max()
        _check(gb, mats, b, off, x, sts, rel)
    assert s.tuned()["multi_mode"] == 2 and s.tuned()["multi_grid"] == (0, 0)  # no shape was tuned
    # new values; then pairs of systems as one
    scaled = [2.0 * A for A in mats]
    s.set_values(2.0 * big.val)
    x, st, sts, its, rel = _solve(gb, s, scaled, b, off, tol=1e-11)
    _check(gb, scaled, b, off, x, sts, rel)
    off2 = np.concatenate([off[::2], off[-1:]]) if (len(off) - 1) % 2 else off[::2]
    x2, st, sts, its, rel = _solve(gb, s, scaled, b, off2, tol=1e-11)
    assert st == gb.GABP_OK and np.allclose(x2, x, rtol=0, atol=1e-8 * np.max(np.abs(x)))
    s.close()


def test_same_rounds_as_the_grid_kernel(gb):
    mats = [synth.from_dense(A) for A in _batch()]
    big = synth.block_diag(mats)
    off = big.meta["offsets"]
    b = torch.from_numpy(synth.rhs(big.n, 4)).cuda()
    its = []
    for mode in (0, 3):
        s = gb.Solver.from_csr(big, multi_mode=mode)
        its.append(s.solve_systems(b, off, tol=1e-11)[3])
        s.close()
    assert np.max(np.abs(its[0] - its[1])) <= 2  # the same rounds but for the rounding of their sums


@pytest.mark.parametrize("opts", [{"inner_max_iter": 1, "max_refine": 3}, {"inner_max_iter": 2, "max_refine": 1},
                                  {"inner_max_iter": 5, "max_refine": 2}])
def test_caps_and_breakdown(gb, opts):
    star = np.array([[2.0, 1, 0, 0], [1, 3, 1, 1], [0, 1, 1, 0], [0, 1, 0, 0.5]])
    mats = _batch()[:40] + [star] + _batch()[40:80]
    big = synth.block_diag([synth.from_dense(A) for A in mats])
    off = big.meta["offsets"]
    b = synth.rhs(big.n, 5)
    got = []
    for mode in (0, 3):
        s = gb.Solver.from_csr(big, multi_mode=mode, **opts)
        got.append(_solve(gb, s, mats, b, off, tol=1e-13, check=False))
        s.close()
    assert got[0][2][40] == gb.GABP_BREAKDOWN
    assert np.array_equal(got[0][2], got[1][2]) and np.max(np.abs(got[0][3] - got[1][3])) <= 2
    ok = got[0][2] != gb.GABP_BREAKDOWN
    for k in np.nonzero(ok)[0]:
        sl = slice(off[k], off[k + 1])
        assert np.allclose(got[0][0][sl], got[1][0][sl], rtol=1e-4, atol=1e-5 * np.max(np.abs(got[1][0][sl])) + 1e-30)


def test_large_systems_beside_small_ones(gb):
    """Two systems above the queue kernel's size go to the grid kernel, the others to the queue."""
    mats = synth.rgg_batch(400, 1024, 2048, 2.0, 4) + synth.rgg_batch(2, 20000, 30000, 2.0, 5)
    mats = mats[:10] + [mats[400]] + mats[10:400] + [mats[401]]
    big = synth.block_diag(mats)
    off = big.meta["offsets"]
    b = synth.rhs(big.n, 6)
    s = gb.Solver.from_csr(big)
    x, st, sts, its, rel = _solve(gb, s, mats, b, off, tol=1e-11)
    assert st == gb.GABP_OK and np.all(rel <= 1e-11) and s.tuned()["multi_grid"] == (0, 0)
    s.close()
    for k in (0, 9, 10, 11, 40, 401):
        sl = slice(off[k], off[k + 1])
        ref = oracle.gabp_broadcast(mats[k], b[sl], max_iter=5000, tol=1e-13)
        assert np.linalg.norm(x[sl] - ref["x"]) <= 1e-9 * np.linalg.norm(ref["x"])


@pytest.mark.parametrize("stop", [10, 11, 12, 14, 16])
def test_kept_precisions_survive_a_batch_on_both_kernels(gb, stop):
    """The precisions a handle keeps between solves are the same before and after a call whose small systems
    go to the queue and whose large ones to the grid kernel (the stops end them at rounds of every
    remainder modulo three, the length of their ring)."""
    mats = synth.rgg_batch(400, 1024, 1100, 2.0, 4) + synth.rgg_batch(2, 20000, 30000, 2.0, 5)
    big = synth.block_diag(mats)
    off = big.meta["offsets"]
    b = torch.from_numpy(synth.rhs(big.n, 6)).cuda()
    s = gb.Solver.from_csr(big, prec_stop_log2=stop)
    B = b.reshape(1, -1)
    s.solve_batched(B, tol=1e-6)
    before = s.marginal_precisions()
    assert s.solve_systems(b, off, tol=1e-10)[1] == gb.GABP_OK
    assert s.tuned()["multi_mode"] == 2 and s.tuned()["multi_grid"] == (0, 0)  # both kernels ran
    s.solve_batched(B, tol=1e-6)
    assert torch.equal(s.marginal_precisions(), before)
    s.close()


@pytest.mark.parametrize("opts", [{}, {"lanes": 4}])
def test_the_queue_is_not_taken_for_a_timed_choice(gb, opts):
    """After a call on the queue, offsets that make one large system of all of them (or a pinned shape) run
    the grid kernel, which one team of blocks cannot match there (one cluster against every SM)."""
    mats = synth.rgg_batch(300, 1024, 1100, 2.0, 4)
    big = synth.block_diag(mats)
    b = torch.from_numpy(synth.rhs(big.n, 6)).cuda()
    s = gb.Solver.from_csr(big)
    x = s.solve_systems(b, big.meta["offsets"], tol=1e-11)[0]
    assert s.tuned()["multi_mode"] == 2 and s.tuned()["multi_grid"] == (0, 0)  # the queue
    s.set_options(**opts)
    one, st, _, _, rel = s.solve_systems(b, np.array([0, big.n], dtype=np.int32), tol=1e-11)
    assert st == gb.GABP_OK and rel[0] <= 1e-11
    assert torch.allclose(one, x, rtol=0, atol=1e-8 * float(x.abs().max()))
    t = s.tuned()
    assert t["multi_mode"] == 1 and (t["multi_grid"] != (0, 0)) == (not opts)  # timed; a pinned shape is not tuned
    s.close()


def test_iterates_beyond_the_square_root_of_fp32(gb):
    """Solutions whose sum of squares is half again FP32's largest value, though no entry's square and no warp's
    sum (a sixteenth of the rows) comes near it, converge as on the grid kernel."""
    mats = synth.rgg_batch(300, 1024, 1100, 2.0, 8)
    big = synth.block_diag(mats)
    off = big.meta["offsets"]
    b = synth.rhs(big.n, 9)
    for k, m in enumerate(mats):
        sl = slice(off[k], off[k + 1])
        if k < 3:  # three systems of this kind, the others as drawn
            x = np.linalg.solve(synth.to_dense(m), b[sl])
            b[sl] *= np.sqrt(5e38) / np.linalg.norm(x)
    got = []
    for mode in (0, 3):
        s = gb.Solver.from_csr(big, multi_mode=mode)
        x, st, sts, its, rel = _solve(gb, s, mats, b, off, tol=1e-11, check=False)
        assert s.tuned()["multi_mode"] == (0 if mode else 2)  # 2: the queue
        s.close()
        assert st == gb.GABP_OK and np.all(sts == gb.GABP_OK) and np.all(rel <= 1e-11)
        got.append(x)
    for k in range(5):
        sl = slice(off[k], off[k + 1])
        assert np.linalg.norm(got[0][sl] - got[1][sl]) <= 1e-9 * np.linalg.norm(got[1][sl])


def _hub(m, width, seed):
    """m with its first row joined to ``width`` others (the diagonal keeps its dominance)."""
    rng = np.random.default_rng(seed)
    rows = np.repeat(np.arange(m.n), np.diff(m.rowptr))
    off = rows != m.col
    j = np.setdiff1d(rng.choice(np.arange(1, m.n), width, replace=False), m.col[m.rowptr[0]:m.rowptr[1]])
    i = np.concatenate([rows[off], np.zeros(j.size, int), j])
    k = np.concatenate([m.col[off], j, np.zeros(j.size, int)])
    v = np.concatenate([m.val[off], np.full(2 * j.size, -0.7)])
    d = 1.1 * np.bincount(i, np.abs(v), minlength=m.n)
    return synth.from_coo(m.n, np.concatenate([i, np.arange(m.n)]), np.concatenate([k, np.arange(m.n)]),
                          np.concatenate([v, np.where(d > 0, d, 1.0)]))


@pytest.mark.parametrize("make,queue", [
    (lambda: [synth.random_sym(2048, 50, 1.1, q) for q in range(8)], False),   # few systems of wide rows
    (lambda: [synth.random_sym(1024, 15, 1.1, q) for q in range(152)], True),  # an SM for each
    (lambda: [_hub(m, 500, 3) for m in synth.rgg_batch(8, 4000, 4096, 2.0, 4)], False),  # hub rows, SMs idle
    (lambda: [_hub(m, 500, 3) for m in synth.rgg_batch(152, 2000, 2048, 2.0, 4)], True),
    (lambda: [_hub(m, 1000, 3) for m in synth.rgg_batch(152, 2000, 2048, 2.0, 4)], False),  # too wide for a lane
], ids=["wide8", "wide152", "hub8", "hub152", "hub_too_wide"])
def test_choice_by_slots_and_widths(gb, make, queue):
    """Systems go to the queue where one SM each is enough for their slots and widest rows."""
    mats = make()
    big = synth.block_diag(mats)
    off = big.meta["offsets"]
    b = synth.rhs(big.n, 6)
    s = gb.Solver.from_csr(big)
    for _ in range(2):
        x, st, sts, its, rel = _solve(gb, s, mats, b, off, tol=1e-11)
        assert st == gb.GABP_OK and np.all(rel <= 1e-11)
    t = s.tuned()
    assert t["multi_mode"] in ((2,) if queue else (1, 2)) and (t["multi_grid"] == (0, 0)) == queue
    s.close()
    for k in (0, 5):
        sl = slice(off[k], off[k + 1])
        ref = np.linalg.solve(synth.to_dense(mats[k]), b[sl])
        assert np.linalg.norm(x[sl] - ref) <= 1e-9 * np.linalg.norm(ref)
