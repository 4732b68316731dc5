"""The wave kernel (static schedule, plans at the planner's block shape) against the oracle, bit
for bit, where it can go wrong: row widths around its batches of 8 entries and around the widest
slice it stages (64 entries), empty rows, ragged last slices, blocks of every width, one group and
many, and more cells than one step of its auxiliary warps (32)."""
import numpy as np
import pytest

import gen
import oracle

torch = pytest.importorskip("torch")
pytestmark = pytest.mark.gpu


@pytest.fixture(scope="module")
def mpk():
    if not torch.cuda.is_available():
        pytest.skip("no CUDA device")
    import paper_2405_12525_gb300 as m
    m.build()
    m.load()
    return m


def _widths_matrix(n, widths, stream):
    """Row i stores widths[i % len] entries (at most its window) near the diagonal, non-symmetric."""
    seed = gen.derive_seed(stream)
    u = gen.splitmix64(seed, n)
    rows, cols = [], []
    for i in range(n):
        w = min(widths[i % len(widths)], n)
        lo = max(0, min(i - w // 2 - int(u[i] % np.uint64(3)), n - w))
        rows += [i] * w
        cols += list(range(lo, lo + w))
    vals = gen.uniform(gen.derive_seed(stream + 1), len(rows))
    return gen.from_coo(n, rows, cols, vals)


def _check(mpk, A, m, p, order, sym=False, val="f64", accum=0, **opts):
    vt = {"f64": mpk.MPK_F64, "f32": mpk.MPK_F32}[val]
    dA = mpk.CsrMatrix.from_host(A, is_symmetric=sym, value_type=vt)
    L = mpk.build_levels(dA, 0)
    P = mpk.plan(dA, L, p_max=p, nrhs=m, order=order, accum=accum, **opts)
    stored = A.with_values(A.val.astype(np.float32).astype(np.float64)) if val == "f32" else A
    X = gen.vector(A.n, m, stream=5)
    perm = L.perm.cpu().numpy()
    Xin = X[perm] if order == mpk.ORDER_PLAN else X
    Y = torch.full((p + 1, A.n, m), float("nan"), dtype=torch.float64, device="cuda")
    for _ in range(2):  # the second launch finds the counters that the first one cleared
        Y.fill_(float("nan"))
        P.apply(torch.from_numpy(np.ascontiguousarray(Xin)).cuda(), p, Y=Y)
        P.sync_status()
        want = oracle.mpk_acc32(stored, X, p) if accum else oracle.mpk(stored, X, p)
        got = Y.cpu().numpy()
        if order == mpk.ORDER_PLAN:
            want = want[:, perm]
        assert np.array_equal(got.view(np.uint64), np.ascontiguousarray(want).view(np.uint64))


@pytest.mark.parametrize("m", [1, 2, 4, 8, 16])
@pytest.mark.parametrize("widths", [(0, 1, 7), (8, 9, 3, 0), (16, 17, 15), (62, 63, 64, 65, 2), (80, 1)])
def test_row_widths(mpk, m, widths):
    _check(mpk, _widths_matrix(1000 + 7 * m, widths, 900), m, 3, mpk.ORDER_ORIGINAL)


@pytest.mark.parametrize("n", [1, 31, 32, 33, 64, 4863, 4864, 4865])
@pytest.mark.parametrize("p", [1, 2, 31])
def test_row_counts(mpk, n, p):
    _check(mpk, _widths_matrix(n, (3, 2), 910), 1, p, mpk.ORDER_PLAN)


@pytest.mark.parametrize("n,p", [(60007, 31), (9000, 31)])
def test_descriptor_ring_wraps(mpk, n, p):
    """Slices of one entry a row: the ring of descriptors, not the entry buffer, limits the lead."""
    _check(mpk, _widths_matrix(n, (1, 0, 1), 920), 1, p, mpk.ORDER_PLAN, cache_bytes=1 << 30)
    _check(mpk, gen.laplacian_3d(17, 9, 6), 2, p, mpk.ORDER_PLAN, sym=True, cache_bytes=20000)


@pytest.mark.parametrize("cache_bytes", [1, 40000, 400000])
@pytest.mark.parametrize("m,val,accum", [(1, "f64", 0), (2, "f64", 0), (8, "f32", 0), (1, "f32", 1), (4, "f32", 1)])
def test_many_groups(mpk, cache_bytes, m, val, accum):
    _check(mpk, gen.laplacian_3d(19, 17, 23), m, 9, mpk.ORDER_PLAN, sym=True, val=val, accum=accum,
           cache_bytes=cache_bytes)


@pytest.mark.parametrize("order", [0, 1])
@pytest.mark.parametrize("m", [1, 2, 8])
@pytest.mark.parametrize("cache_bytes", [0, 60000])
def test_sorted_rows_and_own_numbering(mpk, order, m, cache_bytes):
    """Rows of very different lengths (slices sorted by length), a narrow band, in A's own numbering
    (original order) and in plan order: powers, the recurrence and host buffers."""
    A = _widths_matrix(1501, (1, 30, 4, 17, 0, 9, 2), 930)
    _check(mpk, A, m, 5, order, cache_bytes=cache_bytes)
    dA = mpk.CsrMatrix.from_host(A)
    L = mpk.build_levels(dA, 0)
    P = mpk.plan(dA, L, p_max=5, nrhs=m, order=order, cache_bytes=cache_bytes)
    X = gen.vector(A.n, m, stream=6)
    perm = L.perm.cpu().numpy() if order == mpk.ORDER_PLAN else np.arange(A.n)
    Xin = torch.from_numpy(np.ascontiguousarray(X[perm]))
    c = np.linspace(1.0, -0.5, 12)
    out = P.cheb_filter(Xin.cuda(), 11, c, scale=9.0, shift=0.3).cpu().numpy()
    want = oracle.cheb(A, X, 11, c, scale=9.0, shift=0.3)[perm]
    assert np.array_equal(out.view(np.uint64), np.ascontiguousarray(want).view(np.uint64))
    Yh = P.apply_host(Xin.pin_memory(), 5)
    torch.cuda.synchronize()
    P.sync_status()
    want = oracle.mpk(A, X, 5)[:, perm]
    assert np.array_equal(Yh.numpy().view(np.uint64), np.ascontiguousarray(want).view(np.uint64))


@pytest.mark.parametrize("m,p", [(1, 3), (2, 3), (2, 6)])
def test_hand_over_of_small_cells(mpk, m, p):
    """Cells of a few slices, run many times into poisoned outputs: a block must see every row that
    a cell's counters stand for."""
    A = gen.laplacian_3d(17, 9, 6)
    dA = mpk.CsrMatrix.from_host(A, is_symmetric=True)
    L = mpk.build_levels(dA, 0)
    P = mpk.plan(dA, L, p_max=6, nrhs=m, order=mpk.ORDER_PLAN, cache_bytes=20000)
    X = gen.vector(A.n, m, stream=81)
    perm = L.perm.cpu().numpy()
    want = torch.from_numpy(np.ascontiguousarray(oracle.mpk(A, X, p)[:, perm])).cuda()
    Xd = torch.from_numpy(np.ascontiguousarray(X[perm])).cuda()
    Y = torch.empty((p + 1, A.n, m), dtype=torch.float64, device="cuda")
    for _ in range(300):
        Y.fill_(float("nan"))
        P.apply(Xd, p, Y=Y)
        assert torch.equal(Y, want)


@pytest.mark.parametrize("order", [0, 1])
@pytest.mark.parametrize("m", [1, 4])
@pytest.mark.parametrize("cache_bytes", [0, 30000])
def test_batch_instances(mpk, order, m, cache_bytes):
    """Uneven instances with their own powers, an empty one, outputs apart, in the workspace, and an X
    inside another instance's output."""
    mats = [gen.laplacian_3d(9, 8, 7), gen.laplacian_2d(40, 31), gen.CSR([0], [], np.zeros(0)), gen.laplacian_1d(5),
            _widths_matrix(900, (1, 30, 4, 17, 0), 940), gen.laplacian_3d(15, 14, 13)]
    ps = [5, 2, 3, 7, 4, 6]
    dAs = [mpk.CsrMatrix.from_host(A) for A in mats]
    B = mpk.batch_plan(dAs, ps, nrhs=m, order=order, cache_bytes=cache_bytes)
    Xh = [gen.vector(A.n, m, stream=20 + i) if A.n else np.zeros((0, m)) for i, A in enumerate(mats)]
    perms = [mpk.build_levels(d, 0).perm.cpu().numpy() if A.n else np.zeros(0, int) for d, A in zip(dAs, mats)]
    want = [oracle.mpk(A, X, p) if A.n else np.zeros((p + 1, 0, m)) for A, X, p in zip(mats, Xh, ps)]
    if order == mpk.ORDER_PLAN:
        Xin, out = [X[q] for X, q in zip(Xh, perms)], [w[:, q] for w, q in zip(want, perms)]
    else:
        Xin, out = Xh, want
    Xs = [torch.from_numpy(np.ascontiguousarray(X)).cuda() for X in Xin]

    def same(Ys, ref):
        for Y, w in zip(Ys, ref):
            assert np.array_equal(Y.cpu().numpy().view(np.uint64), np.ascontiguousarray(w).view(np.uint64))

    Ys = [torch.full(w.shape, float("nan"), dtype=torch.float64, device="cuda") for w in out]
    for _ in range(3):
        B.apply(Xs, Ys)
        same(Ys, out)
    same(B.apply(Xs, in_place=True), [w[:, q] for w, q in zip(want, perms)])
    # instance 0's X lies inside instance 5's output
    flat = Ys[5].reshape(-1)
    inside = flat[100:100 + Xs[0].numel()].view(Xs[0].shape)
    inside.copy_(Xs[0])
    B.apply([inside] + Xs[1:], Ys)
    same(Ys, out)


def _few_values(A, count, stream):
    """A with `count` different values, among them -0.0 and the smallest normal of binary32
    (which refuses subnormals)."""
    table = np.concatenate([[-0.0, 0.0, 2.0 ** -126, -1048576.0],
                            (np.arange(max(count, 4)) - 100.5) / 64.0])[:count]
    pick = np.arange(A.nnz) % count  # every value occurs where there are `count` entries
    order = np.argsort(gen.splitmix64(gen.derive_seed(stream), A.nnz), kind="stable")
    return A.with_values(table[pick[order]])


@pytest.mark.parametrize("order", [0, 1])
@pytest.mark.parametrize("count", [1, 255, 256, 257])
@pytest.mark.parametrize("val,accum", [("f64", 0), ("f32", 0), ("f32", 1)])
def test_packed_slices(mpk, order, count, val, accum):
    """Few different values: up to 256 are stored as numbers of a table; rows of 0 to 65 entries
    (the widest are not staged), sorted by length, many groups."""
    A = _few_values(_widths_matrix(3001, (65, 1, 30, 64, 7, 0, 40, 63), 950), count, 951)
    _check(mpk, A, 1, 5, order, val=val, accum=accum, cache_bytes=60000)


@pytest.mark.parametrize("order", [0, 1])
@pytest.mark.parametrize("far", [65529, 65530, 65531, 65600])
def test_packed_slices_far_columns(mpk, order, far):
    """One row of some slices stores a column `far` on: 65534 past the smallest column among the
    slice's rows still fits 16 bits, 65535 does not."""
    n = 150001
    i = np.arange(n)
    off = np.where(i % 64 == 5, far, 1)
    keep = i + off < n
    rows = np.concatenate([i, i[keep]])
    cols = np.concatenate([i, (i + off)[keep]])
    A = gen.from_coo(n, rows, cols, np.zeros(rows.size))
    A = _few_values(A, 9, 960)
    _check(mpk, A, 1, 3, order, cache_bytes=60000)
    dA = mpk.CsrMatrix.from_host(A)
    P = mpk.plan(dA, mpk.build_levels(dA, 0), p_max=4, nrhs=1, order=order, cache_bytes=60000)
    X = gen.vector(n, 1, stream=7)
    perm = mpk.build_levels(dA, 0).perm.cpu().numpy() if order == mpk.ORDER_PLAN else np.arange(n)
    Xin = torch.from_numpy(np.ascontiguousarray(X[perm]))
    c = np.linspace(1.0, -0.5, 8)
    out = P.cheb_filter(Xin.cuda(), 7, c, scale=9.0, shift=0.3).cpu().numpy()
    want = oracle.cheb(A, X, 7, c, scale=9.0, shift=0.3)[perm]
    assert np.array_equal(out.view(np.uint64), np.ascontiguousarray(want).view(np.uint64))
    Yh = P.apply_host(Xin.pin_memory(), 4)
    torch.cuda.synchronize()
    P.sync_status()
    want = oracle.mpk(A, X, 4)[:, perm]
    assert np.array_equal(Yh.numpy().view(np.uint64), np.ascontiguousarray(want).view(np.uint64))


@pytest.mark.parametrize("order", [0, 1])
@pytest.mark.parametrize("m", [1, 8])
@pytest.mark.parametrize("x_in_place", [False, True])
def test_batch_workspace_after_outputs(mpk, order, m, x_in_place):
    """The plan's workspace holds every power, in plan order, also after a call with outputs."""
    mats = [gen.laplacian_3d(9, 8, 7), _widths_matrix(901, (1, 30, 4, 17, 0), 940), gen.laplacian_2d(40, 31)]
    ps = [4, 2, 5]
    dAs = [mpk.CsrMatrix.from_host(A) for A in mats]
    B = mpk.batch_plan(dAs, ps, nrhs=m, order=order)
    perms = [mpk.build_levels(d, 0).perm.cpu().numpy() for d in dAs]
    Xh = [gen.vector(A.n, m, stream=30 + i) for i, A in enumerate(mats)]
    want = [np.ascontiguousarray(oracle.mpk(A, X, p)[:, q]) for A, X, p, q in zip(mats, Xh, ps, perms)]
    Xs = [torch.from_numpy(np.ascontiguousarray(X[q] if order == mpk.ORDER_PLAN else X)).cuda()
          for X, q in zip(Xh, perms)]
    Ys = [torch.full(w.shape, float("nan"), dtype=torch.float64, device="cuda") for w in want]
    if x_in_place:
        for X, Y in zip(Xs, Ys):
            Y[0].copy_(X)
        Xs = [Y[0] for Y in Ys]
    B.apply([torch.zeros_like(X) for X in Xs], in_place=True)
    B.apply(Xs, Ys)
    for V, w in zip(B.views(), want):
        assert np.array_equal(V.cpu().numpy().view(np.uint64), w.view(np.uint64))


@pytest.mark.parametrize("order", [0, 1])
@pytest.mark.parametrize("m", [1, 4])
def test_batch_outputs_that_share_memory(mpk, order, m):
    """Outputs in one buffer (a scratch output given for several blocks): powers 1..p of the last
    block that writes there (every power 0 is copied before any power is written), and all blocks'
    powers in the workspace."""
    mats = [gen.laplacian_3d(9, 8, 7), gen.laplacian_2d(40, 31), gen.laplacian_3d(12, 11, 10)]
    ps = [5, 4, 3]
    dAs = [mpk.CsrMatrix.from_host(A) for A in mats]
    B = mpk.batch_plan(dAs, ps, nrhs=m, order=order)
    perms = [mpk.build_levels(d, 0).perm.cpu().numpy() for d in dAs]
    Xh = [gen.vector(A.n, m, stream=50 + i) for i, A in enumerate(mats)]
    want = [oracle.mpk(A, X, p) for A, X, p in zip(mats, Xh, ps)]
    Xs = [torch.from_numpy(np.ascontiguousarray(X[q] if order == mpk.ORDER_PLAN else X)).cuda()
          for X, q in zip(Xh, perms)]
    pool = torch.empty(max(w.size for w in want) + 7, dtype=torch.float64, device="cuda")
    Ys = [pool[7 * (i % 2):][:w.size].view(w.shape) for i, w in enumerate(want)]
    for _ in range(3):
        pool.fill_(float("nan"))
        B.apply(Xs, Ys)
        last = want[2][:, perms[2]] if order == mpk.ORDER_PLAN else want[2]
        got = Ys[2][1:].cpu().numpy()
        assert np.array_equal(got.view(np.uint64), np.ascontiguousarray(last[1:]).view(np.uint64))
        for V, w, q in zip(B.views(), want, perms):
            assert np.array_equal(V.cpu().numpy().view(np.uint64), np.ascontiguousarray(w[:, q]).view(np.uint64))


def _expires(mpk, P, run):
    """`run` fails with the timeout status; the next `run` succeeds and returns its outputs."""
    run()
    with pytest.raises(mpk.MpkError) as e:
        P.sync_status()
    assert e.value.status == 4
    out = run()
    P.sync_status()
    return out


@pytest.mark.parametrize("order", [0, 1])
@pytest.mark.parametrize("kind", ["one group", "groups", "packed", "sorted rows", "blocks", "staged far"])
def test_a_wait_that_expires(mpk, kind, order):
    """A cell that is never counted as finished: the cells that read it give up after the plan's limit
    with MPK_ERR_TIMEOUT, blocks leave with no copy in flight, and the next launches, of other numbers
    of powers too, find clean counters."""
    A = {"sorted rows": lambda: _widths_matrix(1501, (1, 30, 4, 17, 0, 9, 2), 930),
         "staged far": lambda: gen.laplacian_3d(60, 50, 40)}.get(kind, lambda: gen.laplacian_3d(19, 17, 23))()
    m = 4 if kind == "blocks" else 1
    if kind != "packed":  # (a Laplacian's two values are packed where the matrix is larger than the cache)
        A = A.with_values(gen.uniform(gen.derive_seed(970), A.nnz))
    dA = mpk.CsrMatrix.from_host(A)
    L = mpk.build_levels(dA, 0)
    P = mpk.plan(dA, L, p_max=6, nrhs=m, order=order, wait_limit_ns=20_000_000,
                 cache_bytes={"one group": 0, "staged far": 400000}.get(kind, 40000))
    X = gen.vector(A.n, m, stream=91)
    perm = L.perm.cpu().numpy() if order == mpk.ORDER_PLAN else np.arange(A.n)
    Xd = torch.from_numpy(np.ascontiguousarray(X[perm])).cuda()
    want = np.ascontiguousarray(oracle.mpk(A, X, 6)[:, perm])
    for chunk, k, p in ((0, 1, 6), (3, 2, 5), (10 ** 6, 4, 6)):
        P.debug_drop_release(min(chunk, P.describe()["num_chunks"] - 1), k)
        Y = _expires(mpk, P, lambda: P.apply(Xd, p))
        assert np.array_equal(Y.cpu().numpy().view(np.uint64), want[:p + 1].view(np.uint64))
    Y = P.apply(Xd, 2)
    P.sync_status()
    assert np.array_equal(Y.cpu().numpy().view(np.uint64), want[:3].view(np.uint64))
    c = np.linspace(1.0, -0.5, 8)
    P.debug_drop_release(0, 1)
    out = _expires(mpk, P, lambda: P.cheb_filter(Xd, 7, c, scale=9.0, shift=0.3)).cpu().numpy()
    ref = oracle.cheb(A, X, 7, c, scale=9.0, shift=0.3)[perm]
    assert np.array_equal(out.view(np.uint64), np.ascontiguousarray(ref).view(np.uint64))


@pytest.mark.parametrize("order", [0, 1])
def test_a_wait_that_expires_in_a_batch(mpk, order):
    mats = [gen.laplacian_3d(9, 8, 7), gen.laplacian_2d(40, 31), gen.laplacian_3d(15, 14, 13)]
    ps = [5, 4, 6]
    dAs = [mpk.CsrMatrix.from_host(A) for A in mats]
    B = mpk.batch_plan(dAs, ps, nrhs=1, order=order, cache_bytes=30000, wait_limit_ns=20_000_000)
    perms = [mpk.build_levels(d, 0).perm.cpu().numpy() if order == mpk.ORDER_PLAN else np.arange(d.n) for d in dAs]
    Xh = [gen.vector(A.n, 1, stream=60 + i) for i, A in enumerate(mats)]
    Xs = [torch.from_numpy(np.ascontiguousarray(X[q])).cuda() for X, q in zip(Xh, perms)]
    want = [np.ascontiguousarray(oracle.mpk(A, X, p)[:, q]) for A, X, p, q in zip(mats, Xh, ps, perms)]
    lib, status = mpk.load(), lambda: mpk._check(lib.mpk_sync_status(B._h, None))
    for in_place in (False, True):
        mpk._check(lib.mpk_debug_drop_release(B._h, 1, 2))
        B.apply(Xs, in_place=in_place)
        torch.cuda.synchronize()
        with pytest.raises(mpk.MpkError) as e:
            status()
        assert e.value.status == 4
        Ys = B.apply(Xs)
        torch.cuda.synchronize()
        status()
        for Y, w in zip(Ys, want):
            assert np.array_equal(Y.cpu().numpy().view(np.uint64), w.view(np.uint64))


def test_one_more_copy_beside_the_plans_own(mpk):
    """Rows of very different lengths in a narrow band, original order: the plan's sliced copy and one in
    A's numbering, not a third one in plan order with its rows sorted by length."""
    A = _widths_matrix(40000, (1, 30, 4, 17, 0, 9, 2), 930)
    dA = mpk.CsrMatrix.from_host(A)
    L = mpk.build_levels(dA, 0)
    P = mpk.plan(dA, L, p_max=5)
    vectors = 8 * A.n * 6  # the workspace
    padded = 12 * P.describe()["padded_entries"]
    own = 12 * A.nnz * 1.04 + 4 * A.n  # sorted rows, their map
    fits = P.describe()["device_bytes"]
    assert fits < vectors + padded + own + 60 * A.n + (1 << 20)  # (permutations, tables, records)
    # with room for exactly that the plan is the same, and its resumable recurrence right
    P = mpk.plan(dA, L, p_max=5, mem_budget=fits)
    X = gen.vector(A.n, 1, stream=6)
    Xd = torch.from_numpy(X).cuda()
    c = np.linspace(1.0, -0.5, 12)
    S = P.cheb_begin(Xd, P.cheb_state(), c[0])
    P.cheb_advance(S, 0, 5, c, scale=9.0, shift=0.3)
    P.cheb_advance(S, 5, 11, c, scale=9.0, shift=0.3)
    out = P.cheb_finish(S).cpu().numpy()
    P.sync_status()
    want = oracle.cheb(A, X, 11, c, scale=9.0, shift=0.3)
    assert np.array_equal(out.view(np.uint64), want.view(np.uint64))
    assert P.describe()["device_bytes"] == fits
