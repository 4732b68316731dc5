"""Plans whose gathers of x are scattered (a line a row, little of it read again): the wave kernel
takes its smaller entry buffer for them.  Bit for bit against the oracle where the buffer can go wrong
(slices around its widest, many turns, packed copies, every value type and width), and its time
against the ticketed kernel, which such matrices must not be better off with."""
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


def _scattered(n, widths, stream, count=0):
    """Row i stores widths[i % len] entries in random columns (fewer where they coincide); `count`
    different values, or random ones."""
    w = np.asarray(widths)[np.arange(n) % len(widths)]
    rows = np.repeat(np.arange(n), w)
    cols = (gen.splitmix64(gen.derive_seed(stream), rows.size) % np.uint64(n)).astype(np.int64)
    key = np.unique(rows * n + cols)
    vals = gen.uniform(gen.derive_seed(stream + 1), key.size)
    if count:
        vals = (np.floor(vals * count) - count / 2 + 0.5) / 8.0
    return gen.from_coo(n, key // n, key % n, vals)


def _same(got, want):
    assert np.array_equal(got.view(np.uint64), np.ascontiguousarray(want).view(np.uint64))


@pytest.mark.parametrize("order", [0, 1])
@pytest.mark.parametrize("m", [1, 2, 4])
@pytest.mark.parametrize("widths,val,accum,count,cache_bytes", [
    ((1, 30, 7, 0, 4), "f64", 0, 0, 0),
    ((62, 63, 64, 65, 2), "f64", 0, 0, 0),
    ((62, 63, 64, 65, 2), "f32", 0, 0, 400000),
    ((9, 7, 8), "f32", 1, 0, 400000),
    ((64, 65, 9, 1), "f64", 0, 200, 400000),
])
def test_scattered_gathers(mpk, order, m, widths, val, accum, count, cache_bytes):
    n = 40007
    A = _scattered(n, widths, 980, count)
    vt = {"f64": mpk.MPK_F64, "f32": mpk.MPK_F32}[val]
    dA = mpk.CsrMatrix.from_host(A, value_type=vt)
    stored = A.with_values(A.val.astype(np.float32).astype(np.float64)) if val == "f32" else A
    L = mpk.build_levels(dA, 0)
    P = mpk.plan(dA, L, p_max=4, nrhs=m, order=order, accum=accum, cache_bytes=cache_bytes)
    X = gen.vector(n, m, stream=7)
    perm = L.perm.cpu().numpy() if order == mpk.ORDER_PLAN else np.arange(n)
    Xd = torch.from_numpy(np.ascontiguousarray(X[perm])).cuda()
    want = (oracle.mpk_acc32(stored, X, 4) if accum else oracle.mpk(stored, X, 4))[:, perm]
    Y = torch.full((5, n, m), float("nan"), dtype=torch.float64, device="cuda")
    for _ in range(2):
        Y.fill_(float("nan"))
        P.apply(Xd, 4, Y=Y)
        P.sync_status()
        _same(Y.cpu().numpy(), want)
    if not accum:
        c = np.linspace(1.0, -0.5, 7)
        out = P.cheb_filter(Xd, 6, c, scale=9.0, shift=0.3).cpu().numpy()
        _same(out, oracle.cheb(stored, X, 6, c, scale=9.0, shift=0.3)[perm])
        Yh = P.apply_host(Xd.cpu().pin_memory(), 4)
        torch.cuda.synchronize()
        P.sync_status()
        _same(Yh.numpy(), want)


@pytest.mark.parametrize("order", [0, 1])
def test_a_wait_that_expires_with_the_smaller_buffer(mpk, order):
    n = 40007
    A = _scattered(n, (9, 7, 30), 984)
    dA = mpk.CsrMatrix.from_host(A)
    L = mpk.build_levels(dA, 0)
    P = mpk.plan(dA, L, p_max=4, order=order, wait_limit_ns=20_000_000)
    X = gen.vector(n, 1, stream=8)
    perm = L.perm.cpu().numpy() if order == mpk.ORDER_PLAN else np.arange(n)
    Xd = torch.from_numpy(np.ascontiguousarray(X[perm])).cuda()
    P.debug_drop_release(0, 1)
    P.apply(Xd, 4)
    with pytest.raises(mpk.MpkError) as e:
        P.sync_status()
    assert e.value.status == 4
    Y = P.apply(Xd, 4)
    P.sync_status()
    _same(Y.cpu().numpy(), oracle.mpk(A, X, 4)[:, perm])


@pytest.mark.parametrize("order", [0, 1])
def test_scattered_batch(mpk, order):
    mats = [_scattered(n, (9, 7, 8), 990 + n) for n in (30011, 25000, 7)]
    ps = [4, 3, 2]
    dAs = [mpk.CsrMatrix.from_host(A) for A in mats]
    B = mpk.batch_plan(dAs, ps, nrhs=2, order=order)
    perms = [mpk.build_levels(d, 0).perm.cpu().numpy() if order == mpk.ORDER_PLAN else np.arange(d.n) for d in dAs]
    Xh = [gen.vector(A.n, 2, stream=70 + i) for i, A in enumerate(mats)]
    Ys = B.apply([torch.from_numpy(np.ascontiguousarray(X[q])).cuda() for X, q in zip(Xh, perms)])
    for Y, A, X, p, q in zip(Ys, mats, Xh, ps, perms):
        _same(Y.cpu().numpy(), oracle.mpk(A, X, p)[:, q])


def _permuted_grid(mpk, side, dtype):
    """7-point Laplacian of side^3 with its rows and columns in random order, built on the GPU."""
    n = side ** 3
    g = torch.Generator(device="cuda").manual_seed(11)
    p = torch.randperm(n, generator=g, device="cuda")
    i = torch.arange(n, device="cuda")
    x, y, z = i % side, i // side % side, i // side ** 2
    rows, cols = [i], [i]
    for c, step in ((x, 1), (y, side), (z, side * side)):
        on = c + 1 < side
        rows += [i[on], i[on] + step]
        cols += [i[on] + step, i[on]]
    rows, cols = torch.cat(rows), torch.cat(cols)
    vals = torch.where(rows == cols, 6.0, -1.0)
    key, at = torch.sort(p[rows] * n + p[cols])
    rp = torch.searchsorted(key, torch.arange(n + 1, device="cuda") * n).int()
    return mpk.CsrMatrix(rp, (key % n).int(), vals[at].to(dtype), is_symmetric=True)


def _time(fn):
    best = float("inf")
    for _ in range(3):
        fn()
    for _ in range(7):
        e0, e1 = torch.cuda.Event(enable_timing=True), torch.cuda.Event(enable_timing=True)
        e0.record()
        for _ in range(5):
            fn()
        e1.record()
        e1.synchronize()
        best = min(best, e0.elapsed_time(e1) / 5)
    return best


@pytest.mark.parametrize("dtype", [torch.bfloat16, torch.float32])
def test_scattered_gathers_are_not_slower_than_on_the_ticketed_kernel(mpk, dtype):
    """Plan order, a permuted grid of 126^3: the default plan against the block shapes that run the
    ticketed kernel (0.60 of its speed with the large buffer, about the same with the smaller one)."""
    A = _permuted_grid(mpk, 126, dtype)
    L = mpk.build_levels(A, 0)
    X = torch.rand((A.n, 1), dtype=torch.float64, device="cuda")
    Y = torch.empty((9, A.n, 1), dtype=torch.float64, device="cuda")
    t = {}
    for shape in (0, 1, 2):
        P = mpk.plan(A, L, p_max=8, order=mpk.ORDER_PLAN, shape=shape)
        t[shape] = _time(lambda: P.apply(X, 8, Y=Y))
    assert t[0] < 1.25 * min(t[1], t[2]), t


def _shuffled_grid(mpk, side, window, dtype):
    """The same grid in its own order but for rows shuffled inside windows."""
    n = side ** 3
    i = torch.arange(n, device="cuda")
    g = torch.Generator(device="cuda").manual_seed(12)
    p = torch.argsort(i // window + 0.999 * torch.rand(n, generator=g, device="cuda", dtype=torch.float64))
    x, y, z = i % side, i // side % side, i // side ** 2
    rows, cols = [i], [i]
    for c, step in ((x, 1), (y, side), (z, side * side)):
        on = c + 1 < side
        rows += [i[on], i[on] + step]
        cols += [i[on] + step, i[on]]
    rows, cols = torch.cat(rows), torch.cat(cols)
    vals = torch.where(rows == cols, 6.0, -1.0)
    key, at = torch.sort(p[rows] * n + p[cols])
    rp = torch.searchsorted(key, torch.arange(n + 1, device="cuda") * n).int()
    return mpk.CsrMatrix(rp, (key % n).int(), vals[at].to(dtype), is_symmetric=True)


@pytest.mark.parametrize("dtype,accum", [(torch.float64, 0), (torch.bfloat16, 1)])
def test_a_numbering_without_locality_is_left_to_the_levels(mpk, dtype, accum):
    """A's order, 126^3 with its rows shuffled in windows of 10 000, recurrence of 32 steps: against the
    ticketed kernel, which gathers and scatters the vectors (0.46 to 0.56 of its speed in A's numbering)."""
    A = _shuffled_grid(mpk, 126, 10000, dtype)
    L = mpk.build_levels(A, 0)
    X = torch.rand((A.n, 1), dtype=torch.float64, device="cuda")
    out = torch.empty_like(X)
    c = np.ones(33)
    t = {}
    for shape in (0, 1, 2):
        P = mpk.plan(A, L, p_max=8, shape=shape, accum=accum)
        t[shape] = _time(lambda: P.cheb_filter(X, 32, c, scale=13.0, shift=6.0, out=out))
    assert t[0] < 1.25 * min(t[1], t[2]), t


@pytest.mark.parametrize("cache_bytes", [0, 4000000])
@pytest.mark.parametrize("val,accum", [("f64", 0), ("bf16", 1)])
def test_original_order_through_the_levels(mpk, cache_bytes, val, accum):
    """70^3 (343000 rows) shuffled in windows of 10 000: gathered into the levels' order, computed there
    and scattered, bit for bit: powers, into host memory too, the recurrence, whole and in pieces."""
    A = _shuffled_grid(mpk, 70, 10000, torch.float64 if val == "f64" else torch.bfloat16)
    host = gen.CSR(A.row_ptr.cpu().numpy(), A.col.cpu().numpy(), A.val.double().cpu().numpy())
    L = mpk.build_levels(A, 0)
    P = mpk.plan(A, L, p_max=5, accum=accum, cache_bytes=cache_bytes)
    X = gen.vector(A.n, 1, stream=9)
    Xd = torch.from_numpy(X).cuda()
    want = oracle.mpk_acc32(host, X, 5) if accum else oracle.mpk(host, X, 5)
    Y = torch.full((6, A.n, 1), float("nan"), dtype=torch.float64, device="cuda")
    for p in (5, 1):
        Y.fill_(float("nan"))
        P.apply(Xd, p, Y=Y)
        P.sync_status()
        _same(Y[:p + 1].cpu().numpy(), want[:p + 1])
    Yh = P.apply_host(torch.from_numpy(X).pin_memory(), 5)
    torch.cuda.synchronize()
    P.sync_status()
    _same(Yh.numpy(), want)
    if not accum:
        c = np.linspace(1.0, -0.5, 9)
        ref = oracle.cheb(host, X, 8, c, scale=13.0, shift=6.0)
        _same(P.cheb_filter(Xd, 8, c, scale=13.0, shift=6.0).cpu().numpy(), ref)
        S = P.cheb_begin(Xd, P.cheb_state(), c[0])
        P.cheb_advance(S, 0, 3, c, scale=13.0, shift=6.0)
        P.cheb_advance(S, 3, 8, c, scale=13.0, shift=6.0)
        _same(P.cheb_finish(S).cpu().numpy(), ref)
        P.sync_status()
