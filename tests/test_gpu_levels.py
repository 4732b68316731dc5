"""The level search (one cooperative launch) on graphs that are hard on its schedule: narrow levels
of much work, which one block expands alone while the others wait for it, and many components."""
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


def _chain_of_stars(mpk, hubs, leaves):
    """Hub h is vertex h * (leaves + 1), its leaves follow it, and it is linked to hubs h - 1, h + 1."""
    w, n = leaves + 1, hubs * (leaves + 1)
    hub = torch.arange(hubs, device="cuda") * w
    deg = torch.ones(n, dtype=torch.int64, device="cuda")
    deg[hub] = leaves + 2
    deg[0] -= 1
    deg[hub[-1]] -= 1
    rp = torch.zeros(n + 1, dtype=torch.int64, device="cuda")
    rp[1:] = deg.cumsum(0)
    col = torch.empty(int(rp[-1]), dtype=torch.int32, device="cuda")
    i = torch.arange(n, device="cuda")
    leaf = i % w != 0
    col[rp[:-1][leaf]] = (i // w * w)[leaf].int()
    first = rp[:-1][hub]
    col[first[1:]] = hub[:-1].int()
    first = first + (torch.arange(hubs, device="cuda") > 0)
    for j in range(leaves):
        col[first + j] = (hub + 1 + j).int()
    col[(first + leaves)[:-1]] = hub[1:].int()
    return mpk.CsrMatrix(rp.int(), col, torch.ones(col.numel(), dtype=torch.float64, device="cuda"), is_symmetric=True)


def test_narrow_levels_of_long_rows(mpk):
    """Levels of 512 vertices with one row of 513 entries (about 0.2 ms each): 16384 of them take
    longer than one wait of the other blocks may.  The levels are the vertices in order: hub 0, then
    each hub's leaves with the next hub."""
    hubs, leaves = 16384, 511
    A = _chain_of_stars(mpk, hubs, leaves)
    L = mpk.build_levels(A, root=0)
    assert L.num_levels == hubs + 1
    ptr = torch.as_tensor(L.level_ptr).cpu().numpy()
    want = np.concatenate([[0], 1 + np.arange(hubs + 1) * (leaves + 1)])
    want[-1] = A.n
    assert np.array_equal(ptr, want)
    assert torch.equal(L.perm, torch.arange(A.n, dtype=torch.int32, device="cuda"))


def _components(kind, n):
    """Edges of a graph of n vertices with many components."""
    i = np.arange(n)
    if kind == "isolated":
        return i[:0], i[:0]
    if kind == "far":  # one component of every vertex but 7, which lie 8191, 8192, 8193 .. apart
        skip = np.cumsum([100, 8191, 8192, 8193, 2, 9000, 1])
        v = np.setdiff1d(i, skip)
        return v[:-1], v[1:]
    if kind == "stars":  # wide levels (700 leaves) between narrow ones, then vertices without edges
        hub = i // 701 * 701
        on = (i != hub) & (i < n - 3000)
        return hub[on], i[on]
    return i[:-1][i[:-1] % 3 > 0], i[1:][i[:-1] % 3 > 0]  # "paths" of three vertices


@pytest.mark.parametrize("symmetric", [True, False])
@pytest.mark.parametrize("kind,n", [("isolated", 1), ("isolated", 1500), ("far", 45000), ("stars", 20000), ("paths", 5000)])
def test_many_components(mpk, kind, n, symmetric):
    """The search goes on from the smallest untouched vertex, near (found beside the narrow levels)
    or far (found by the whole grid), from the first vertex and from one in the middle."""
    r, c = _components(kind, n)
    if symmetric:
        r, c = np.concatenate([r, c]), np.concatenate([c, r])
    A = gen.from_coo(n, r, c, np.ones(r.size))
    dA = mpk.CsrMatrix.from_host(A, is_symmetric=symmetric)
    for root in (0, n // 2):
        L = mpk.build_levels(dA, root=root)
        lo, pe, ip, lp = oracle.levels(A, root)
        assert L.num_levels == lp.size - 1
        assert np.array_equal(L.level_ptr.cpu().numpy(), lp)
        assert np.array_equal(L.perm.cpu().numpy(), pe)
        assert np.array_equal(L.level_of.cpu().numpy(), lo)
