"""The sort behind the CSR build at the edges of its tiles and block shapes, against numpy's stable sort: tile sizes 2048 and
8192 (the larger from 4 * 148 * 8192 candidates on), key and value in one word or apart, digits that are all equal."""
import numpy as np
import pytest

torch = pytest.importorskip("torch")
pytestmark = pytest.mark.gpu

SL, DD, SY, LIGHT = 1, 2, 4, 8
LARGE = 4 * 148 * 8192


@pytest.fixture(scope="module")
def g():
    import paper_2104_03058_b200 as lib
    lib.lib()
    return lib


def reference(n, src, dst, flags):
    """row_ptr, col, perm by a stable sort (or by destination only for the light build)"""
    e = len(src)
    s, d, p = src.astype(np.int64), dst.astype(np.int64), np.arange(e)
    if flags & SY:
        rev = s != d
        s, d, p = np.concatenate([s, d[rev]]), np.concatenate([d, s[rev]]), np.concatenate([p, e + p[rev]])
    if flags & SL:
        keep = s != d
        own = np.arange(n)
        s, d, p = np.concatenate([s[keep], own]), np.concatenate([d[keep], own]), np.concatenate([p[keep], np.full(n, -1)])
    order = np.argsort(d if flags & LIGHT else d * n + s, kind="stable")
    s, d, p = s[order], d[order], p[order]
    if flags & DD:
        first = np.ones(len(s), bool)
        first[1:] = (s[1:] != s[:-1]) | (d[1:] != d[:-1])
        s, d, p = s[first], d[first], p[first]
    return np.searchsorted(d, np.arange(n + 1)), s, p


def check(g, n, src, dst, flags):
    csr = g.build_csr(n, torch.from_numpy(src).cuda(), torch.from_numpy(dst).cuda(), flags)
    row_ptr, col, perm = reference(n, src, dst, flags)
    assert csr.nnz == len(col)
    np.testing.assert_array_equal(csr.row_ptr.cpu().numpy(), row_ptr)
    np.testing.assert_array_equal(csr.col_idx.cpu().numpy(), col)
    np.testing.assert_array_equal(csr.perm.cpu().numpy(), perm)
    deg = np.diff(row_ptr)
    assert csr.max_degree == deg.max()
    assert csr.bin_count == [int(((deg > lo) & (deg <= hi)).sum()) for lo, hi in
                             ((-1, 8), (8, 32), (32, 128), (128, 2048), (2048, 1 << 31))]
    order = csr.row_order.cpu().numpy()
    assert np.array_equal(np.sort(order), np.arange(n))
    c = deg[order].astype(np.int64)
    o = np.int64(np.log2(np.maximum(c - 1, 8)))                     # classes: exact degree to 8, quarter octaves, hub rows
    cls = np.where(c <= 8, c, np.where(c > 2048, 41, 9 + (o - 3) * 4 + ((c - 1) >> (o - 2) & 3)))
    assert ((cls[1:] > cls[:-1]) | ((cls[1:] == cls[:-1]) & (order[1:] > order[:-1]))).all()


@pytest.mark.parametrize("m", [1, 31, 2047, 2048, 2049, 4097, 148 * 4 * 2048 + 5, LARGE - 1, LARGE, LARGE + 8191])
@pytest.mark.parametrize("ids", [np.int32, np.int64])
def test_tile_edges(g, m, ids):
    rng = np.random.default_rng(m)
    n = 1000 if m < 100_000 else 70_001
    check(g, n, rng.integers(0, n, m).astype(ids), rng.integers(0, n, m).astype(ids), 0)


@pytest.mark.parametrize("flags", [SL, SY, SL | SY | DD, DD, LIGHT | SL | SY])
def test_candidates_that_are_no_plain_edges_fill_tiles(g, flags):
    rng = np.random.default_rng(flags)
    n, e = 30_000, LARGE // 2 + 777                                 # reverses and loops begin inside a tile
    check(g, n, rng.integers(0, n, e).astype(np.int32), rng.integers(0, n, e).astype(np.int32), flags)


@pytest.mark.parametrize("m", [300_000, LARGE + 1])
@pytest.mark.parametrize("flags", [0, DD, SL, LIGHT])
def test_key_and_value_apart(g, m, flags):
    n = (1 << 22) + 3                                               # 23 + 23 key bits and at least 19 value bits: two words
    rng = np.random.default_rng(m + flags)
    check(g, n, rng.integers(0, n, m).astype(np.int32), rng.integers(n - 5000, n, m).astype(np.int32), flags)


@pytest.mark.parametrize("m", [10_000, LARGE + 100])
@pytest.mark.parametrize("kind", ["one pair", "one destination", "pairs in turn", "sorted"])
def test_equal_and_ordered_digits(g, m, kind):
    n = 5000
    rng = np.random.default_rng(7)
    i = np.arange(m)
    src, dst = {"one pair": (np.full(m, 4999), np.full(m, 17)), "one destination": (rng.integers(0, n, m), np.full(m, 3)),
                "pairs in turn": (i // 2 % n, i // 3 % n), "sorted": (i * n // m, i * n // m)}[kind]
    check(g, n, src.astype(np.int32), dst.astype(np.int32), 0)


# ------------------------------------------------------------------ the give-up path, drilled without a fault

GUARD = 1 << 20


def guarded(nbytes):
    """a buffer of ones (leftover words that look like published sums) with guard bytes on both sides"""
    whole = torch.full((nbytes + 2 * GUARD,), 0xFF, dtype=torch.uint8, device="cuda")
    whole[:GUARD] = whole[GUARD + nbytes:] = 0xAB
    return whole, whole[GUARD:GUARD + nbytes]


# (vertices, candidates, passes): key and value in one word and apart
@pytest.mark.parametrize("n,m,passes", [(70_001, 200_000, 4), ((1 << 22) + 3, 300_000, 6)])
@pytest.mark.parametrize("sweep", ["first", "second", "last", "rows"])
@pytest.mark.parametrize("flags", [0, DD | SL])
def test_a_tile_that_is_never_published_ends_the_build_with_an_error(g, n, m, passes, sweep, flags):
    rng = np.random.default_rng(m)
    src, dst = (rng.integers(0, n, m).astype(np.int32) for _ in range(2))
    ds, dd = torch.from_numpy(src).cuda(), torch.from_numpy(dst).cuda()
    pb, sb = g.csr_workspace_bytes(n, m, flags)
    (p_all, persistent), (s_all, scratch) = guarded(pb), guarded(sb)
    g.debug_build_fault(1024, {"first": 0, "second": 1, "last": passes - 1, "rows": passes}[sweep])
    with pytest.raises(g.GnnfdError) as err:
        g.build_csr(n, ds, dd, flags, persistent=persistent, scratch=scratch)
    assert err.value.status == g.CUDA_ERROR
    torch.cuda.synchronize()
    for whole, nbytes in ((p_all, pb), (s_all, sb)):
        assert bool((whole[:GUARD] == 0xAB).all()) and bool((whole[GUARD + nbytes:] == 0xAB).all())
    # the drill is one-shot: the next build, from the same buffers, is an ordinary one
    csr = g.build_csr(n, ds, dd, flags, persistent=persistent, scratch=scratch)
    row_ptr, col, perm = reference(n, src, dst, flags)
    np.testing.assert_array_equal(csr.row_ptr.cpu().numpy(), row_ptr)
    np.testing.assert_array_equal(csr.col_idx.cpu().numpy(), col)
    np.testing.assert_array_equal(csr.perm.cpu().numpy(), perm)


# the one-shot path, whose words are keys alone (17 destination bits, two digits of 9; 23 bits, three): each sweep over the edges, the last of which writes the
# entries, the rows' order, and the chain of the row pointers' sums
@pytest.mark.parametrize("n,passes", [(70_001, 2), ((1 << 22) + 3, 3)])
@pytest.mark.parametrize("sweep", ["first", "last", "rows", "sums"])
@pytest.mark.parametrize("model", ["gcn", "sage"])
def test_a_light_build_that_gives_up_ends_the_call_with_an_error(g, n, passes, sweep, model):
    m = 200_000
    rng = np.random.default_rng(m)
    src, dst = (rng.integers(0, n, m).astype(np.int32) for _ in range(2))
    ds, dd, x = torch.from_numpy(src).cuda(), torch.from_numpy(dst).cuda(), torch.randint(-8, 9, (n, 4), device="cuda").float()
    need = g.oneshot_workspace_bytes(n, m, 0, 4)
    s_all, scratch = guarded(need)
    out = torch.full((n, 4), 7.0, device="cuda")
    g.debug_build_fault(1024, {"first": 0, "last": passes - 1, "rows": passes, "sums": passes + 1}[sweep])
    with pytest.raises(g.GnnfdError) as err:
        g.oneshot(model, n, ds, dd, x, out=out, scratch=scratch)
    assert err.value.status == g.CUDA_ERROR
    torch.cuda.synchronize()
    assert bool((s_all[:GUARD] == 0xAB).all()) and bool((s_all[GUARD + need:] == 0xAB).all()) and bool((out == 7.0).all())
    got = g.oneshot(model, n, ds, dd, x, out=out, scratch=scratch)
    csr = g.build_csr(n, ds, dd, LIGHT)
    assert torch.equal(got, (g.aggregate_gcn if model == "gcn" else g.aggregate_sage)(csr, x))


def test_the_drill_refuses_row_sums_where_there_are_none(g):
    ids = torch.zeros(200_000, dtype=torch.int32, device="cuda")
    x = torch.zeros((70_001, 4), device="cuda")
    for sweep, call in ((5, lambda: g.build_csr(70_001, ids, ids, 0)), (5, lambda: g.oneshot("gcn", 70_001, ids, ids, x, flags=DD)),
                        (3, lambda: g.oneshot("gcn", 2000, ids, ids, x[:2000]))):       # edge ids, duplicate removal; a single tile of rows
        g.debug_build_fault(1024, sweep)
        with pytest.raises(g.GnnfdError) as err:
            call()
        assert err.value.status == g.INVALID_ARG


def test_the_drill_refuses_sweeps_that_nobody_would_miss(g):
    src = torch.arange(3000, dtype=torch.int32, device="cuda")
    for sweep in (0, 9):                                             # one tile of edges only; no such sweep
        g.debug_build_fault(1024, sweep)
        with pytest.raises(g.GnnfdError) as err:
            g.build_csr(3000, src[:2000], src[1000:], 0)
        assert err.value.status == g.INVALID_ARG
    assert g.build_csr(3000, src[:2000], src[1000:], 0).nnz == 2000
