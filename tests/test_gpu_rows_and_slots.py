"""Row pointers, entry weights and duplicate removal at the edges of their tiles (2048 rows, 2048 entries, 2048 candidates), with empty rows
before, between and behind the others."""
import numpy as np
import pytest

torch = pytest.importorskip("torch")
pytestmark = pytest.mark.gpu


def destinations(kind, n, m, rng):
    if kind == "one row":
        return np.full(m, n // 2)
    if kind == "last row":
        return np.full(m, n - 1)
    if kind == "first rows":
        return rng.integers(0, min(n, 3), m)
    if kind == "far apart":
        return rng.choice(np.array([0, n // 3, n - 1]), m)
    return rng.integers(0, n, m)


@pytest.mark.parametrize("n,m", [(1, 1), (1, 5000), (2047, 2048), (2048, 2047), (2049, 6145), (40_000, 2048), (300_001, 10), (300_001, 40_961),
                                 (5000, 0)])
@pytest.mark.parametrize("kind", ["one row", "last row", "first rows", "far apart", "any"])
@pytest.mark.parametrize("flags", [0, 2])                     # without and with duplicate removal
def test_rows_and_weights(n, m, kind, flags):
    import paper_2104_03058_b200 as g
    rng = np.random.default_rng(n + m)
    src, dst = rng.integers(0, max(1, n // 2), m).astype(np.int32), destinations(kind, n, m, rng).astype(np.int32)
    order = np.lexsort((src, dst))
    s, d, p = src[order], dst[order], order
    if flags and m:
        first = np.r_[True, (s[1:] != s[:-1]) | (d[1:] != d[:-1])]
        s, d, p = s[first], d[first], p[first]
    row_ptr = np.searchsorted(d, np.arange(n + 1))
    deg = np.diff(row_ptr)
    dinv = np.where(deg > 0, 1 / np.sqrt(np.maximum(deg, 1).astype(np.float64)), 0).astype(np.float32)
    csr = g.build_csr(n, torch.from_numpy(src).cuda(), torch.from_numpy(dst).cuda(), flags)
    assert csr.nnz == len(s) and csr.max_degree == deg.max()
    for name, want in (("row_ptr", row_ptr), ("col_idx", s), ("perm", p), ("dinv_sqrt", dinv), ("edge_weight", dinv[s] * dinv[d])):
        np.testing.assert_array_equal(getattr(csr, name).cpu().numpy(), want, err_msg=name)
    assert np.array_equal(np.sort(csr.row_order.cpu().numpy()), np.arange(n))


@pytest.mark.parametrize("n,m", [(1, 1), (1, 5000), (2047, 2048), (2048, 2047), (2049, 6145), (40_000, 2048), (300_001, 10), (300_001, 40_961),
                                 (5000, 0), (70_001, 148 * 4 * 8192 + 1)])
@pytest.mark.parametrize("kind", ["one row", "last row", "first rows", "far apart", "any"])
def test_light_build(n, m, kind):
    """The same edges through the one-shot path, whose last sweep writes the entries and counts the degrees; sums of whole numbers."""
    import paper_2104_03058_b200 as g
    rng = np.random.default_rng(n + m)
    src, dst = rng.integers(0, n, m).astype(np.int32), destinations(kind, n, m, rng).astype(np.int32)
    x = rng.integers(-8, 9, (n, 4)).astype(np.float32)
    ds, dd, dx = (torch.from_numpy(a).cuda() for a in (src, dst, x))
    deg = np.bincount(dst, minlength=n)
    sums = np.stack([np.bincount(dst, weights=x[src, j], minlength=n) for j in range(4)], axis=1)
    rdeg = np.where(deg > 0, 1 / np.maximum(deg, 1).astype(np.float64), 0).astype(np.float32)
    got = g.oneshot("sage", n, ds, dd, dx).cpu().numpy()
    np.testing.assert_array_equal(got, sums.astype(np.float32) * rdeg[:, None])
    dinv = np.where(deg > 0, 1 / np.sqrt(np.maximum(deg, 1).astype(np.float64)), 0)
    want, scale = (np.stack([np.bincount(dst, weights=dinv[src] * dinv[dst] * v[src, j], minlength=n) for j in range(4)], axis=1)
                   for v in (x.astype(np.float64), np.abs(x).astype(np.float64)))
    got = g.oneshot("gcn", n, ds, dd, dx).cpu().numpy()
    assert (np.abs(got - want) <= 1e-5 * scale + 1e-6).all()


def kernel_ms(g, call, kernel, rounds=5):
    """least time of one launch of `kernel` over a few calls"""
    call()
    least = float("inf")
    for _ in range(rounds):
        g.kernel_timing_enable(True)
        call()
        torch.cuda.synchronize()
        least = min(least, g.kernel_timing_read()[kernel][0])
        g.kernel_timing_enable(False)
    return least


@pytest.mark.parametrize("rows", ["first", "both ends", "any"])
def test_entry_weights_do_not_wait_for_rows_without_entries(rows):
    """A few thousand entries on 2 M vertices: a handful of blocks must not walk millions of row pointers (which took 2 ms; the same
    entries on 1000 vertices about 6 us)."""
    import paper_2104_03058_b200 as g
    n, m, x = 2_000_000, 4000, torch.ones((2_000_000, 4), device="cuda")
    rng = np.random.default_rng(5)
    src, dst = rng.integers(0, 1000, m), rng.integers(0, 1000, m)
    few = [torch.from_numpy(a.astype(np.int32)).cuda() for a in (src, dst)]
    dst = {"first": dst, "both ends": np.where(dst % 2, dst, n - 1 - dst), "any": rng.integers(0, n, m)}[rows]
    many = [torch.from_numpy(a.astype(np.int32)).cuda() for a in (src, dst)]
    short = kernel_ms(g, lambda: g.oneshot("gcn", 1000, *few, x[:1000]), "slot_weights")
    assert kernel_ms(g, lambda: g.oneshot("gcn", n, *many, x), "slot_weights") < 10 * short + 0.02
    assert (g.oneshot("sage", n, *many, x).sum(1) > 0).sum() == len(np.unique(dst))


def test_row_pointers_of_one_long_row():
    """The rows of the pieces of one row of 8 M entries are not written by a single thread (which took 20 us)."""
    import paper_2104_03058_b200 as g
    n, m, x = 5000, 8_000_000, torch.ones((5000, 4), device="cuda")
    src = torch.randint(n, (m,), dtype=torch.int32, device="cuda")
    one, every = torch.full_like(src, 7), torch.randint(n, (m,), dtype=torch.int32, device="cuda")
    spread = kernel_ms(g, lambda: g.oneshot("gcn", n, src, every, x), "rows_from_degrees")
    assert kernel_ms(g, lambda: g.oneshot("gcn", n, src, one, x), "rows_from_degrees") < spread + 0.008


@pytest.mark.parametrize("rows", [1, 10, 3000])
def test_long_rows_are_counted_as_fast_as_short_ones(rows):
    """The last sweep of the one-shot path adds a run of equal destinations once, not once per 32 entries (which took twice as long for
    rows of millions of entries)."""
    import paper_2104_03058_b200 as g
    n, m = 130_000, 20_000_000
    src, dst = (torch.randint(n, (m,), dtype=torch.int32, device="cuda") for _ in range(2))
    x, few = torch.ones((n, 4), device="cuda"), dst % rows * (n // rows)
    spread = kernel_ms(g, lambda: g.oneshot("sage", n, src, dst, x), "radix_sweep")
    assert kernel_ms(g, lambda: g.oneshot("sage", n, src, few, x), "radix_sweep") < 1.4 * spread


@pytest.mark.parametrize("m", [31, 32, 33, 2047, 2048, 6200, 148 * 4 * 8192 + 77])
def test_degrees_of_runs(m):
    """Runs of lengths around the 32 entries that a warp looks at together, in tiles of both sizes."""
    import paper_2104_03058_b200 as g
    rng = np.random.default_rng(m)
    for lengths in (rng.integers(1, 100, m), rng.choice([31, 32, 33, 63, 64, 65, 96], m), rng.choice([1, 2000, 2100], m), np.full(m, 32)):
        dst = np.repeat(np.arange(m), lengths)[:m].astype(np.int32)
        n = int(dst[-1]) + 2
        src, dst = rng.integers(0, n, m).astype(np.int32), dst[rng.permutation(m)]
        got = g.oneshot("sage", n, torch.from_numpy(src).cuda(), torch.from_numpy(dst).cuda(), torch.from_numpy(np.arange(n, dtype=np.float32)[:, None] % 64).cuda())
        deg = np.bincount(dst, minlength=n)
        want = (np.bincount(dst, weights=src % 64, minlength=n).astype(np.float32) * np.where(deg > 0, 1 / np.maximum(deg, 1), 0).astype(np.float32))
        np.testing.assert_array_equal(got.cpu().numpy()[:, 0], want)


@pytest.mark.parametrize("rows", [1000, 8_000_000])
def test_row_pointers_of_many_vertices(rows):
    """Blocks of vertices without entries find their row pointers without searching all keys thread by thread (which took twice the time
    of the sweep over the rows)."""
    import paper_2104_03058_b200 as g
    n, m = 8_000_000, 1_000_000
    src, dst = (torch.randint(k, (m,), dtype=torch.int32, device="cuda") for k in (n, rows))
    times = [kernel_ms(g, lambda: g.build_csr(n, src, dst, 0), k) for k in ("rows_and_degrees", "radix_sweep_rows")]
    assert times[0] < (1.6 if rows == 1000 else 2.0) * times[1]
    csr, deg = g.build_csr(n, src, dst, 0), torch.bincount(dst, minlength=n)
    assert torch.equal(csr.row_ptr.long(), torch.cat([deg.new_zeros(1), deg.cumsum(0)]))
