"""Large inputs whose keys and values do not share a word: the first sweep makes buckets of the destination's highest digit, the others sort each
bucket by itself."""
import numpy as np
import pytest

from test_gpu_sort_sweeps import DD, GUARD, LARGE, LIGHT, SL, SY, check, guarded, reference

torch = pytest.importorskip("torch")
pytestmark = pytest.mark.gpu

N = (1 << 21) + 5                                                  # 22 + 22 key bits and 23 value bits


@pytest.fixture(scope="module")
def g():
    import paper_2104_03058_b200 as lib
    lib.lib()
    return lib


def destinations(kind, m, rng):
    if kind == "one bucket":
        return rng.integers(0, 1000, m)
    if kind == "two far apart":
        return rng.choice(np.array([1, N - 1]), m)
    if kind == "tiles that are just full":                         # 8192 in each of the first buckets, the rest in the last one
        return np.concatenate([np.arange(8192 * 20) // 8192 << 13, np.full(m - 8192 * 20, N - 1)])[rng.permutation(m)]
    return rng.integers(0, N, m)


@pytest.mark.parametrize("kind", ["one bucket", "two far apart", "tiles that are just full", "any"])
@pytest.mark.parametrize("flags,ids", [(0, np.int32), (DD, np.int64), (SL | SY | DD, np.int32), (LIGHT | SL, np.int32)])
def test_buckets(g, kind, flags, ids):
    m = LARGE + 4321
    rng = np.random.default_rng(m + flags)
    check(g, N, rng.integers(0, N, m).astype(ids), destinations(kind, m, rng).astype(ids), flags)


@pytest.mark.parametrize("sweep", [0, 5])                          # the one that makes the buckets; the rows', after 5 over the edges
def test_a_tile_that_is_never_published_ends_the_build_with_an_error(g, sweep):
    rng = np.random.default_rng(sweep)
    src, dst = (rng.integers(0, N, LARGE).astype(np.int32) for _ in range(2))
    ds, dd = torch.from_numpy(src).cuda(), torch.from_numpy(dst).cuda()
    pb, sb = g.csr_workspace_bytes(N, LARGE, 0)
    (p_all, persistent), (s_all, scratch) = guarded(pb), guarded(sb)
    g.debug_build_fault(1024, sweep)
    with pytest.raises(g.GnnfdError) as err:
        g.build_csr(N, ds, dd, 0, persistent=persistent, scratch=scratch)
    assert err.value.status == g.CUDA_ERROR
    torch.cuda.synchronize()
    for whole, nbytes in ((p_all, pb), (s_all, sb)):
        assert bool((whole[:GUARD] == 0xAB).all()) and bool((whole[GUARD + nbytes:] == 0xAB).all())
    csr = g.build_csr(N, ds, dd, 0, persistent=persistent, scratch=scratch)
    row_ptr, col, perm = reference(N, src, dst, 0)
    np.testing.assert_array_equal(csr.row_ptr.cpu().numpy(), row_ptr)
    np.testing.assert_array_equal(csr.col_idx.cpu().numpy(), col)
    np.testing.assert_array_equal(csr.perm.cpu().numpy(), perm)


def test_the_drill_refuses_sweeps_inside_buckets(g):
    ids = torch.zeros(LARGE, dtype=torch.int32, device="cuda")
    for sweep in (1, 4):
        g.debug_build_fault(1024, sweep)
        with pytest.raises(g.GnnfdError) as err:
            g.build_csr(N, ids, ids, 0)
        assert err.value.status == g.INVALID_ARG


@pytest.mark.parametrize("flags", [0, DD, LIGHT])
def test_words_that_fill_64_bits(g, flags):
    """2^25 - 1 vertices and 4.85 to 8.4 M candidates: 41 key bits and 23 value bits.  Out of buffers sized for one more vertex, with which
    there are no buckets."""
    n, m = (1 << 25) - 1, LARGE + 12_345
    rng = np.random.default_rng(flags)
    src = rng.integers(0, n, m).astype(np.int32)
    dst = np.where(np.arange(m) % 3 == 0, n - 1, rng.integers(n // 2, n, m)).astype(np.int32)
    src[:9], src[9:18], dst[:18] = n - 1, 0, n - 1
    pb, sb = g.csr_workspace_bytes(n + 1, m, flags)
    persistent, scratch = (torch.empty(b, dtype=torch.uint8, device="cuda") for b in (pb, sb))
    csr = g.build_csr(n, torch.from_numpy(src).cuda(), torch.from_numpy(dst).cuda(), flags, persistent=persistent, scratch=scratch)
    row_ptr, col, perm = reference(n, src, dst, flags)
    for name, want in (("row_ptr", row_ptr), ("col_idx", col), ("perm", perm)):
        np.testing.assert_array_equal(getattr(csr, name).cpu().numpy(), want, err_msg=name)
