"""Features whose rows or chunks do not start on 16-byte boundaries: the aligned copy that a larger scratch buffer allows, against the
oracle and, bit for bit, against features laid out aligned; and long rows shared by several warps of a block."""
import numpy as np
import pytest

import oracle as orc

torch = pytest.importorskip("torch")
pytestmark = pytest.mark.gpu


@pytest.fixture(scope="module")
def g():
    import paper_2104_03058_b200 as lib
    lib.lib()
    return lib


@pytest.fixture(scope="module")
def graph(g):
    rng = np.random.default_rng(5)
    n, e = 1500, 1_200_000
    dst = np.where(rng.random(e) < 0.2, 7, rng.integers(0, n - 1, e)).astype(np.int32)      # a hub row and an empty one
    src = rng.integers(0, n, e).astype(np.int32)
    row_ptr, col, _ = orc.build_csr(n, src, dst, 0)
    return g.build_csr(n, torch.from_numpy(src).cuda(), torch.from_numpy(dst).cuda()), row_ptr, col


def scratch(nbytes):
    return torch.empty(nbytes, dtype=torch.uint8, device="cuda")


@pytest.mark.parametrize("model", ["gcn", "sage"])
@pytest.mark.parametrize("dtype", [torch.float32, torch.bfloat16])
@pytest.mark.parametrize("f,ld,cw", [(57, 57, 57), (59, 64, 35), (66, 67, 64), (130, 130, 33), (301, 301, 64), (305, 306, 305)])
def test_aligned_copy(g, graph, model, dtype, f, ld, cw):
    csr, row_ptr, col = graph
    fn = {"gcn": g.aggregate_gcn, "sage": g.aggregate_sage}[model]
    gen = torch.Generator().manual_seed(f * 1000 + cw)
    x = torch.full((csr.n, ld), float("nan"), dtype=dtype)                                  # padding never counts
    x[:, :f] = torch.randn((csr.n, f), generator=gen).to(dtype)
    x = x.cuda()
    small, best = g.aggregate_workspace_bytes(csr, f), g.aggregate_best_workspace_bytes(csr, x, f, cw)
    assert best > small > 0
    plain = fn(csr, x, f=f, chunk_width=cw, scratch=scratch(small))
    assert torch.equal(plain, fn(csr, x, f=f, chunk_width=cw, scratch=scratch(best - 256)))      # not enough for the copy
    copied = fn(csr, x, f=f, chunk_width=cw)
    assert torch.equal(copied, fn(csr, x, f=f, chunk_width=cw, scratch=scratch(best)))
    if cw >= f or cw % 8 == 0:
        wide = torch.zeros((csr.n, (f + 15) // 16 * 16), dtype=dtype, device="cuda")
        wide[:, :f] = x[:, :f]
        assert torch.equal(copied, fn(csr, wide, f=f, chunk_width=cw))
    want, scale = orc.aggregate(model, row_ptr, col, np.ascontiguousarray(x[:, :f].float().cpu().numpy()), f)
    for got in (plain, copied):
        assert (np.abs(got.cpu().numpy() - want) <= 1e-5 * scale + 1e-6).all()
    if model == "gcn":
        out = torch.empty((csr.n, f), device="cuda")
        assert torch.equal(plain, g.aggregate_gcn_static(csr, x, f=f, chunk_width=cw, out=out))


def test_shifted_rows(g, graph):
    csr, _, _ = graph
    base = torch.randn((csr.n, 72), device="cuda")
    for shift in (1, 2, 3, 5):
        part = base[:, shift:shift + 64]
        assert torch.equal(g.aggregate_gcn(csr, part), g.aggregate_gcn(csr, part.contiguous()))


def test_where_no_copy_is_planned(g, graph):
    n = 50_000
    rng = np.random.default_rng(3)
    csr = g.build_csr(n, *(torch.from_numpy(rng.integers(0, n, 3 * n).astype(np.int32)).cuda() for _ in range(2)))
    x = torch.randn((n, 301), device="cuda")
    assert g.aggregate_best_workspace_bytes(csr, x) == g.aggregate_workspace_bytes(csr, 301)         # few entries per row
    x = torch.randn((graph[0].n, 31), device="cuda")
    assert g.aggregate_best_workspace_bytes(graph[0], x) == g.aggregate_workspace_bytes(graph[0], 31)  # narrow fp32
    x = torch.randn((graph[0].n, 64), device="cuda")
    assert g.aggregate_best_workspace_bytes(graph[0], x) == g.aggregate_workspace_bytes(graph[0], 64)  # aligned


@pytest.mark.parametrize("dtype", [torch.float32, torch.bfloat16])
@pytest.mark.parametrize("heads,dim,ld,cw", [(4, 7, 28, 28), (4, 7, 32, 7), (5, 3, 15, 15), (3, 20, 61, 40), (6, 4, 24, 24), (2, 33, 66, 33),
                                             (1, 41, 41, 41), (8, 7, 56, 14)])
def test_padded_heads(g, graph, dtype, heads, dim, ld, cw):
    csr, row_ptr, col = graph
    f = heads * dim
    gen = torch.Generator().manual_seed(f)
    z = torch.full((csr.n, ld), float("nan"), dtype=dtype)
    z[:, :f] = torch.randn((csr.n, f), generator=gen).to(dtype)
    a = [torch.randn((heads, dim), generator=gen) * 0.3 for _ in range(2)]
    dev = [t.cuda() for t in (z, *a)]
    small = scratch(g.gat_workspace_bytes(csr, heads, dim))
    plain = g.aggregate_gat(csr, *dev, heads, dim, 0.2, chunk_width=cw, scratch=small)
    out = torch.full((csr.n, f + 3), 9.0, device="cuda")
    got = g.aggregate_gat(csr, *dev, heads, dim, 0.2, chunk_width=cw, out=out)
    assert (out[:, f:] == 9.0).all()
    want, scale = orc.aggregate_gat(row_ptr, col, np.ascontiguousarray(z[:, :f].float().numpy()), a[0].numpy(), a[1].numpy(), heads, dim, 0.2)
    for t in (plain, got[:, :f]):
        assert (np.abs(t.cpu().numpy() - want) <= 1e-5 * scale + 1e-6).all()


@pytest.fixture(scope="module")
def long_graph(g):
    rng = np.random.default_rng(6)
    n, e = 5000, 7_100_000                                  # 4 columns put 14 M lanes on a chunk: copies start at 10 M
    dst = np.where(rng.random(e) < 0.001, 7, rng.integers(0, n - 1, e)).astype(np.int32)
    src = rng.integers(0, n, e).astype(np.int32)
    row_ptr, col, _ = orc.build_csr(n, src, dst, 0)
    return g.build_csr(n, torch.from_numpy(src).cuda(), torch.from_numpy(dst).cuda()), row_ptr, col


# Which features get an aligned copy, and how large it may be: from 3 bf16 / 33 fp32 columns and at most 8/3 of the features; heads
# of three columns or more in chunks of more than four.
@pytest.mark.parametrize("dtype,f,ld,cw,copied", [
    (torch.bfloat16, 17, 17, 1, False), (torch.bfloat16, 17, 17, 2, False), (torch.bfloat16, 19, 21, 3, True), (torch.bfloat16, 5, 5, 5, True),
    (torch.bfloat16, 23, 23, 7, True), (torch.bfloat16, 23, 23, 8, True), (torch.bfloat16, 26, 27, 9, True), (torch.bfloat16, 41, 41, 41, True),
    (torch.float32, 65, 65, 32, False), (torch.float32, 66, 67, 33, True), (torch.float32, 40, 41, 40, True)])
@pytest.mark.parametrize("model", ["gcn", "sage"])
def test_what_is_copied(g, long_graph, model, dtype, f, ld, cw, copied):
    csr, row_ptr, col = long_graph
    fn = {"gcn": g.aggregate_gcn, "sage": g.aggregate_sage}[model]
    x = torch.full((csr.n, ld), float("nan"), dtype=dtype)
    x[:, :f] = torch.randn((csr.n, f), generator=torch.Generator().manual_seed(f)).to(dtype)
    x = x.cuda()
    small, best = g.aggregate_workspace_bytes(csr, f), g.aggregate_best_workspace_bytes(csr, x, f, cw)
    size = csr.n * f * x.element_size()
    assert (best > small) == copied and best - small <= 8 / 3 * size + csr.n * 128 + 256
    plain, got = fn(csr, x, f=f, chunk_width=cw, scratch=scratch(max(small, 256))), fn(csr, x, f=f, chunk_width=cw)
    if copied:
        assert torch.equal(plain, fn(csr, x, f=f, chunk_width=cw, scratch=scratch(best - 256)))
    else:
        assert torch.equal(plain, got)
    want, scale = orc.aggregate(model, row_ptr, col, np.ascontiguousarray(x[:, :f].float().cpu().numpy()), f)
    for t in (plain, got):
        assert (np.abs(t.cpu().numpy() - want) <= 1e-5 * scale + 1e-6).all()


@pytest.mark.parametrize("dtype,heads,dim,ld,cw,copied", [
    (torch.float32, 8, 1, 8, 8, False), (torch.float32, 64, 1, 64, 64, False), (torch.bfloat16, 8, 1, 8, 8, False),
    (torch.bfloat16, 8, 2, 16, 16, False), (torch.float32, 1, 3, 3, 3, False), (torch.bfloat16, 1, 4, 4, 4, False),
    (torch.float32, 8, 2, 16, 18, False), (torch.float32, 32, 2, 65, 64, False), (torch.float32, 5, 3, 15, 15, True), (torch.bfloat16, 5, 3, 15, 15, True),
    (torch.bfloat16, 1, 5, 5, 5, True), (torch.bfloat16, 6, 4, 24, 24, True), (torch.float32, 4, 7, 32, 7, True),
    (torch.bfloat16, 4, 7, 28, 14, True), (torch.float32, 4, 7, 28, 10, False), (torch.float32, 6, 4, 24, 24, False)])
def test_which_heads_are_padded(g, long_graph, dtype, heads, dim, ld, cw, copied):
    csr, row_ptr, col = long_graph
    f = heads * dim
    gen = torch.Generator().manual_seed(f)
    z = torch.full((csr.n, ld), float("nan"), dtype=dtype)
    z[:, :f] = torch.randn((csr.n, f), generator=gen).to(dtype)
    a = [torch.randn((heads, dim), generator=gen) * 0.3 for _ in range(2)]
    dev = [t.cuda() for t in (z, *a)]
    small, best = g.gat_workspace_bytes(csr, heads, dim), g.gat_best_workspace_bytes(csr, dev[0], heads, dim, cw)
    assert (best > small) == copied
    plain = g.aggregate_gat(csr, *dev, heads, dim, 0.2, chunk_width=cw, scratch=scratch(small))
    got = g.aggregate_gat(csr, *dev, heads, dim, 0.2, chunk_width=cw)
    if copied:
        assert torch.equal(plain, g.aggregate_gat(csr, *dev, heads, dim, 0.2, chunk_width=cw, scratch=scratch(best - 256)))
    else:
        assert torch.equal(plain, got)
    want, scale = orc.aggregate_gat(row_ptr, col, np.ascontiguousarray(z[:, :f].float().numpy()), a[0].numpy(), a[1].numpy(), heads, dim, 0.2)
    for t in (plain, got):
        assert (np.abs(t.cpu().numpy() - want) <= 1e-5 * scale + 1e-6).all()


def test_calls_do_without_the_copy_where_there_is_no_room(g, long_graph, monkeypatch):
    csr, _, _ = long_graph
    gen = torch.Generator().manual_seed(1)
    x = torch.randn((csr.n, 41), generator=gen).cuda()
    z, a = torch.randn((csr.n, 28), generator=gen).cuda(), [torch.randn((4, 7), generator=gen).cuda() * 0.3 for _ in range(2)]
    feats, w_t = torch.randn((csr.n, 32), generator=gen).cuda(), torch.randn((28, 32), generator=gen).cuda()
    layer = dict(a_src=a[0], a_dst=a[1], heads=4, dim=7, mode="fp32")
    sizes = {"gcn": (g.aggregate_workspace_bytes(csr, 41), g.aggregate_best_workspace_bytes(csr, x)),
             "gat": (g.gat_workspace_bytes(csr, 4, 7), g.gat_best_workspace_bytes(csr, z, 4, 7)),
             "layer": (g.layer_workspace_bytes(csr, "gat", 28, 4, 7), g.layer_best_workspace_bytes(csr, "gat", 28, 4, 7))}
    assert all(best > least for least, best in sizes.values())
    plain = [g.aggregate_gcn(csr, x, scratch=scratch(sizes["gcn"][0])), g.aggregate_gat(csr, z, *a, 4, 7, scratch=scratch(sizes["gat"][0])),
             g.layer(csr, "gat", feats, w_t, scratch=scratch(sizes["layer"][0]), **layer)]
    copied = [g.aggregate_gcn(csr, x), g.aggregate_gat(csr, z, *a, 4, 7), g.layer(csr, "gat", feats, w_t, **layer)]
    alloc, largest = g.binding._alloc_bytes, {least for least, _ in sizes.values()}

    def no_room(nbytes, device, stream=None):
        if nbytes not in largest:
            raise torch.OutOfMemoryError("no room")
        return alloc(nbytes, device, stream)
    monkeypatch.setattr(g.binding, "_alloc_bytes", no_room)
    got = [g.aggregate_gcn(csr, x), g.aggregate_gat(csr, z, *a, 4, 7), g.layer(csr, "gat", feats, w_t, **layer)]
    assert g.tune_chunk_width(csr, x, candidates=[41, 20])[0] in (41, 20)
    for p, c, t in zip(plain, copied, got):
        assert torch.equal(p, t) and not torch.equal(p, c) and torch.allclose(p, c, rtol=1e-3, atol=1e-4)


# Rows of lengths around the octave bounds of the shared classes (a row of up to 256 / 512 / 1024 / 2048 entries is one, two, four or
# eight warps' work when the graph is small), hub rows, and enough short rows beside them.
@pytest.mark.parametrize("dtype", [torch.float32, torch.bfloat16])
@pytest.mark.parametrize("f", [4, 20, 40, 100, 264, 520])
@pytest.mark.parametrize("model", ["gcn", "sage", "gat", "softmax"])
def test_long_rows_of_small_graphs(g, model, f, dtype):
    lengths = [0, 1, 8, 9, 32, 33, 128, 129, 255, 256, 257, 511, 512, 513, 1023, 1024, 1025, 2047, 2048, 2049, 3072, 5000] + [3] * 900
    n = len(lengths)
    rng = np.random.default_rng(f)
    dst = np.repeat(np.arange(n), lengths).astype(np.int32)
    src = rng.integers(0, n, len(dst)).astype(np.int32)
    order = rng.permutation(len(dst))
    src, dst = src[order], dst[order]
    row_ptr, col, _ = orc.build_csr(n, src, dst, 0)
    csr = g.build_csr(n, torch.from_numpy(src).cuda(), torch.from_numpy(dst).cuda())
    x = torch.randn((n, f), generator=torch.Generator().manual_seed(1)).to(dtype)
    xs = np.ascontiguousarray(x.float().numpy())
    if model in ("gcn", "sage"):
        fn = {"gcn": g.aggregate_gcn, "sage": g.aggregate_sage}[model]
        want, scale = orc.aggregate(model, row_ptr, col, xs, f)
        run = lambda: fn(csr, x.cuda())
    elif model == "gat":
        heads, dim = (1, f) if f < 40 else (4, f // 4)
        a = [torch.randn((heads, dim), generator=torch.Generator().manual_seed(k)) * 0.3 for k in (2, 3)]
        want, scale = orc.aggregate_gat(row_ptr, col, xs, a[0].numpy(), a[1].numpy(), heads, dim, 0.2)
        run = lambda: g.aggregate_gat(csr, x.cuda(), a[0].cuda(), a[1].cuda(), heads, dim, 0.2)
    else:
        s = [torch.randn((n, min(f // 4, 12)), generator=torch.Generator().manual_seed(k)) for k in (2, 3)]
        want = scale = orc.edge_softmax(row_ptr, col, s[0].numpy(), s[1].numpy(), 0.2)
        run = lambda: g.edge_softmax(csr, s[0].cuda(), s[1].cuda(), 0.2)
    got = run()
    assert (np.abs(got.cpu().numpy() - want) <= 1e-5 * scale + (1e-7 if model == "softmax" else 1e-6)).all()
    assert torch.equal(got, run())
