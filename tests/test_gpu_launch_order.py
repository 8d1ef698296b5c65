"""Launches that start before the one ahead of them has ended: calls lined up on one stream, without a wait between them, give the bits of calls
that run alone, also where every buffer is written again and again, and are no slower."""
import pytest

import graphgen as gg

torch = pytest.importorskip("torch")
pytestmark = pytest.mark.gpu


def graph(n, e, seed):
    return (torch.from_numpy(a).cuda() for a in gg.powerlaw_graph(n, e, 2.1, None, seed))


@pytest.mark.parametrize("n,e", [(300, 3000), (5000, 120_000)])
def test_lined_up_calls_on_the_same_buffers(n, e):
    import paper_2104_03058_b200 as g
    csr = g.build_csr(n, *graph(n, e, 3), g.CSR_ADD_SELF_LOOPS)
    gen = torch.Generator(device="cuda").manual_seed(1)
    inputs = [torch.randn((n, 41), generator=gen, device="cuda") for _ in range(12)]
    w_t, att = torch.randn((56, 44), generator=gen, device="cuda"), torch.randn((8, 7), generator=gen, device="cuda")
    x, padded = torch.empty((n, 41), device="cuda"), torch.zeros((n, 44), device="cuda")
    need = max(g.aggregate_best_workspace_bytes(csr, x, 41, 41), g.gat_workspace_bytes(csr, 8, 7), g.layer_workspace_bytes(csr, "gat", 56, 8, 7), 1 << 20)
    scratch = torch.empty(2 * need, dtype=torch.uint8, device="cuda")
    att4 = att[:, :4].contiguous()

    def calls(values, wait):
        x.copy_(values)
        padded[:, :41].copy_(values)
        out = []
        for call in (lambda: g.aggregate_gcn(csr, x, scratch=scratch), lambda: g.aggregate_sage(csr, x, chunk_width=16, scratch=scratch),
                     lambda: g.layer(csr, "gat", padded, w_t, a_src=att, a_dst=att, heads=8, dim=7, scratch=scratch),
                     lambda: g.edge_softmax(csr, *g.gat_scores(padded, att4, att4, 8, 4), 0.2),
                     lambda: g.layer(csr, "gcn", padded, w_t, scratch=scratch)):
            out.append(call())
            if wait:
                torch.cuda.synchronize()
        return out

    alone = [calls(values, True) for values in inputs]
    for _ in range(5):
        torch.cuda.synchronize()
        lined_up = [calls(values, False) for values in inputs]
        for a, b in zip(alone, lined_up):
            assert all(torch.equal(p, q) for p, q in zip(a, b))


def test_lined_up_builds_and_aggregations_on_the_same_buffers():
    import paper_2104_03058_b200 as g
    n, e = 3000, 50_000
    graphs = [tuple(graph(n, e, seed)) for seed in range(6)]
    least = min(len(src) for src, _ in graphs)
    graphs = [(src[:least].contiguous(), dst[:least].contiguous()) for src, dst in graphs]
    x = torch.randn((n, 24), device="cuda")
    scratch = torch.empty(g.oneshot_workspace_bytes(n, least, 1, 24), dtype=torch.uint8, device="cuda")
    pb, sb = g.csr_workspace_bytes(n, least, 1)
    persistent, build = (torch.empty(b, dtype=torch.uint8, device="cuda") for b in (pb, sb))

    def calls(src, dst):
        csr = g.build_csr(n, src, dst, 1, persistent=persistent, scratch=build)
        return [g.aggregate_gcn(csr, x), csr.col_idx.clone(), g.oneshot("gcn", n, src, dst, x, flags=1, scratch=scratch)]

    alone = []
    for src, dst in graphs:
        alone.append(calls(src, dst))
        torch.cuda.synchronize()
    for _ in range(10):
        for (src, dst), want in zip(graphs, alone):
            assert all(torch.equal(p, q) for p, q in zip(calls(src, dst), want))


@pytest.mark.parametrize("heads,dim", [(4, 32), (1, 64)])
def test_lined_up_calls_are_no_slower(heads, dim):
    """Small graphs whose longest rows decide: with several launches lined up, a few SMs got most of them (a fifth slower)."""
    import paper_2104_03058_b200 as g
    n = 5000
    csr = g.build_csr(n, *graph(n, 500_000, 1), g.CSR_ADD_SELF_LOOPS)
    z, att = torch.randn((n, heads * dim), device="cuda"), torch.randn((heads, dim), device="cuda") * 0.1
    out, one = torch.empty_like(z), torch.zeros(1, device="cuda")

    def us(between):
        begin, end, least = torch.cuda.Event(enable_timing=True), torch.cuda.Event(enable_timing=True), float("inf")
        for _ in range(6):
            begin.record()
            for _ in range(100):
                g.aggregate_gat(csr, z, att, att, heads, dim, 0.2, out=out)
                if between:
                    one.add_(1)                          # a kernel that lets nobody start early
            end.record()
            end.synchronize()
            least = min(least, begin.elapsed_time(end) * 10)
        return least

    us(False)
    assert us(False) < 1.04 * us(True)


@pytest.mark.parametrize("f", [72, 96])
def test_long_rows_of_sage_are_split_as_finely_as_its_blocks_need(f):
    """GraphSAGE keeps four blocks on an SM where GCN keeps three: with rows split as for three it took a seventh longer than GCN, which
    reads a weight per entry as well, on graphs whose longest rows decide."""
    import paper_2104_03058_b200 as g
    n = 20_000
    csr = g.build_csr(n, *graph(n, 1_000_000, 1), g.CSR_ADD_SELF_LOOPS)
    x, out = torch.randn((n, f), device="cuda"), torch.empty((n, f), device="cuda")

    def us(call):
        begin, end, least = torch.cuda.Event(enable_timing=True), torch.cuda.Event(enable_timing=True), float("inf")
        for _ in range(6):
            begin.record()
            for _ in range(100):
                call(csr, x, out=out)
            end.record()
            end.synchronize()
            least = min(least, begin.elapsed_time(end) * 10)
        return least

    assert us(g.aggregate_sage) < 1.05 * us(g.aggregate_gcn)


def test_gcn_just_above_the_size_that_splits_rows():
    """Between the sizes at which rows are split for three and for four blocks on an SM, GCN keeps three: with four, a quarter more entries
    took half as long again, for the longest rows' sake."""
    import paper_2104_03058_b200 as g
    n, f, times = 100_000, 96, []
    for e in (3_300_000, 4_200_000):
        csr = g.build_csr(n, *graph(n, e, 1), g.CSR_ADD_SELF_LOOPS)
        x, out = torch.randn((n, f), device="cuda"), torch.empty((n, f), device="cuda")
        begin, end, least = torch.cuda.Event(enable_timing=True), torch.cuda.Event(enable_timing=True), float("inf")
        for _ in range(6):
            begin.record()
            for _ in range(50):
                g.aggregate_gcn(csr, x, out=out)
            end.record()
            end.synchronize()
            least = min(least, begin.elapsed_time(end) * 20)
        times.append((least, csr.nnz))
    (small, few), (large, many) = times
    assert few < 3_640_000 < many < 4_700_000
    assert large / small < 1.15 * many / few, times
