"""The C-ABI library builds for sm_100a, loads without a GPU and exports what include/gnnfd.h declares."""
import ctypes
import os
import re

ROOT = os.path.dirname(os.path.dirname(os.path.abspath(__file__)))


def declared_functions():
    text = open(os.path.join(ROOT, "include", "gnnfd.h")).read()
    text = re.sub(r"/\*.*?\*/", "", text, flags=re.S)
    return sorted(set(re.findall(r"\b(gnnfd_[a-z0-9_]+)\s*\(", text)))


def test_library_exports_every_declared_symbol():
    from paper_2104_03058_b200 import build
    path = build.build_library()
    lib = ctypes.CDLL(path)
    names = declared_functions()
    assert len(names) >= 15 and "gnnfd_build_csr" in names and "gnnfd_edge_softmax" in names
    for name in names:
        assert hasattr(lib, name), name


def test_host_only_entry_points_work_without_a_device():
    import paper_2104_03058_b200 as g
    assert g.lib().gnnfd_status_string(0) == b"ok"
    assert b"range" in g.lib().gnnfd_status_string(g.BAD_INDEX)
    pb, sb = g.csr_workspace_bytes(1000, 10_000, g.CSR_ADD_SELF_LOOPS | g.CSR_SYMMETRIZE)
    m = 2 * 10_000 + 1000
    assert pb >= 3 * 4 * m and sb >= 2 * 8 * m          # col_idx, perm, weights; two buffers of 64-bit sort words
    try:
        g.csr_workspace_bytes(10, -1, 0)
    except g.GnnfdError as err:
        assert err.status == g.INVALID_ARG
    else:
        raise AssertionError("negative edge count accepted")
    assert g.launch_count() >= 0


def test_workspaces_never_shrink_as_a_graph_grows():
    """A buffer sized for the largest graph has to hold every smaller one: sizes around the points where the build changes its tiles
    (4,849,664 candidates or rows) or parts keys and values, and between."""
    import paper_2104_03058_b200 as g
    switch = 4 * 148 * 8192
    around = [switch + d for d in (-500_000, -200_000, -2049, -2048, -1, 0, 1, 8192, 200_000, 500_000, 2_000_000, 14_000_000, 15_000_000)]
    edges = sorted([0, 1, 2047, 2048, 2049, 1 << 16, 1 << 20, 1 << 22, 30_000_000, 60_000_000, 115_000_000, 1_000_000_000] + around +
                   [a - 100_000 for a in around] + [a // 2 for a in around])
    for n in (1, 100_000, 1 << 20, (1 << 22) + 3, 1 << 24):
        for flags in (0, 1, 2, 7, 8, 13):
            sizes = [g.csr_workspace_bytes(n, e, flags) for e in edges if (2 if flags & 4 else 1) * e + n < 1 << 31]
            for small, large in zip(sizes, sizes[1:]):
                assert small[0] <= large[0] and small[1] <= large[1]
            if not flags & 8:
                one = [g.oneshot_workspace_bytes(n, e, flags, 32) for e in edges if (2 if flags & 4 else 1) * e + n < 1 << 31]
                assert one == sorted(one)
    rows = sorted([1, 1000, 1 << 17, 1 << 20, 1 << 22, 20_000_000] + around)
    for e in (0, 100_000, 4_000_000, 40_000_000):
        for flags in (0, 1, 8):
            sizes = [g.csr_workspace_bytes(n, e, flags) for n in rows]
            for small, large in zip(sizes, sizes[1:]):
                assert small[0] <= large[0] and small[1] <= large[1]


def test_workspaces_never_shrink_around_the_end_of_the_bucket_sort():
    """The same at the sizes where the build makes buckets or no longer (at 2^25 vertices with 4.85 to 8.4 M candidates, at 2^24 with twice
    as many) or widens its source ranges (behind 2^25)."""
    import paper_2104_03058_b200 as g
    switch = 4 * 148 * 8192
    around = [switch + d for d in (-500_000, -200_000, -2049, -2048, -1, 0, 1, 8192, 200_000, 500_000, 2_000_000, 14_000_000, 15_000_000)]
    edges = sorted([0, 1, 2047, 2048, 2049, 1 << 16, 1 << 20, 1 << 22, 30_000_000, 60_000_000, 115_000_000, 1_000_000_000] + around +
                   [a - 100_000 for a in around] + [a // 2 for a in around])
    for n in ((1 << 25) - 1, 1 << 25, (1 << 25) + 1):
        for flags in (0, 1, 2, 7, 8, 13):
            sizes = [g.csr_workspace_bytes(n, e, flags) for e in edges if (2 if flags & 4 else 1) * e + n < 1 << 31]
            for small, large in zip(sizes, sizes[1:]):
                assert small[0] <= large[0] and small[1] <= large[1]
            if not flags & 8:
                one = [g.oneshot_workspace_bytes(n, e, flags, 32) for e in edges if (2 if flags & 4 else 1) * e + n < 1 << 31]
                assert one == sorted(one)
    rows = sorted([1, 1000, 1 << 17, 1 << 20, 1 << 22, 20_000_000, 1 << 30] + around +
                  [(1 << bits) + d for bits in range(21, 28) for d in (-1, 0, 1)])
    for e in (0, 100_000, 4_000_000, 4_900_000, 5_500_000, 6_500_000, 8_380_000, 8_400_000, 12_000_000, 16_800_000, 40_000_000):
        for flags in (0, 1, 2, 4, 8):
            sizes = [g.csr_workspace_bytes(n, e, flags) for n in rows]
            for small, large in zip(sizes, sizes[1:]):
                assert small[0] <= large[0] and small[1] <= large[1]
            one = [g.oneshot_workspace_bytes(n, e, flags, 8) for n in rows if not flags & 8]
            assert one == sorted(one)


def test_header_constants_match_binding():
    import paper_2104_03058_b200 as g
    text = open(os.path.join(ROOT, "include", "gnnfd.h")).read()
    assert int(re.search(r"#define GNNFD_HUB_DEGREE (\d+)", text).group(1)) == g.HUB_DEGREE
    assert int(re.search(r"#define GNNFD_HUB_SEGMENT (\d+)", text).group(1)) == g.HUB_SEGMENT
    for name, val in (("ADD_SELF_LOOPS", 1), ("DEDUP", 2), ("SYMMETRIZE", 4)):
        assert int(re.search(r"GNNFD_CSR_%s = (\d+)" % name, text).group(1)) == val == getattr(g, "CSR_" + name)


def test_default_chunk_candidates_are_host_only():
    import torch

    import paper_2104_03058_b200 as g
    assert g.default_chunk_candidates(602) == [602, 256, 128, 64, 32, 16, 8]
    assert g.default_chunk_candidates(64) == [64, 32, 16, 8]
    assert g.default_chunk_candidates(8, torch.bfloat16) == [8]
    assert g.default_chunk_candidates(256, torch.bfloat16) == [256, 128, 64, 32, 16]
