"""GPU parity at the sizes where tiles, groups and index words end.

Bit-exact against the oracle, or against values put together from the
oracle's Philox and threshold functions where a whole graph is too large for
it. Inputs are seeded.
"""
import numpy as np
import pytest
import torch

import oracle as o
import paper_1003_3684_gb300 as pg
from paper_1003_3684_gb300 import workloads as W

pytestmark = pytest.mark.gpu

ZERO_ENDS = [[0.0, 0.6], [0.4, 0.0]]


@pytest.fixture(scope="module", autouse=True)
def _built():
    from paper_1003_3684_gb300 import build
    build.build()
    yield
    torch.cuda.synchronize()


def host(t):
    a = t.cpu().numpy()
    return a.view(np.uint64 if a.dtype == np.int64 else np.uint32).astype(np.uint64)


def kron_edge(P, k, seed, e):
    """Edge e of the stochastic Kronecker graph, level by level."""
    n0 = len(P)
    T = o.kron_thresholds(P)
    key = (seed & 0xFFFFFFFF, seed >> 32)
    row = col = 0
    for level in range(k):
        w = o.philox4x32_10((e & 0xFFFFFFFF, e >> 32, level // 4, 3), key)[level % 4]
        cell = o.kron_pick(T, int(w))
        row, col = row * n0 + cell // n0, col * n0 + cell % n0
    return row, col


@pytest.mark.parametrize("P", [W.KRON_INITIATOR, ZERO_ENDS])
@pytest.mark.parametrize("k,id64", [(1, False), (7, False), (20, False), (30, True), (32, False),
                                    (33, True), (34, True), (64, True)])
@pytest.mark.parametrize("begin", [2**32 - 5, 2**32 - 4, 2**33 - 1])
def test_kronecker_range_across_an_index_word(P, k, id64, begin):
    n, seed = 11, 2**40 + 9
    if k == 64 and P is W.KRON_INITIATOR and begin == 2**33 - 1:
        n = 12
    got = host(pg.gen_kronecker_range(P, k, 2**34, begin, begin + n, seed=seed, id64=id64))
    want = np.array([kron_edge(P, k, seed, begin + i) for i in range(n)], dtype=np.uint64)
    assert np.array_equal(got, want)


@pytest.mark.parametrize("id64", [False, True])
def test_batch_kronecker_tiles_at_odd_arena_edges(id64):
    """Jobs of every edge count around a tile's and a pair's end, so that jobs
    and tiles start at odd arena edges; more levels than 32 with 64-bit ids."""
    jobs = []
    for i, E in enumerate([1, 2, 3, 63, 64, 65, 127, 129, 191, 1, 1, 257]):
        k = (35 if i % 3 == 0 else 33) if id64 and i % 2 else 1 + 2 * i
        jobs.append(dict(kind="kron", initiator=ZERO_ENDS if i % 4 == 1 else W.KRON_INITIATOR,
                         k=k, n_edges=E, seed=100 + i))
    plan = pg.BatchPlan(jobs, tile_edges=64, id64=id64)
    arena = pg.gen_batch(plan)
    torch.cuda.synchronize()
    for i, j in enumerate(jobs):
        assert np.array_equal(host(plan.edges_of(arena, i)),
                              o.kron(j["initiator"], j["k"], j["n_edges"], j["seed"])), i


@pytest.mark.parametrize("id64", [False, True])
def test_batch_csr_of_jobs_around_a_union_run(id64):
    """CSR jobs of 0, 1 and about 128 edges (a warp's run of union slots),
    between jobs without CSR."""
    jobs = []
    for i, E in enumerate([0, 1, 127, 128, 129, 0, 0, 300, 5, 2, 128]):
        jobs.append(dict(kind="kron", initiator=W.KRON_INITIATOR, k=3 + i % 5, n_edges=E,
                         seed=i, want_csr=True))
        jobs.append(dict(kind="kron", initiator=W.KRON_INITIATOR, k=6, n_edges=777, seed=i + 50))
        jobs.append(dict(kind="pba", n=E // 3, m=3, n0=4, seed=i, want_csr=i % 2 == 0))
    plan = pg.BatchPlan(jobs, tile_edges=64, id64=id64)
    arena = pg.gen_batch(plan)
    rp, col = pg.gen_batch_csr(plan, arena, check=True)
    torch.cuda.synchronize()
    for i, j in enumerate(jobs):
        if not j.get("want_csr"):
            continue
        edges = (o.kron(j["initiator"], j["k"], j["n_edges"], j["seed"]) if j["kind"] == "kron"
                 else o.ba(j["n"], 3, 4, j["seed"]))
        ref_rp, ref_col = o.csr(np.asarray(edges).astype(np.uint64), pg._job_vertices(j))
        got_rp, got_col = plan.csr_of(rp, col, i)
        assert np.array_equal(host(got_rp), ref_rp), i
        assert np.array_equal(host(got_col), ref_col), i


@pytest.mark.parametrize("B,n_b,m,Wf,f,n0,id64", [
    (2, 512, 1, 1, 0.2, 2, False),         # one segment of 512 entries, exactly
    (3, 513, 1, 1, 0.2, 3, False),         # a second segment of one entry
    (7, 2049, 1, 1, 0.1, 2, True),         # one entry past the prefix
    (5, 8192, 1, 5, 0.0, 2, False),        # every block in one faction, one level
    (130, 1700, 5, 2, 0.1, 6, False),      # segments longer than 512 (2 B entries)
    (300, 400, 5, 1, 0.3, 6, False),       # 2000 entries per block, uneven segments
    (31, 9001, 3, 1, 0.1, 4, False),       # 31 targets: fewer than a warp's lanes
    (33, 9001, 3, 1, 0.1, 4, True),        # two CTAs of targets in the scan
    (256, 2**14, 5, 1, 0.1, 6, False),     # short segments under a large pass
    (320, 20_011, 5, 1, 0.1, 6, False),    # one level past the long prefix
])
def test_pba_segments(B, n_b, m, Wf, f, n0, id64):
    n = B * n_b
    got = pg.gen_pba(n, m, B, n0, Wf, f, 77, id64=id64)
    ref = o.pba(n, m, B, n0, Wf, f, 77)[0]
    assert np.array_equal(host(got), np.asarray(ref).astype(np.uint64))


@pytest.mark.parametrize("b_begin,b_end", [(0, 7), (3, 4), (6, 7), (2, 5)])
def test_pba_block_ranges_with_segments_that_do_not_fill_a_cta(b_begin, b_end):
    B, n_b, m, n0, seed = 7, 1111, 3, 4, 5
    ref = np.asarray(o.pba(B * n_b, m, B, n0, 1, 0.1, seed)[0]).astype(np.uint64)
    ws = pg.pg_pba_prepare(B * n_b, m, B, n0, seed=seed)
    part = pg.gen_pba_blocks(ws, B * n_b, m, B, b_begin, b_end, n0=n0, seed=seed)
    per = ref.shape[0] // B
    assert np.array_equal(host(part), ref[b_begin * per:b_end * per])


def test_noalloc_takes_a_graph_whose_smallest_workspace_fits():
    """The workspace of short segments exceeds the fixed scratch; that of
    whole granules does not."""
    import ctypes as C
    L = pg.lib()
    L.gen_pba_noalloc.argtypes = [C.c_uint64, C.c_uint32, C.c_uint32, C.c_uint32, C.c_uint32,
                                  C.c_double, C.c_uint64, C.c_int, C.c_void_p, C.c_uint64,
                                  C.POINTER(C.c_uint64), C.c_void_p]
    L.pg_pba_noalloc_scratch_bytes.restype = C.c_size_t
    B, n_b, m = 16, 193_750, 5
    n = B * n_b
    assert pg.pg_pba_workspace_size(n, m, B) > L.pg_pba_noalloc_scratch_bytes()
    E = pg.pg_pba_edge_count(n, m, B, 6)
    out = torch.full((E, 2), -1, dtype=torch.int32, device="cuda")
    cnt = C.c_uint64(0)
    st = L.gen_pba_noalloc(n, m, B, 6, 1, 0.1, 3, 0, C.c_void_p(out.data_ptr()), E, C.byref(cnt),
                           C.c_void_p(torch.cuda.current_stream().cuda_stream))
    assert st == pg.PG_OK and cnt.value == E
    assert torch.equal(out, pg.gen_pba(n, m, B, 6, 1, 0.1, 3))


@pytest.mark.parametrize("N", [2**32, 2**32 + 1])
@pytest.mark.parametrize("flags", [0, pg.CSR_SYMMETRIZE | pg.CSR_DEDUP])
def test_csr_of_64_bit_ids_on_both_sides_of_the_narrow_sort(N, flags):
    """64-bit ids below 2^32 are sorted as pairs of 32-bit ids, larger ones as
    they are. The row pointers (34 GB) are checked on the device, at the rows
    that have edges and right after them."""
    rng = np.random.default_rng(5 + flags)
    e = rng.integers(0, N, size=(20_011, 2), dtype=np.uint64)
    e[:300] = e[300:600]                  # repeated pairs
    e[1000:1200, 0] = N - 1
    e[1200:1400, 1] = N - 1
    t = torch.from_numpy(e.view(np.int64)).cuda()
    rp, col = pg.edges_to_csr_opts(t, N, flags) if flags else pg.edges_to_csr(t, N, check=True)
    if flags:
        e = np.unique(np.concatenate([e, e[:, ::-1]]), axis=0)
    e = e[np.lexsort((e[:, 1], e[:, 0]))]
    rows, first, counts = np.unique(e[:, 0], return_index=True, return_counts=True)
    at = torch.from_numpy(rows.view(np.int64)).cuda()
    assert np.array_equal(host(rp[at]), first.astype(np.uint64))
    assert np.array_equal(host(rp[at + 1]), (first + counts).astype(np.uint64))
    assert int(rp[0]) == 0 and int(rp[-1]) == e.shape[0]
    assert np.array_equal(host(col)[:e.shape[0]], e[:, 1])


@pytest.mark.parametrize("flags", [pg.CSR_ODD, pg.CSR_ODD | pg.CSR_NO_LOOPS, pg.CSR_DEDUP,
                                   pg.CSR_SYMMETRIZE | pg.CSR_ODD, pg.CSR_NO_LOOPS])
@pytest.mark.parametrize("run", [1, 2, 3, 31, 32, 33, 64, 511, 513, 4095, 4097])
def test_csr_options_with_runs_around_words_and_tiles(flags, run):
    """Runs of equal pairs of odd and even lengths that start at every offset
    of a 32-position word, cross words, a warp's positions and tiles."""
    lens = [run, 1, run + 1, 2, run, 3, run + 2, 5, 1, run] + [1 + i % 7 for i in range(400)]
    n = len(lens)
    src = np.arange(n) // 9
    dst = np.where(np.arange(n) % 9 == 4, src, 1000 + np.arange(n) % 9)     # some self-loops
    e = np.repeat(np.stack([src, dst], 1), lens, axis=0).astype(np.uint32)
    e = e[np.random.default_rng(run).permutation(e.shape[0])]
    N = 1100
    rp, col = pg.edges_to_csr_opts(torch.from_numpy(e.view(np.int32)).cuda(), N, flags)
    ref_rp, ref_col = o.csr_opts(e.astype(np.uint64), N, flags)
    assert np.array_equal(host(rp), ref_rp)
    assert np.array_equal(host(col)[:ref_col.shape[0]], ref_col)


@pytest.mark.parametrize("N", [1, 31, 4094, 4095, 4096, 8 * 4096 - 1, 8 * 4096, 8 * 4096 + 1,
                               9 * 4096 + 17])
@pytest.mark.parametrize("off", [0, 1])
def test_csr_rows_without_edges(N, off):
    """Row pointers over long gaps, into row_ptr buffers that are and are not
    aligned to 16 bytes, at the sizes where one CTA stops scanning them."""
    rng = np.random.default_rng(N)
    e = rng.integers(0, N, size=(7, 2), dtype=np.uint32)
    buf = torch.full((N + 3,), -7, dtype=torch.int64, device="cuda")
    rp, col = pg.edges_to_csr(torch.from_numpy(e.view(np.int32)).cuda(), N, row_ptr=buf[off:])
    ref_rp, ref_col = o.csr(e.astype(np.uint64), N)
    assert np.array_equal(host(buf[off:off + N + 1]), ref_rp)
    assert np.array_equal(host(col), ref_col)
    assert (buf[off + N + 1:] == -7).all() and (off == 0 or int(buf[0]) == -7)


@pytest.mark.parametrize("N", [1, 2, 31, 32, 33, 255, 256, 257, 2500, 70_001])
@pytest.mark.parametrize("id64", [False, True])
def test_bfs_around_words_and_switches(N, id64):
    """Random graphs whose searches switch direction both ways, at vertex
    counts around a bitmap word and a warp's words; a hub with more slices of
    a narrow and of a wide level than one row may have; unreached vertices."""
    rng = np.random.default_rng(N)
    e = rng.integers(0, max(N - N // 7, 1), size=(3 * N, 2), dtype=np.uint64)
    chain = np.arange(N - N // 7, N - 1, dtype=np.uint64)      # a long tail of narrow levels
    e = np.concatenate([e, np.stack([chain[::2], chain[::2] + 1], 1)]) if N > 60 else e
    hub = np.stack([np.full(N // 3, N // 2), rng.integers(0, N, N // 3)], 1).astype(np.uint64)
    e = np.concatenate([e, hub])
    for flags in (0, o.CSR_SYMMETRIZE):
        rp_h, col_h = o.csr_opts(e, N, flags)
        rp = torch.from_numpy(rp_h.view(np.int64)).cuda()
        col = torch.from_numpy(col_h.astype(np.uint64 if id64 else np.uint32)
                               .view(np.int64 if id64 else np.int32)).cuda()
        for s in {0, N // 2, N - 1}:
            ref = o.bfs(rp_h, col_h, s)
            for undirected in ([False, True] if flags else [False]):
                dist, levels, scanned = pg.bfs(rp, col, s, undirected=undirected)
                assert np.array_equal(dist.cpu().numpy().view(np.uint32), ref[0]), (s, flags)
                assert (levels, scanned) == ref[1:], (s, flags, undirected)


@pytest.mark.parametrize("which", [pg.DEG_OUT, pg.DEG_IN, pg.DEG_TOTAL])
@pytest.mark.parametrize("M", [1, 31, 32, 33, 1000])
def test_degrees_of_grouped_sources(which, M):
    """Runs of one source inside a warp, across warps and at the list's end;
    sources past the vertex count."""
    rng = np.random.default_rng(M)
    src = np.repeat(np.arange(M), 1 + np.arange(M) % 40)[:M]
    e = np.stack([src, rng.integers(0, 12, M)], 1).astype(np.uint32)
    N = max(int(src.max()), 1)                                  # the last source is outside
    deg = pg.degrees(torch.from_numpy(e.view(np.int32)).cuda(), N, which)
    assert np.array_equal(host(deg), o.degrees(e.astype(np.uint64), N, which))


@pytest.mark.parametrize("n_b", [2, 3, 5, 127, 1023, 1025, 3000, 65_537])
@pytest.mark.parametrize("m,n0", [(1, 2), (5, 6), (3, 23), (3, 24)])
def test_pba_links_for_any_block_size(n_b, m, n0):
    """Block sizes that are no power of two, seed cliques that just fit the
    links' table (n0 = 23) and that do not."""
    B = 4
    got = pg.gen_pba(B * n_b, m, B, n0, 1, 0.2, 31)
    ref = o.pba(B * n_b, m, B, n0, 1, 0.2, 31)[0]
    assert np.array_equal(host(got), np.asarray(ref).astype(np.uint64))


@pytest.mark.parametrize("row", [1, 2, 5, 31, 32, 33])
@pytest.mark.parametrize("M", [1, 33, 2047, 2048, 2049, 4127, 4128, 4129, 70_000])
@pytest.mark.parametrize("id64", [False, True])
def test_csr_grouped_rows_across_tiles(row, M, id64):
    """Rows of one length cross every tile boundary at every offset; then one
    edge at a tile's first or last position breaks the order (or, rows of 32,
    makes a row too long), so that a list partly placed is sorted after all."""
    rng = np.random.default_rng(M * row)
    src = (np.arange(M) + rng.integers(0, row)) // row
    N = 3 * int(src.max()) + 4
    e = np.stack([3 * src + 1, rng.integers(0, min(N, 50), M)], 1).astype(np.int64)

    def check(e):
        t = torch.from_numpy(e if id64 else e.astype(np.uint32).view(np.int32)).cuda()
        rp, col = pg.edges_to_csr(t, N, check=True)
        ref_rp, ref_col = o.csr(e.astype(np.uint64), N)
        np.testing.assert_array_equal(host(rp), ref_rp)
        np.testing.assert_array_equal(host(col), ref_col)

    check(e)
    for at in {1, min(2048, M - 1), M - 1} & set(range(1, M)):
        bad = e.copy()
        if row == 32:
            bad[max(at - 32, 0):at + 1, 0] = bad[at, 0]
        else:
            bad[at, 0] = 0
        check(bad)


@pytest.mark.parametrize("M", [786_433, 96 * 8192 - 1, 97 * 8192, 97 * 8192 + 1, 2_600_003])
@pytest.mark.parametrize("N", [2**14, 2**15, 2**16])
@pytest.mark.parametrize("spread", [0, 1, 3, 16])
@pytest.mark.parametrize("id64", [False, True])
def test_csr_sort_of_long_lists(M, N, spread, id64):
    """Digits of 7 and 8 bits, full and ragged last tiles, more tiles than the
    GPU holds CTAs; ids of `spread` random bits, so that whole warps share a
    digit or few lanes do."""
    rng = np.random.default_rng(M + spread)
    e = rng.integers(0, min(N, 1 << spread), (M, 2), dtype=np.int64) * (N >> min(spread, 14)) % N
    t = torch.from_numpy(e if id64 else e.astype(np.uint32).view(np.int32)).cuda()
    rp, col = pg.edges_to_csr(t, N, check=True)
    ref_rp, ref_col = o.csr(e.astype(np.uint64), N)
    np.testing.assert_array_equal(host(rp), ref_rp)
    np.testing.assert_array_equal(host(col), ref_col)


@pytest.mark.parametrize("M", [2, 4095, 4096, 4097, 9 * 4096 + 1, 786_431, 786_432])
@pytest.mark.parametrize("N", [2, 2**9, 2**13 + 1, 2**20])
@pytest.mark.parametrize("flags,id64", [(0, False), (0, True), (pg.CSR_SYMMETRIZE, False),
                                        (pg.CSR_ODD, True)])
def test_csr_sort_of_short_lists(M, N, flags, id64):
    """Digits of up to 9 bits, full and ragged tiles, both sides of the longest
    short list (a symmetrised list has twice the pairs); few pairs take most
    of the edges, so that every option has something to drop."""
    rng = np.random.default_rng(M * 7 + flags)
    e = rng.integers(0, N, (M, 2), dtype=np.int64)
    e[::3] = e[0]
    t = torch.from_numpy(e if id64 else e.astype(np.uint32).view(np.int32)).cuda()
    rp, col = pg.edges_to_csr_opts(t, N, flags) if flags else pg.edges_to_csr(t, N, check=True)
    ref_rp, ref_col = (o.csr_opts(e.astype(np.uint64), N, flags) if flags else
                       o.csr(e.astype(np.uint64), N))
    np.testing.assert_array_equal(host(rp), ref_rp)
    np.testing.assert_array_equal(host(col)[:int(ref_rp[-1])], ref_col)


@pytest.mark.parametrize("N", [608 * 4096 - 2, 608 * 4096 - 1, 608 * 4096, 2 * 608 * 4096 + 5])
@pytest.mark.parametrize("flags", [0, pg.CSR_DEDUP])
def test_csr_rows_of_more_tiles_than_ctas(N, flags):
    """Where a CTA of the row kernel goes from one tile to several."""
    rng = np.random.default_rng(N)
    e = rng.integers(0, N, size=(999, 2), dtype=np.uint32)
    t = torch.from_numpy(e.view(np.int32)).cuda()
    rp, col = pg.edges_to_csr_opts(t, N, flags) if flags else pg.edges_to_csr(t, N, check=True)
    ref_rp, ref_col = (o.csr_opts(e.astype(np.uint64), N, flags) if flags else
                       o.csr(e.astype(np.uint64), N))
    np.testing.assert_array_equal(host(rp), ref_rp)
    np.testing.assert_array_equal(host(col)[:int(ref_rp[-1])], ref_col)


@pytest.mark.parametrize("N", [13 * 2**20 - 1, 13 * 2**20, 13 * 2**20 + 1, 2**24 + 384])
@pytest.mark.parametrize("id64", [False, True])
def test_degrees_counted_in_32_bits_and_widened(N, id64):
    """Both sides of the size where counts move to 32 bits in the result's own
    memory: every vertex's count, the first and last ones with long runs."""
    rng = np.random.default_rng(N)
    e = rng.integers(0, N, size=(2_000_003, 2), dtype=np.int64)
    e[::5] = (N - 1, 0)
    e[1::5, 1] = rng.integers(0, 64, e[1::5].shape[0])
    t = torch.from_numpy(e if id64 else e.astype(np.uint32).view(np.int32)).cuda()
    deg = torch.full((N + 2,), -7, dtype=torch.int64, device="cuda")
    pg.degrees(t, N, pg.DEG_TOTAL, out=deg[1:N + 1])
    np.testing.assert_array_equal(host(deg[1:N + 1]), o.degrees(e.astype(np.uint64), N, o.DEG_TOTAL))
    assert int(deg[0]) == -7 and int(deg[N + 1]) == -7


@pytest.mark.parametrize("N", [1, 2, 30, 31, 32, 60, 1000, 4097])
@pytest.mark.parametrize("shape", ["path", "star", "two_stars", "complete"])
def test_bfs_of_graphs_that_change_direction(N, shape):
    """Searches that start bottom-up, end in either direction, or go back to
    top-down: a path's frontier is always one vertex, a star's whole graph."""
    v = np.arange(N, dtype=np.int64)
    if shape == "path":
        e = np.stack([v[:-1], v[1:]], 1)
    elif shape == "star":
        e = np.stack([np.zeros(N, np.int64), v], 1)
    elif shape == "two_stars":   # joined by a path of a quarter of the vertices
        q = N // 4
        a, b = v[:q + 1], v[2 * q:]
        e = np.concatenate([np.stack([np.zeros_like(a), a], 1), np.stack([v[q:2 * q], v[q + 1:2 * q + 1]], 1),
                            np.stack([np.full_like(b, 2 * q), b], 1)])
    else:
        k = v[:40]
        e = np.stack(np.meshgrid(k, k), -1).reshape(-1, 2)
    rp_h, col_h = o.csr_opts(e.astype(np.uint64), N, pg.CSR_SYMMETRIZE)
    rp = torch.from_numpy(rp_h.astype(np.int64)).cuda()
    col = torch.from_numpy(np.append(col_h, 0).astype(np.uint32).view(np.int32)).cuda()
    for source in {0, N // 3, N - 1}:
        ref = o.bfs(rp_h, col_h, source)
        for undirected in (False, True):
            dist, levels, scanned = pg.bfs(rp, col, source, undirected=undirected)
            assert np.array_equal(dist.cpu().numpy().view(np.uint32), ref[0]), (source, undirected)
            assert (levels, scanned) == tuple(ref[1:3]), (source, undirected)


@pytest.mark.parametrize("M", [20_011, 900_001])                 # a short sort and a long one
@pytest.mark.parametrize("N", [5000, 2**13])
@pytest.mark.parametrize("flags", [0, pg.CSR_DEDUP, pg.CSR_ODD, pg.CSR_NO_LOOPS])
def test_csr_drops_sources_whose_low_word_names_a_vertex(M, N, flags):
    """64-bit sources above 2^32, whose low 32 bits are a vertex, some of them
    in a copy of a valid pair: no row may hold them, and no option may take
    them for that pair."""
    rng = np.random.default_rng(M + N + flags)
    e = rng.integers(0, N - 1, (M, 2), dtype=np.int64)           # (N - 1, N - 1) does not occur
    e[2::9] = e[1::9][:e[2::9].shape[0]]
    e[2::9, 0] += 2**32
    e[3::9, 0] += rng.integers(1, 2**31, e[3::9].shape[0]) << 32
    t = torch.from_numpy(e).cuda()
    rp, col = pg.edges_to_csr_opts(t, N, flags) if flags else pg.edges_to_csr(t, N, check=True)
    kept = e[e[:, 0] < N].astype(np.uint64)
    ref_rp, ref_col = o.csr_opts(kept, N, flags) if flags else o.csr(kept, N)
    np.testing.assert_array_equal(host(rp), ref_rp)
    np.testing.assert_array_equal(host(col)[:ref_col.shape[0]], ref_col)


@pytest.mark.parametrize("M", [3, 2049, 70_000, 800_000])
@pytest.mark.parametrize("more", [-2, -1, 0, 1])
@pytest.mark.parametrize("id64", [False, True])
def test_csr_of_more_rows_than_edges_after_a_grouped_start(M, more, id64):
    """The list is grouped but for its last edge, so most row ends are written
    and must go again: on both sides of the vertex count from which the
    list's rows alone are cleared, and well above it."""
    N = 12 * M + more if more < 1 else 50 * M
    src = np.sort(np.random.default_rng(M).integers(0, N, M))
    src[-1] = 0
    e = np.stack([src, np.arange(M)[::-1] % N], 1).astype(np.int64)
    t = torch.from_numpy(e if id64 else e.astype(np.uint32).view(np.int32)).cuda()
    rp, col = pg.edges_to_csr(t, N, check=True)
    ref_rp, ref_col = o.csr(e.astype(np.uint64), N)
    np.testing.assert_array_equal(host(rp), ref_rp)
    np.testing.assert_array_equal(host(col), ref_col)


def _median_ms(call):
    call()
    times = []
    for _ in range(7):
        a, b = torch.cuda.Event(enable_timing=True), torch.cuda.Event(enable_timing=True)
        a.record()
        call()
        b.record()
        b.synchronize()
        times.append(a.elapsed_time(b))
    return sorted(times)[3]


def test_csr_of_few_edges_on_many_vertices_takes_no_longer_than_with_options():
    """Both calls clear and scan the same rows, and sort a list that is nothing
    beside them; with options there is no grouped pass to undo."""
    M, N = 1000, 2**26
    t = torch.randint(0, N, (M, 2), dtype=torch.int32, device="cuda")
    rp = torch.empty(N + 1, dtype=torch.int64, device="cuda")
    plain = _median_ms(lambda: pg.edges_to_csr(t, N, row_ptr=rp))
    dedup = _median_ms(lambda: pg.edges_to_csr_opts(t, N, pg.CSR_DEDUP, row_ptr=rp))
    assert plain < 2 * dedup, (plain, dedup)


@pytest.mark.parametrize("N", [13 * 2**20 - 1, 13 * 2**20 + 1, 2**24])
@pytest.mark.parametrize("more", [-1, 0, 1])
def test_degrees_of_three_edges_per_four_vertices(N, more):
    """Both sides of the edge count from which many vertices' counts are taken
    in 32 bits; the first and last vertices with long runs."""
    M = N - N // 4 + more
    rng = np.random.default_rng(M)
    e = rng.integers(0, N, size=(M, 2), dtype=np.int64)
    e[::5] = (N - 1, 0)
    e[1::5, 1] = rng.integers(0, 64, e[1::5].shape[0])
    deg = torch.full((N + 2,), -7, dtype=torch.int64, device="cuda")
    pg.degrees(torch.from_numpy(e.astype(np.uint32).view(np.int32)).cuda(), N, pg.DEG_TOTAL,
               out=deg[1:N + 1])
    np.testing.assert_array_equal(host(deg[1:N + 1]), o.degrees(e.astype(np.uint64), N, o.DEG_TOTAL))
    assert int(deg[0]) == -7 and int(deg[N + 1]) == -7


def test_degrees_of_few_edges_on_many_vertices_take_as_long_for_both_ends_as_for_one():
    """Either call is the clearing of the counts and little else."""
    N = 2**24
    t = torch.randint(0, N, (1000, 2), dtype=torch.int32, device="cuda")
    deg = torch.empty(N, dtype=torch.int64, device="cuda")
    both = _median_ms(lambda: pg.degrees(t, N, pg.DEG_TOTAL, out=deg))
    one = _median_ms(lambda: pg.degrees(t, N, pg.DEG_OUT, out=deg))
    assert both < 2 * one, (both, one)


def _csr_on_gpu(e, N, id64=False):
    rp_h, col_h = o.csr_opts(e.astype(np.uint64), N, pg.CSR_SYMMETRIZE)
    col = col_h.astype(np.uint64 if id64 else np.uint32).view(np.int64 if id64 else np.int32)
    return rp_h, col_h, torch.from_numpy(rp_h.view(np.int64)).cuda(), torch.from_numpy(col).cuda()


@pytest.mark.parametrize("own", [254, 255, 256, 257, 256 + 2047, 256 + 2048, 256 + 2049, 20_000])
@pytest.mark.parametrize("hubs", [1, 40])
@pytest.mark.parametrize("id64", [False, True])
def test_bfs_of_hubs_found_at_the_end_of_their_rows(own, hubs, id64):
    """Hubs one bottom-up level away, the neighbour in the frontier the last of
    their row, or the last but one, or missing: rows around what a lane walks
    and around the slices of what is left of them."""
    K = own * hubs // 4 + 100                       # the source's leaves: a wide frontier
    hub = 1 + np.arange(hubs)
    leaves = 1 + hubs + np.arange(hubs * own)
    last = 1 + hubs + hubs * own + np.arange(K)
    joined = hub[hub % 5 != 3]                      # the others are in components of their own
    e = np.concatenate([
        np.stack([np.zeros_like(last), last], 1),
        np.stack([np.repeat(hub, own), leaves], 1),
        np.stack([joined, last[joined]], 1),
        np.stack([joined[::2], last[joined[::2]] + 1], 1)])
    N = int(last[-1]) + 1
    rp_h, col_h, rp, col = _csr_on_gpu(e, N, id64)
    for source in (0, 1, int(last[0])):
        ref = o.bfs(rp_h, col_h, source)
        dist, levels, scanned = pg.bfs(rp, col, source, undirected=True)
        assert np.array_equal(dist.cpu().numpy().view(np.uint32), ref[0]), source
        assert (levels, scanned) == tuple(ref[1:3]), source


def test_bfs_past_a_hub_that_no_level_reaches_keeps_its_barriers_short():
    """A hub of 2^20 entries in another component: walked by one lane it holds a
    bottom-up level up for 0.1 s, and the others' barrier waits, here of some ten
    milliseconds, give up."""
    H, K = 2**20, 2**18
    e = np.concatenate([np.stack([np.full(H, 1), 2 + np.arange(H)], 1),
                        np.stack([np.zeros(K, np.int64), 2 + H + np.arange(K)], 1)])
    N = 2 + H + K
    _, _, rp, col = _csr_on_gpu(e, N)
    pg.pg_barrier_test_wait_hook(1 << 14, 0xFFFFFFFF)
    try:
        dist, levels, scanned = pg.bfs(rp, col, 0, undirected=True)
    finally:
        pg.pg_barrier_test_wait_hook(0, 0xFFFFFFFF)
    want = np.full(N, -1, np.int32)
    want[0], want[2 + H:] = 0, 1
    assert np.array_equal(dist.cpu().numpy(), want) and (levels, scanned) == (2, 2 * K)


@pytest.mark.parametrize("n,m,B,n0,most", [
    (1_000_000, 8, 1000, 9, 28_041_728), (2**20, 2, 2, 3, 4_199_424),
    (15 * 2**20, 4, 5, 5, 126_061_568), (256 * 3000, 5, 256, 6, None),
    (2**26, 5, 1024, 6, 922_789_120),      # the column scan in three steps
])
@pytest.mark.parametrize("id64", [False, True])
def test_pba_takes_the_smallest_workspace_and_none_below(n, m, B, n0, most, id64):
    """Whole-granule segments, `most` bytes or less (what these graphs took
    when they had no others): the same edges through every entry point."""
    need = pg.pg_pba_min_workspace_size(n, m, B)
    assert need <= pg.pg_pba_workspace_size(n, m, B) and (most is None or need <= most)
    buf = torch.full((need + 64,), 0x5A, dtype=torch.uint8, device="cuda")
    ws = buf[:need]
    ref = pg.gen_pba(n, m, B, n0, 1, 0.1, 3, id64=id64)
    assert torch.equal(pg.gen_pba(n, m, B, n0, 1, 0.1, 3, id64=id64, workspace=ws), ref)
    out = torch.empty_like(ref)
    host_out = torch.empty(ref.shape, dtype=ref.dtype, pin_memory=True)
    pg.gen_pba_to_host(host_out, n, m, B, n0, 1, 0.1, 3, id64=id64, out=out, workspace=ws)
    torch.cuda.synchronize()
    assert torch.equal(out, ref) and torch.equal(host_out.cuda(), ref)
    alone = [[b] for b in range(B)]            # width-1 factions, as a table
    got = pg.gen_pba_factions(n, m, alone, n0=n0, inter_frac=0.1, seed=3, id64=id64, out=out,
                              workspace=ws)
    assert torch.equal(got, ref)
    pg.pg_pba_prepare(n, m, B, n0, seed=3, workspace=ws)
    per = ref.shape[0] // B
    part = pg.gen_pba_blocks(ws, n, m, B, B // 2, B, n0=n0, seed=3, id64=id64)
    assert torch.equal(part, ref[B // 2 * per:])
    assert bool((buf[need:] == 0x5A).all())
    for call in (lambda w: pg.gen_pba(n, m, B, n0, 1, 0.1, 3, id64=id64, out=out, workspace=w),
                 lambda w: pg.pg_pba_prepare(n, m, B, n0, seed=3, workspace=w)):
        with pytest.raises(pg.PgenError) as err:
            call(ws[:need - 1])
        assert err.value.status == pg.PG_ENOMEM


def test_batch_takes_the_smallest_workspace_of_its_two_phase_jobs():
    jobs = [dict(kind="pba", n=256 * 3000, m=5, n0=6, seed=1, blocks=256, inter_frac=0.1),
            dict(kind="pba", n=2**20, m=2, n0=3, seed=2, blocks=2, inter_frac=0.1),
            dict(kind="kron", initiator=W.KRON_INITIATOR, k=12, n_edges=30_001, seed=3)]
    plan = pg.BatchPlan(jobs, tile_edges=2048)
    need = 256 + max(pg.pg_pba_min_workspace_size(j["n"], j["m"], j["blocks"]) for j in jobs[:2])
    assert need < pg.pg_batch_workspace_size(plan)
    ref = pg.gen_batch(plan)
    buf = torch.full((need + 64,), 0x5A, dtype=torch.uint8, device="cuda")
    got = pg.gen_batch(plan, workspace=buf[:need])
    for i in range(len(jobs)):
        assert torch.equal(plan.edges_of(got, i), plan.edges_of(ref, i)), i
    assert bool((buf[need:] == 0x5A).all())
    with pytest.raises(pg.PgenError) as err:
        pg.gen_batch(plan, workspace=buf[:need - 1])
    assert err.value.status == pg.PG_ENOMEM


@pytest.mark.parametrize("N,degree", [
    (2**18, 32), (2**18, 64),                         # rows around 64 and 128 in a level of most vertices
    ((5 << 18) + 1, 4), ((5 << 20) - 31, 3),          # more CTAs per SM, up to the last of them
    ((5 << 20) + 1, 2), ((5 << 20) + 1, 4), ((5 << 20) + 1, 12)])   # all CTAs, or the first few
def test_bfs_of_uniform_graphs_around_the_switches_of_wide_levels(N, degree):
    """Symmetrised lists of `degree` edges per vertex: row lengths on both sides
    of what is long in a narrow and in a wide level, and graphs on both sides
    of the rules for the number of CTAs (8 and 24 entries per row)."""
    rng = np.random.default_rng(N + degree)
    e = rng.integers(0, N, size=(N * degree, 2), dtype=np.uint32)
    rp, col = pg.edges_to_csr_opts(torch.from_numpy(e.view(np.int32)).cuda(), N, pg.CSR_SYMMETRIZE)
    rp_h, col_h = host(rp), host(col)
    for source in (0, N - 1):
        ref = o.bfs(rp_h, col_h, source)
        for undirected in (False, True):
            dist, levels, scanned = pg.bfs(rp, col, source, undirected=undirected)
            assert np.array_equal(dist.cpu().numpy().view(np.uint32), ref[0]), (source, undirected)
            assert (levels, scanned) == tuple(ref[1:3]), (source, undirected)


@pytest.mark.parametrize("which", [pg.DEG_OUT, pg.DEG_IN, pg.DEG_TOTAL])
@pytest.mark.parametrize("M", [1, 63, 64, 65, 511, 513, 152 * 6 * 512 - 1, 152 * 6 * 512 + 33])
@pytest.mark.parametrize("id64", [False, True])
def test_degrees_of_runs_across_a_warps_groups(which, M, id64):
    """Runs of every length up to 70 over the two groups of 32 edges a warp
    counts at once and over its trips; some ids past the vertex count."""
    rng = np.random.default_rng(M)
    src = np.repeat(rng.integers(0, 5000, M // 20 + 2), rng.integers(1, 71, M // 20 + 2))
    src = np.resize(src, M)
    e = np.stack([src, rng.integers(0, 5000, M)], 1).astype(np.int64)
    t = torch.from_numpy(e if id64 else e.astype(np.uint32).view(np.int32)).cuda()
    deg = pg.degrees(t, 4900, which)
    assert np.array_equal(host(deg), o.degrees(e.astype(np.uint64), 4900, which))
