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
