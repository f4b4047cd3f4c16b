"""Performance cases of the library: the calls its users make, through the public binding.

Every case is a dict of plain values. `prepare` makes what a program holds before the call (output
buffers, workspaces, an edge list, a CSR, a batch plan), `run` makes the call and returns its whole
outputs, `work` states the bytes one pass cannot do without. All results are integers: they are a
pure function of the arguments and have no rounding.

Kinds:
  ba        gen_pba with one block (serial Barabasi-Albert)
  pba       gen_pba with blocks > 1 (two-phase PBA), edge list only
  pba_csr   the same followed by edges_to_csr (a list grouped by source)
  kron_csr  gen_kronecker (stochastic) followed by edges_to_csr (a list that needs the sort)
  kron_det  gen_kronecker, deterministic expansion
  kron_xor  gen_kronecker and gen_random_cells in one list, and the CSR of its odd cells
            (the steps of kronecker_xor_random)
  simple    edges_to_csr_opts of a Kronecker list: symmetrised, without duplicates and loops
  analyze   degrees, degree histogram and breadth-first searches of a PBA graph
  batch     gen_batch of a mix of graphs, then gen_batch_csr of the small ones
"""
import math
import random

import torch

import paper_1003_3684_gb300 as pg
from paper_1003_3684_gb300 import workloads

UNDIRECTED_SIMPLE = pg.CSR_SYMMETRIZE | pg.CSR_DEDUP | pg.CSR_NO_LOOPS
MAX_DEGREE = 4096          # buckets of the analysis' degree histogram
SMALL_JOB_EDGES = 1 << 17  # batch jobs below this get their CSR from the batch's one sort


def listed():
    return [
        # the serial BA configuration: a small graph, one launch, bound by latency
        dict(name="ba_n100k_m4", kind="ba", n=100_000, m=4, n0=5, id64=False),
        # a small two-phase graph with block sizes that are no power of two, and its CSR: the
        # first thing a user tries, many launches on little work
        dict(name="pba_n160k_b16_csr", kind="pba_csr", n=160_000, m=4, blocks=16, n0=5, width=2,
             frac=0.3, id64=False),
        # a two-phase graph of ordinary size (the one the path-length study searches)
        dict(name="pba_n2p24_b64", kind="pba", n=2**24, m=5, blocks=64, n0=6, width=1, frac=0.1,
             id64=False),
        # the paper's headline graph: 2^30 vertices, 5.37e9 edges
        dict(name="pba_n2p30_b1024", kind="pba", n=2**30, m=5, blocks=1024, n0=6, width=1,
             frac=0.1, id64=False),
        # a served request of ordinary size with an odd edge count, and its CSR
        dict(name="kron_k13_csr", kind="kron_csr", k=13, n_edges=100_003, id64=False),
        # the Kronecker configuration: 2^20 vertices, 16 edges per vertex, with CSR
        dict(name="kron_k20_csr", kind="kron_csr", k=20, n_edges=16 * 2**20, id64=False),
        # the same at 2^26 vertices and 2^30 edges
        dict(name="kron_k26_csr", kind="kron_csr", k=26, n_edges=16 * 2**26, id64=False),
        # the paper's deterministic expansion of its Fig. 2 seed
        dict(name="kron_det_fig2_k8", kind="kron_det", k=8, id64=False),
        # the paper's randomisation of a Kronecker graph by exclusive-or with a random graph
        dict(name="kron_k20_xor", kind="kron_xor", k=20, n_edges=16 * 2**20, n_random=2**20,
             id64=False),
        # a simple undirected graph from a directed list with 64-bit ids, ragged edge count
        dict(name="kron_k21_id64_simple", kind="simple", k=21, n_edges=20_000_003, id64=True),
        # the study of Sec. 4: degrees, their histogram, path lengths from eight sources
        dict(name="analyze_pba_n2p24", kind="analyze", n=2**24, m=5, blocks=64, n0=6, sources=8),
        # many graphs of uneven sizes at once, and the CSRs of the small ones
        dict(name="batch_256_mixed", kind="batch", n_jobs=256),
    ]


def _log_int(rng, lo, hi):
    """An integer between lo and hi, uniform in its logarithm."""
    return max(lo, min(hi, int(round(math.exp(rng.uniform(math.log(lo), math.log(hi)))))))


def draw(rng):
    kind = rng.choice(["ba", "pba", "pba_csr", "kron_csr", "kron_csr", "kron_det", "kron_xor",
                       "simple", "analyze", "batch"])
    id64 = rng.random() < 0.25
    if kind == "ba":
        m = rng.randint(1, 8)
        return dict(kind=kind, n=_log_int(rng, 1000, 2**26 // m), m=m, n0=m + 1, id64=id64)
    if kind in ("pba", "pba_csr", "analyze"):
        m = rng.randint(2, 8)
        blocks = rng.choice([2, 5, 8, 16, 50, 64, 128, 256, 1000, 1024])
        top = {"pba": 2**30, "pba_csr": 2**28, "analyze": 2**26}[kind]
        per = _log_int(rng, 64, max(65, min(2**20, top // m // blocks)))
        if rng.random() < 0.3:
            per = 2 ** int(math.log2(per))   # the block sizes the configurations use
        c = dict(kind=kind, n=per * blocks, m=m, blocks=blocks, n0=m + 1)
        if kind == "analyze":
            return dict(c, sources=rng.randint(1, 8))
        width = rng.choice([1, 1, 2 if blocks % 2 == 0 else 1])
        return dict(c, width=width, frac=rng.choice([0.05, 0.1, 0.3]), id64=id64)
    if kind == "kron_det":
        return dict(kind=kind, k=rng.randint(3, 8), id64=id64)
    if kind == "batch":
        return dict(kind=kind, n_jobs=_log_int(rng, 4, 256))
    # Kronecker lists of about 16 edges per vertex
    n_edges = _log_int(rng, 2**12, 2**28 if kind == "kron_csr" else 2**25)
    k = max(1, math.ceil(math.log2(n_edges / 16)))
    c = dict(kind=kind, k=k, n_edges=n_edges, id64=id64)
    if kind == "kron_xor":
        # 32-bit ids want one of the two lists of even length
        c["n_random"] = max(2, n_edges // 16) & ~1
    return c


def _ids(id64):
    return torch.int64 if id64 else torch.int32


def _pair_bytes(id64):
    return 16 if id64 else 8


def _edges(case):
    if case["kind"] in ("ba", "pba", "pba_csr", "analyze"):
        return pg.pg_pba_edge_count(case["n"], case["m"], case.get("blocks", 1), case["n0"])
    if case["kind"] == "kron_det":
        return 11 ** case["k"]
    return case["n_edges"]


def _vertices(case):
    if case["kind"] in ("ba", "pba", "pba_csr", "analyze"):
        return case["n"] + case.get("blocks", 1) * case["n0"]
    return 2 ** case["k"]


def _csr_buffers(s, E, N, id64, flags=0):
    listed_edges = 2 * E if flags & pg.CSR_SYMMETRIZE else E
    s["row_ptr"] = torch.empty(N + 1, dtype=torch.int64, device="cuda")
    # zeros: with options the call writes the entries it keeps and leaves the rest alone
    s["col"] = torch.zeros(max(listed_edges, 1), dtype=_ids(id64), device="cuda")
    if not flags:   # the options' workspace is made by the call itself
        s["csr_ws"] = torch.empty(pg.pg_csr_workspace_size(E, N), dtype=torch.uint8,
                                  device="cuda")


def _batch_jobs(n_jobs, seed):
    jobs = workloads.batch_jobs(n_jobs)
    for i, j in enumerate(jobs):
        edges = j["n"] * j["m"] if j["kind"] == "pba" else j["n_edges"]
        j["seed"] = seed + i
        j["want_csr"] = edges < SMALL_JOB_EDGES
    return jobs


def prepare(case, seed):
    kind, id64 = case["kind"], case.get("id64", False)
    s = dict(case, seed=seed)
    if kind == "batch":
        plan = pg.BatchPlan(_batch_jobs(case["n_jobs"], seed), tile_edges=4096)
        s["plan"] = plan
        s["arena"] = torch.empty((max(plan.total_edges, 1), 2), dtype=torch.int32, device="cuda")
        s["ws"] = torch.empty(pg.pg_batch_workspace_size(plan), dtype=torch.uint8, device="cuda")
        s["row_ptr"] = torch.empty(max(plan.csr_rows_total, 1), dtype=torch.int64, device="cuda")
        s["col"] = torch.empty(max(plan.csr_cols_total, 1), dtype=torch.int32, device="cuda")
        s["csr_ws"] = torch.empty(max(pg.pg_batch_csr_workspace_size(plan), 256),
                                  dtype=torch.uint8, device="cuda")
        return s
    E, N = _edges(case), _vertices(case)
    if kind == "analyze":
        # a PBA graph as its edge list and its undirected CSR
        s["edges"] = pg.gen_pba(case["n"], case["m"], case["blocks"], case["n0"], 1, 0.1, seed)
        s["row_ptr"], s["col"] = pg.edges_to_csr_opts(s["edges"], N, pg.CSR_SYMMETRIZE)
        rng = random.Random(seed)
        s["from"] = [rng.randrange(N) for _ in range(case["sources"])]
        s["deg"] = torch.empty(N, dtype=torch.int64, device="cuda")
        s["dist"] = [torch.empty(N, dtype=torch.int32, device="cuda") for _ in s["from"]]
        # two frontiers and a long-row list of N words each, the counters and a bitmap
        s["ws"] = torch.empty(16 * (N + 64) + 256 + N // 8 + 512, dtype=torch.uint8,
                              device="cuda")
        return s
    if kind == "kron_xor":
        # both lists in one buffer; the random one first, as its length is even and the second
        # list starts on a 16-byte boundary
        s["edges"] = torch.empty((case["n_random"] + E, 2), dtype=_ids(id64), device="cuda")
        _csr_buffers(s, case["n_random"] + E, N, id64, pg.CSR_ODD)
        return s
    if kind == "simple":
        s["edges"] = pg.gen_kronecker(workloads.KRON_INITIATOR, case["k"], E, seed, id64=id64)
        _csr_buffers(s, E, N, id64, UNDIRECTED_SIMPLE)
        return s
    s["edges"] = torch.empty((E, 2), dtype=_ids(id64), device="cuda")
    if kind == "kron_det":
        # the Fig. 2 seed graph with its vertices numbered in another order
        at = random.Random(seed).sample(range(5), 5)
        s["graph"] = [[workloads.PK_FIG2_SEED[a][b] for b in at] for a in at]
    if kind in ("pba", "pba_csr"):
        need = pg.pg_pba_workspace_size(case["n"], case["m"], case["blocks"])
        s["ws"] = torch.empty(need, dtype=torch.uint8, device="cuda")
    if kind in ("pba_csr", "kron_csr"):
        _csr_buffers(s, E, N, id64)
    return s


def run(s):
    kind, id64, seed = s["kind"], s.get("id64", False), s["seed"]
    if kind == "ba":
        return pg.gen_pba(s["n"], s["m"], 1, s["n0"], 1, 0.0, seed, id64=id64, out=s["edges"])
    if kind in ("pba", "pba_csr"):
        edges = pg.gen_pba(s["n"], s["m"], s["blocks"], s["n0"], s["width"], s["frac"], seed,
                           id64=id64, out=s["edges"], workspace=s["ws"])
        if kind == "pba":
            return edges
        return [edges, *pg.edges_to_csr(edges, _vertices(s), row_ptr=s["row_ptr"], col=s["col"],
                                        workspace=s["csr_ws"])]
    if kind == "kron_csr":
        edges = pg.gen_kronecker(workloads.KRON_INITIATOR, s["k"], s["n_edges"], seed, id64=id64,
                                 out=s["edges"])
        return [edges, *pg.edges_to_csr(edges, _vertices(s), row_ptr=s["row_ptr"], col=s["col"],
                                        workspace=s["csr_ws"])]
    if kind == "kron_det":
        return pg.gen_kronecker(s["graph"], s["k"], deterministic=True, id64=id64,
                                out=s["edges"])
    if kind == "kron_xor":
        first = s["n_random"]
        pg.gen_random_cells(_vertices(s), first, seed, id64=id64, out=s["edges"][:first])
        pg.gen_kronecker(workloads.KRON_INITIATOR, s["k"], s["n_edges"], seed, id64=id64,
                         out=s["edges"][first:])
        return pg.edges_to_csr_opts(s["edges"], _vertices(s), pg.CSR_ODD, row_ptr=s["row_ptr"],
                                    col=s["col"])
    if kind == "simple":
        return pg.edges_to_csr_opts(s["edges"], _vertices(s), UNDIRECTED_SIMPLE,
                                    row_ptr=s["row_ptr"], col=s["col"])
    if kind == "analyze":
        deg = pg.degrees(s["edges"], _vertices(s), pg.DEG_TOTAL, out=s["deg"])
        out = [deg, pg.degree_histogram(deg, MAX_DEGREE)]
        for source, dist in zip(s["from"], s["dist"]):
            out += pg.bfs(s["row_ptr"], s["col"], source, dist=dist, workspace=s["ws"],
                          undirected=True)
        return out
    arena = pg.gen_batch(s["plan"], arena=s["arena"], workspace=s["ws"])
    if s["plan"].csr_rows_total == 0:
        return arena
    return [arena, *pg.gen_batch_csr(s["plan"], arena, row_ptr=s["row_ptr"], col=s["col"],
                                     workspace=s["csr_ws"])]


def work(case):
    """Bytes that must move: each output written once, each input list read once, a list that a
    later stage of the same pass consumes written once and read once. The arithmetic is integer
    (Philox draws and index arithmetic), so there are no floating-point operations."""
    kind, id64 = case["kind"], case.get("id64", False)
    if kind == "batch":
        total = csr = rows = 0
        for j in _batch_jobs(case["n_jobs"], 0):
            if j["kind"] == "pba":
                e, v = j["n"] * j["m"] + j["n0"] * (j["n0"] - 1) // 2, j["n"] + j["n0"]
            else:
                e, v = j["n_edges"], 2 ** j["k"]
            total += e
            if j["want_csr"]:
                csr, rows = csr + e, rows + v + 1
        return dict(bytes=total * 8 + csr * (8 + 4) + rows * 8, flops=0)
    E, N = _edges(case), _vertices(case)
    pair = _pair_bytes(id64)
    if kind in ("ba", "pba", "kron_det"):
        return dict(bytes=E * pair, flops=0)
    if kind in ("pba_csr", "kron_csr"):
        return dict(bytes=E * (2 * pair + pair // 2) + (N + 1) * 8, flops=0)
    if kind == "kron_xor":
        M = E + case["n_random"]
        return dict(bytes=M * (2 * pair + pair // 2) + (N + 1) * 8, flops=0)
    if kind == "simple":
        return dict(bytes=E * (pair + 2 * (pair // 2)) + (N + 1) * 8, flops=0)
    # degrees read the list and write N counts, the histogram reads them; a search writes N
    # distances and reads the rows it scans, at least one entry of each vertex
    search = N * (4 + 8 + 4)
    return dict(bytes=E * 8 + 2 * N * 8 + (MAX_DEGREE + 2) * 8 + case["sources"] * search, flops=0)


def exact(case, seed):
    """Nothing to add: every output is a whole number, equal or wrong."""
    return None
