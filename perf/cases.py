"""What the speed of this library is measured on.

A case is one call of the retrieval stage as a serving program makes it: IVF-PQ search over an index that is loaded
once (`rago_search` on device tensors, `rago_search_host` on host buffers, 8-bit or 4-bit codes, one- or two-level
coarse quantiser) and exact flat search over a small database.  Sizes are those of the benchmark shapes in
`synth.CONFIGS` (the largest database cut to what three indexes of it leave room for), of the test suite, and generic
batch sizes between them.
"""

import math

import torch

from paper_2503_14649_b200 import binding, synth

TREE_B1 = 8  # level-1 nodes a two-level search keeps


def _ivf(name, N, d, nlist, M, nq, nprobe, k, metric="l2", coarse="f32", bits=8, zipf=0.0, tree=0, host=False):
    """M = code bytes per vector; zipf = exponent of the list sizes (0: even); tree = level-1 nodes (0: one level)."""
    c = dict(kind="ivf", N=N, d=d, nlist=nlist, M=M, nq=nq, nprobe=nprobe, k=k, metric=metric, coarse=coarse, bits=bits,
             zipf=zipf, tree=tree, host=host)
    return dict(c, name=name) if name else c


def _flat(name, N, d, nq, k):
    c = dict(kind="flat", N=N, d=d, nq=nq, k=k)
    return dict(c, name=name) if name else c


def listed():
    return [
        # Iterative retrieval: one sequence asks for its next passage while it generates, so each call is a single
        # query and its latency stalls the decoder.
        _ivf("iterative_1", 100_000_000, 512, 16_384, 32, 1, 16, 20),
        # The same stream when a decode batch of 16 sequences reaches its retrieval points together.
        _ivf("iterative_16", 100_000_000, 512, 16_384, 32, 16, 16, 20),
        # A few sequences at a time through the two-level quantiser that larger list counts ask for.
        _ivf("iterative_tree_5", 100_000_000, 512, 16_384, 32, 5, 16, 20, tree=128),
        # A small private index (a tenant's documents, a test corpus), one modest batch.
        _ivf("tiny_64", 100_000, 128, 256, 16, 64, 8, 10),
        # BERT-width passages with skewed topics, a throughput-oriented batch.
        _ivf("mid_1024", 10_000_000, 768, 4096, 96, 1024, 32, 100, zipf=1.1),
        # The same index behind a serving front end: a ragged batch that arrives in host memory and is answered there.
        _ivf("mid_host_77", 10_000_000, 768, 4096, 96, 77, 32, 100, zipf=1.1, host=True),
        # Low-precision codes (two 4-bit codes per byte) for a corpus that has to stay small, an ordinary batch.
        _ivf("pq4_300", 10_000_000, 768, 4096, 48, 300, 32, 100, bits=4, zipf=1.1),
        # One GPU's part of a hyperscale passage database: the largest batch, many short lists, inner product over a
        # bf16 coarse quantiser.
        _ivf("hyperscale_4096", 250_000_000, 768, 65_536, 64, 4096, 64, 100, metric="ip", coarse="bf16"),
        # The same index when traffic is low: a ragged batch just above what the small-batch kernels take.
        _ivf("hyperscale_33", 250_000_000, 768, 65_536, 64, 33, 64, 100, metric="ip", coarse="bf16"),
        # Chunks of one long document searched exactly for a single question.
        _flat("flat_chunks_1", 100_000, 768, 1, 10),
        # A ragged chunk store and a few questions at once.
        _flat("flat_37", 1_000_003, 768, 37, 100),
        # The full chunk store and a throughput batch.
        _flat("flat_256", 10_000_000, 1024, 256, 100),
    ]


def _log_int(rng, lo, hi):
    return max(lo, min(hi, int(round(math.exp(rng.uniform(math.log(lo), math.log(hi)))))))


def draw(rng):
    if rng.random() < 0.3:
        d = 64 * rng.choice([2, 4, 6, 8, 12, 16])
        N = _log_int(rng, 20_000, 10_000_000)
        return _flat(None, N, d, _log_int(rng, 1, 256), _log_int(rng, 1, 128))
    bits = 4 if rng.random() < 0.2 else 8
    M = rng.choice([16, 32, 48, 64, 96] if bits == 4 else [16, 32, 48, 64, 96, 128])
    dsub = rng.choice([s for s in (4, 8, 12, 16) if M * s <= 1024])
    N = _log_int(rng, 100_000, 100_000_000 if bits == 8 else 10_000_000)
    nlist = max(64, min(65_536, N // _log_int(rng, 400, 8000)))
    nprobe = _log_int(rng, 4, 64)
    nq = _log_int(rng, 1, 4096)
    k = _log_int(rng, 1, 128)
    coarse = rng.choice(["f32", "bf16"])
    tree = 64 if nlist >= 4096 and nq <= 64 and rng.random() < 0.3 else 0
    # no more than the largest listed case costs: bytes of code scanned, and multiply-adds of the coarse step
    nq = max(1, min(nq, int(40e9 / (nprobe * (N / nlist) * M)), int(400e9 / (nlist * M * dsub * (6 if coarse == "f32" else 1)))))
    return _ivf(None, N, M * dsub, nlist, M, nq, nprobe, k, metric=rng.choice(["l2", "ip"]), coarse=coarse, bits=bits,
                zipf=rng.choice([0.0, 1.1]) if N <= 2_000_000 and not tree else 0.0, tree=tree, host=rng.random() < 0.2)


def _ivf_data(c, seed):
    kw = dict(metric=c["metric"], seed=seed, coarse_bf16=c["coarse"] == "bf16", device="cuda")
    if c["bits"] == 4:
        return synth.make_ivfpq4(c["N"], c["d"], c["nlist"], 2 * c["M"], c["nq"], zipf=c["zipf"] or None, **kw)
    if c["zipf"] or (c["N"] <= 2_000_000 and not c["tree"]):  # vectors drawn from the mixture and encoded
        return synth.make_ivfpq(c["N"], c["d"], c["nlist"], c["M"], c["nq"], zipf=c["zipf"] or None, **kw)
    return synth.make_ivfpq_hashed(c["N"], c["d"], c["nlist"], c["M"], c["nq"], tree_n1=c["tree"] or None, **kw)


def prepare(case, seed):
    if case["kind"] == "flat":
        db, queries = synth.make_flat(case["N"], case["d"], case["nq"], seed=seed, device="cuda")
        return dict(case=case, db=db, queries=queries)
    data = _ivf_data(case, seed)
    index = binding.load_index_from(data, "cuda")
    if case["tree"]:
        index.rago_index_set_coarse_tree(data.extra["level1"].cuda(), data.extra["child_offsets"].cuda(), b1=TREE_B1)
    state = dict(case=case, index=index)
    if not case["host"]:
        state["queries"] = data.queries.contiguous()
        return state
    nq, k = case["nq"], case["k"]
    need = index.search_workspace_bytes(nq, case["nprobe"], k) + index.host_staging_bytes(nq, k)
    state["queries"] = data.queries.cpu().contiguous().pin_memory()
    state["ids"] = torch.empty((nq, k), dtype=torch.int64).pin_memory()
    state["dists"] = torch.empty((nq, k), dtype=torch.float32).pin_memory()
    state["workspace"] = torch.empty(need, dtype=torch.uint8, device="cuda")
    return state


def run(state):
    c = state["case"]
    if c["kind"] == "flat":
        return binding.rago_flat_search(state["db"], state["queries"], c["k"])
    if c["host"]:
        state["index"].rago_search_host(state["queries"], c["nprobe"], c["k"], state["ids"], state["dists"],
                                        state["workspace"])
        return state["ids"], state["dists"]
    return state["index"].rago_search(state["queries"], c["nprobe"], c["k"])


def _scan_sizes(c):
    """(vectors scored, distinct vectors read) by one search: a query probes its own list, drawn by list size, and
    lists that are as good as random."""
    n, q, p = c["nlist"], c["nq"], c["nprobe"]
    w = synth.zipf_weights(n, c["zipf"]) if c["zipf"] else torch.full((n,), 1.0 / n, dtype=torch.float64)
    own = q * float((w * w).sum()) * c["N"]
    scored = own + q * (p - 1) * c["N"] / n
    missed = (1.0 - w) ** q * (1.0 - (p - 1) / n) ** q  # chance that no query probes the list
    return scored, c["N"] * float((w * (1.0 - missed)).sum())


def work(case):
    """Codes of the probed lists, coarse centroids, queries and answers, each once; two operations for each
    coordinate of a coarse (or flat) score and one for each code byte of a scored vector."""
    nq, d, k = case["nq"], case["d"], case["k"]
    if case["kind"] == "flat":
        return dict(bytes=2.0 * d * (case["N"] + nq) + 12.0 * nq * k, flops=2.0 * nq * case["N"] * d)
    rows = case["nlist"]
    if case["tree"]:
        rows = case["tree"] + min(rows, nq * TREE_B1 * rows // case["tree"])
    scored, read = _scan_sizes(case)
    cb = 2 if case["coarse"] == "bf16" else 4
    books = (32 if case["bits"] == 4 else 256) * d * 4
    bytes_ = read * (case["M"] + (4 if case["metric"] == "l2" else 0)) + rows * d * cb + books + nq * d * 4.0 + 12.0 * nq * k
    per_query = case["tree"] + TREE_B1 * case["nlist"] // case["tree"] if case["tree"] else case["nlist"]
    return dict(bytes=bytes_, flops=2.0 * nq * per_query * d + scored * case["M"])


def tolerance(case):
    """About four times what the results differ by from the same scores summed in 64 bits (over the listed and some
    drawn cases: IVF-PQ rel 8e-8, max 3e-7; flat rel 1e-6, max 2e-6), and the share of ids that ties within such
    differences reorder (up to 6e-4 and 1e-3 seen)."""
    if case["kind"] == "flat":
        return {"rel": 4e-6, "max": 1e-5, "differ": 0.004}
    return {"rel": 4e-7, "max": 2e-6, "differ": 0.004}
