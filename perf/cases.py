"""Performance cases: what a user of this framework has it do.

Four kinds of work, each through a public entry point:

* ``search``  -- ``Index.search``: a batch of queries against a resident
  index (Algorithm 1 per query): one interactive query, a few hundred, a
  full batch; one k for the batch or k and ef per query; small and large
  beams; the learned stop; cosine with the fast JLT rotation.
* ``trace``   -- ``Index.search_trace`` with the expansion path: the
  candidate search that index construction runs for every base vector.
* ``adjust``  -- ``index_builder.build_graph`` on the GPU: index
  construction's prune / reverse-edge / angle-rule step, host arrays in and
  out as its caller has them.
* ``train``   -- ``learned_stop.grad`` and ``adam``: one training step of
  the stop network.

Indexes are handles that a program loads once and keeps, so each is built
once per process, on synthetic vectors of a fixed seed, and shared by all
states; the queries (and the graph data, the training rows) come from the
state's own seed, drawn from the same mixtures as the index's vectors.
"""

from __future__ import annotations

import functools
import math
import os
import tempfile

import numpy as np
import torch

from paper_2411_12229_gb300 import index_builder as ib
from paper_2411_12229_gb300 import learned_stop as ls
from paper_2411_12229_gb300 import synth
from paper_2411_12229_gb300.api import Index

# The repository's own workloads at sizes that are built in seconds.  All but
# the tiny one are larger than the GPU's 129 MB L2 cache, as a real index is.
#   name: (workload, vectors, rotation, metric, out-degree)
INDEXES = {
    "tiny-d128": (synth.TINY_10K_D128, 10_000, "dense", "l2", 32),
    "sift-d128": (synth.BATCHED_1M_D128, 300_000, "dense", "l2", 32),
    "deep-d96": (synth.SERVING_4M_D96, 200_000, "dense", "l2", 32),
    "gist-d960": (synth.HIGHDIM_1M_D960, 30_000, "dense", "l2", 64),
    "unit-d1536": (synth.UNEVEN_1M_D1536, 24_000, "dense", "l2", 32),
    "cosine-d1024": (synth.HIGHDIM_1M_D960, 24_000, "fjlt", "cosine", 32),  # 960 columns padded to 1024
}


def block_bytes(index: str) -> int:
    """Bytes of one vertex block: raw vector, codes, four factor words and
    the id of every neighbour, padded to 128."""
    w, _, rotation, _, r = INDEXES[index]
    d = w.d if rotation == "dense" else 1 << math.ceil(math.log2(w.d))
    return -(-(4 * d + r * d // 8 + 16 * r + 4 * r) // 128) * 128


def workload(index: str) -> synth.Workload:
    w, n, _, _, _ = INDEXES[index]
    return synth.small(w, n, 1)


@functools.lru_cache(maxsize=None)
def resident(index: str) -> Index:
    """The index, built with Algorithm 2 on the GPU and loaded: the handle a
    serving program keeps for its lifetime."""
    _, _, rotation, metric, r = INDEXES[index]
    with tempfile.TemporaryDirectory() as td:
        path = os.path.join(td, "index.sqg")
        ib.build_index(path, synth.base(workload(index)), r, device=torch.cuda.current_device(), init="random",
                       iterations=3, ef_build=160, rotation=rotation, metric=metric)
        return Index(path)


@functools.lru_cache(maxsize=None)
def mixture(index: str):
    """Centres and per-dimension scales of the index's vectors, on the GPU."""
    w = workload(index)
    s = synth.dim_scales(w)
    return torch.from_numpy(synth.centers(w)).cuda(), None if s is None else torch.from_numpy(s).cuda()


def draw_queries(index: str, nq: int, gen: torch.Generator) -> torch.Tensor:
    """nq rows of the mixture the index's vectors come from."""
    w = workload(index)
    centres, scale = mixture(index)
    c = torch.randint(0, centres.shape[0], (nq,), generator=gen, device="cuda")
    x = centres[c] + w.noise_std * torch.randn((nq, w.d), generator=gen, device="cuda")
    if scale is not None:
        x = x * scale
    if w.dim_scale == "power":
        x = x.abs()
    if w.unit_norm:
        x = x / x.norm(dim=1, keepdim=True)
    return x.contiguous()


@functools.lru_cache(maxsize=None)
def stop_network() -> torch.Tensor:
    """A stop network with a clear rule -- stop once the share of the beam
    expanded without an improvement grows past a point -- plus the small
    weights that training leaves everywhere else."""
    p = 0.05 * ls.init_params(0)
    w1, w2, w3 = p[:1024].reshape(64, 16), p[1088:5184].reshape(64, 64), p[5248:5312]
    w1[0, 1] = 1.0    # expansions since the last improvement / ef
    w2[0, 0] = 1.0
    w3[0] = 8.0
    p[5312] = -2.5
    return torch.from_numpy(p).cuda()


def listed():
    return [
        # one interactive query: latency, launches and host work
        {"name": "one_query_d128", "kind": "search", "index": "sift-d128", "nq": 1, "k": 10, "ef": 64},
        # a small request batch against an index that fits in L2
        {"name": "small_batch_d128", "kind": "search", "index": "tiny-d128", "nq": 200, "k": 10, "ef": 64},
        # the full batch of the benchmark, at the beam that recall 0.95 needs
        {"name": "full_batch_d128", "kind": "search", "index": "sift-d128", "nq": 10_000, "k": 10, "ef": 40},
        # recall@100 retrieval: many results, a beam past 128 entries
        {"name": "top100_d128", "kind": "search", "index": "sift-d128", "nq": 2_001, "k": 100, "ef": 200},
        # one batch of the serving loop: k and ef per query, the caller's
        # output buffers and workspace, nothing read back
        {"name": "serving_mix_d96", "kind": "search", "index": "deep-d96", "nq": 719, "ks": "10,100", "ef": 160},
        # image descriptors: large blocks, out-degree 64
        {"name": "full_batch_d960", "kind": "search", "index": "gist-d960", "nq": 10_000, "k": 10, "ef": 112},
        # text embeddings, every request with its own k in {1, 10, 100} and
        # its own beam between k and 8 k
        {"name": "uneven_d1536", "kind": "search", "index": "unit-d1536", "nq": 5_000, "ks": "1,10,100", "ef_factor": 8},
        # cosine similarity with the fast JLT rotation, a ragged batch size
        {"name": "cosine_fjlt_d1024", "kind": "search", "index": "cosine-d1024", "nq": 1_501, "k": 10, "ef": 64},
        # the learned stop at a high-recall beam
        {"name": "learned_stop_d128", "kind": "search", "index": "sift-d128", "nq": 5_003, "k": 10, "ef": 96,
         "stop_every": 16},
        # index construction: candidates of a slice of the base vectors, at
        # the paper's beam of 400, with the path from the entry point
        {"name": "build_candidates_d128", "kind": "trace", "index": "sift-d128", "nq": 16_384, "k": 64, "ef": 400},
        # index construction: pruning, reverse edges and the angle rule
        {"name": "build_adjust_d128", "kind": "adjust", "n": 20_000, "d": 128, "cand": 96, "r": 32},
        # training the stop network: the minibatch of learned_stop.train
        {"name": "stop_train_step", "kind": "train", "n": 8_192},
    ]


_COST = 1.0e10  # nq * ef * block bytes of a drawn search: under the largest listed one


def _log_int(rng, lo, hi):
    return min(hi, max(lo, int(round(math.exp(rng.uniform(math.log(lo), math.log(hi)))))))


def draw(rng):
    kind = rng.choice(("search",) * 7 + ("trace", "adjust", "train"))
    if kind == "train":
        return {"kind": kind, "n": _log_int(rng, 200, 16_384)}
    if kind == "adjust":
        d = rng.choice((96, 128, 256))
        return {"kind": kind, "n": _log_int(rng, 2_000, 20_000 * 128 // max(d, 128)), "d": d,
                "cand": rng.randint(64, 96), "r": 32}
    index = rng.choice(list(INDEXES))
    if kind == "trace":
        index = rng.choice(("tiny-d128", "sift-d128", "deep-d96"))
        ef = _log_int(rng, 100, 400)
        return {"kind": kind, "index": index, "nq": _log_int(rng, 500, 16_384), "k": rng.randint(32, 64), "ef": ef}
    case = {"kind": kind, "index": index}
    form = rng.choice(("one", "one", "mix", "factor", "stop"))
    if form == "mix":
        case["ks"] = rng.choice(("10,100", "1,10", "1,10,100"))
        case["ef"] = ef = _log_int(rng, 100, 256)
    elif form == "factor":
        case["ks"] = rng.choice(("1,10", "1,10,100"))
        case["ef_factor"] = rng.randint(2, 8)
        ef = 400
    else:
        case["k"] = rng.choice((1, 10, 10, rng.randint(2, 100)))
        case["ef"] = ef = _log_int(rng, max(16, case["k"]), 300)
        if form == "stop":
            case["stop_every"] = rng.choice((4, 8, 16))
    most = int(min(10_000, _COST / (ef * block_bytes(index))))
    case["nq"] = _log_int(rng, 1, most)
    return case


def _generator(seed: int) -> torch.Generator:
    g = torch.Generator(device="cuda")
    g.manual_seed(int(seed))
    return g


def _prepare_search(case, gen):
    ix = resident(case["index"])
    nq = case["nq"]
    st = {"kind": "search", "ix": ix, "q": draw_queries(case["index"], nq, gen), "kw": {}}
    if "ks" not in case:
        st["k"], st["ef"] = case["k"], case["ef"]
        if "stop_every" in case:
            st["kw"] = {"stop_mlp": stop_network(), "stop_logit": 0.0, "stop_every": case["stop_every"]}
        return st
    # every request has its own k and ef; the caller knows the bounds and
    # keeps output buffers and a workspace, as the serving loop does
    choices = [int(s) for s in case["ks"].split(",")]
    # every k equally often, in an order of the seed's own
    order = torch.randperm(nq, generator=gen, device="cuda")
    k = torch.tensor(choices, device="cuda")[order % len(choices)]
    if "ef_factor" in case:
        top = case["ef_factor"] * k
        ef = k + (torch.rand(nq, generator=gen, device="cuda") * (top - k + 1)).long().clamp(max=top - k)
        max_ef = case["ef_factor"] * max(choices)
    else:
        max_ef = case["ef"]
        ef = torch.full((nq,), max_ef, device="cuda")
    max_k, total = max(choices), int(k.sum())
    st.update(k=k.int(), ef=ef.int())
    st["kw"] = {"max_k": max_k, "max_ef": max_ef,
                "out": (torch.empty(total, dtype=torch.int32, device="cuda"),
                        torch.empty(total, dtype=torch.float32, device="cuda")),
                "workspace": torch.empty(ix.workspace_size(nq, max_k, max_ef), dtype=torch.uint8, device="cuda")}
    return st


def _prepare_adjust(case, gen):
    """Vectors of a clustered mixture and each one's candidates: its nearest
    vectors and the vertices of a search path (here: random ones)."""
    n, d, m = case["n"], case["d"], case["cand"]
    centres = 2.0 * torch.randn((max(4, n // 1000), d), generator=gen, device="cuda")
    x = centres[torch.randint(0, centres.shape[0], (n,), generator=gen, device="cuda")]
    x = x + torch.randn((n, d), generator=gen, device="cuda")
    near = m - m // 3
    sq = (x * x).sum(1)
    cand = torch.empty((n, m), dtype=torch.int64, device="cuda")
    for a in range(0, n, 4096):
        dist = sq[None, :] - 2.0 * (x[a:a + 4096] @ x.T)
        cand[a:a + 4096, :near] = torch.topk(dist, near + 1, dim=1, largest=False).indices[:, 1:]
    cand[:, near:] = torch.randint(0, n, (n, m - near), generator=gen, device="cuda")
    entry = int((x - x.mean(0)).square().sum(1).argmin())
    return {"kind": "adjust", "x": x.cpu().numpy(), "cand": cand.int().cpu().numpy().view(np.uint32), "r": case["r"],
            "entry": entry}


def _train_inputs(case, gen):
    """Parameters and Adam's moments in mid-training, and a minibatch of
    feature rows with their labels and class weights."""
    n = case["n"]
    p = torch.from_numpy(ls.init_params(1)).cuda()
    p = p + 0.02 * torch.randn(p.shape, generator=gen, device="cuda")
    m = 1e-3 * torch.randn(p.shape, generator=gen, device="cuda")
    v = 1e-5 * (0.1 + torch.rand(p.shape, generator=gen, device="cuda"))
    x = torch.rand((n, 16), generator=gen, device="cuda").mul_(2.0)
    y = (torch.rand(n, generator=gen, device="cuda") < 0.3).float()
    w = torch.where(y > 0.5, 0.5 / 0.3, 0.5 / 0.7).float()
    return p, m, v, x, y, w


def prepare(case, seed):
    gen = _generator(seed)
    kind = case["kind"]
    if kind == "search":
        return _prepare_search(case, gen)
    if kind == "trace":
        return {"kind": kind, "ix": resident(case["index"]), "q": draw_queries(case["index"], case["nq"], gen),
                "k": case["k"], "ef": case["ef"]}
    if kind == "adjust":
        return _prepare_adjust(case, gen)
    return {"kind": kind, "in": _train_inputs(case, gen)}


def run(state):
    kind = state["kind"]
    if kind == "search":
        return state["ix"].search(state["q"], state["k"], state["ef"], stats=True, **state["kw"])
    if kind == "trace":
        ids, dists, st, _, _, _, path = state["ix"].search_trace(state["q"], state["k"], state["ef"], None, 0,
                                                                 path_cap=state["ix"].degree)
        return ids, dists, st, path
    if kind == "adjust":
        adj, info = ib.build_graph(state["x"], state["cand"], state["r"], state["entry"],
                                   device=torch.cuda.current_device())
        return adj.view(np.int32), info["supplemented"], info["random_filled"], info["repairs"]
    p, m, v, x, y, w = state["in"]
    loss, g = ls.grad(p, x, y, w)
    ls.adam(p, g, m, v, 1000, 3e-4)
    return loss, g, p, m, v


def work(case):
    kind = case["kind"]
    if kind == "train":
        n, p = case["n"], 5313
        return {"bytes": 4.0 * (n * 18 + 7 * p + 1), "flops": 6.0 * n * 5184}
    if kind == "adjust":
        # the rows and the lists once; the distances of every candidate and of
        # the pairs that the rules compare, at least one per candidate
        n, d, m, r = case["n"], case["d"], case["cand"], case["r"]
        return {"bytes": 4.0 * n * (d + m + r), "flops": 3.0 * d * n * (2 * m)}
    # About ef expansions per query (0.7 to 1.1 ef over these beams).  A block
    # is needed once by every query that expands it and the index is an input
    # once: no more than the whole index.
    w, n, rotation, _, r = INDEXES[case["index"]]
    nq, bb = case["nq"], block_bytes(case["index"])
    if "ks" in case:
        ks = [int(s) for s in case["ks"].split(",")]
        k = sum(ks) / len(ks)
        ef = case.get("ef") or k * (1 + case["ef_factor"]) / 2
    else:
        k, ef = case["k"], case["ef"]
    d = w.d
    per_block = 3 * d + r * (2 * d + 8)  # the exact distance, and an integer dot product per neighbour
    rot = 2.0 * d * d if rotation == "dense" else 6.0 * 1024 * 10
    out = 8.0 * k + 8 + (4 * r if kind == "trace" else 0)
    return {"bytes": min(nq * ef, n) * bb + nq * (4.0 * d + out), "flops": nq * (ef * per_block + rot)}


def exact(case, seed):
    """The training step in 64 bits.  A search's outputs are decided by its
    own fp32 estimates and an adjusted graph is whole numbers: neither has a
    value that plain 64-bit arithmetic would give."""
    if case["kind"] != "train":
        return None
    p, m, v, x, y, w = (t.double() for t in _train_inputs(case, _generator(seed)))
    p.requires_grad_(True)
    w1, b1, w2 = p[:1024].view(64, 16), p[1024:1088], p[1088:5184].view(64, 64)
    b2, w3, b3 = p[5184:5248], p[5248:5312], p[5312]
    z = torch.relu(torch.relu(x @ w1.T + b1) @ w2.T + b2) @ w3 + b3
    loss = (w * (torch.nn.functional.softplus(z) - y * z)).sum() / w.sum()
    g, = torch.autograd.grad(loss, p)
    m2, v2 = 0.9 * m + 0.1 * g, 0.999 * v + 0.001 * g * g
    step = (m2 / (1 - 0.9 ** 1000)) / ((v2 / (1 - 0.999 ** 1000)).sqrt() + 1e-8)
    return loss.detach().view(1), g, p.detach() - 3e-4 * step, m2, v2
