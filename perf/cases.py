"""The work a decoding program has this library do, as measurable cases.

Three kinds of pass, each through the public entry points of `paper_2505_20776_b200`:

  verify   one verification step of a target model: attention of the draft tree over the prefix cache and the
           tree, layer by layer; the last layer also yields the chunk scores, which are ranked (SelectChunks) and
           followed by the rewrite of the draft model's cache (UpdateDraftCache).
  draft    one forward of the draft model on that compact cache, whose length is an int32 on the device.
  prefill  causal self-attention over a prompt.

Everything is bf16 with fp32 statistics, the library's only data type.  A case is a dict of plain values:
`prepare` makes what a program holds before the call, `run` is one pass, `work` what a pass cannot do without.
"""
import math

import torch

from paper_2505_20776_b200 import api
from paper_2505_20776_b200.hotpath import HotPath

_WIDTH = 10                       # nodes per level of a draft tree


def _verify(name, layers, heads, prefix, capacity, nodes, chunk, top_k, draft):
    q, kv, dim = heads
    dl, dh, dd = draft
    return {"name": name, "kind": "verify", "layers": layers, "q_heads": q, "kv_heads": kv, "dim": dim,
            "prefix": prefix, "capacity": capacity, "nodes": nodes, "chunk": chunk, "top_k": top_k,
            "draft_layers": dl, "draft_heads": dh, "draft_dim": dd}


def _draft(name, layers, heads, nodes, capacity, tokens):
    q, kv, dim = heads
    return {"name": name, "kind": "draft", "layers": layers, "q_heads": q, "kv_heads": kv, "dim": dim,
            "nodes": nodes, "capacity": capacity, "tokens": tokens}


def _prefill(name, heads, tokens):
    q, kv, dim = heads
    return {"name": name, "kind": "prefill", "q_heads": q, "kv_heads": kv, "dim": dim, "tokens": tokens}


_GQA8B = (32, 8, 128)             # Llama-3.1-8B layer shape
_GQA70B = (64, 8, 128)            # 70B-class layer shape
_MHA = (32, 32, 128)              # one query head per KV head (Vicuna-7B layer shape)
_SMALL_DRAFT = (12, 12, 64)       # 68M-class draft model
_EAGLE_CACHE = (1, 8, 128)        # draft cache of one layer with the target's KV heads: layers, heads, dim
_SMALL_CACHE = (2, 12, 64)        # draft cache of a two-layer 68M-class model


def listed():
    return [
        # one drafting step of an EAGLE-class head (a level of 10 nodes) on a 1K working cache whose last chunk is short
        _draft("draft_eagle_1k", 1, _GQA8B, 10, 1024, 1012),
        # the same for a 68M-class two-layer draft model, single-token decoding after a level of its tree
        _draft("draft_small_1k", 2, _SMALL_DRAFT, 8, 1024, 1024),
        # a short conversation: four layers of the target at a ragged 1K prefix
        _verify("verify_1k", 4, _GQA8B, 1003, 2048, 60, 32, 32, _EAGLE_CACHE),
        # one scored layer and its retrieval at 4K
        _verify("verify_4k_scored", 1, _GQA8B, 4096, 4096, 60, 32, 32, _EAGLE_CACHE),
        # the first retrieval after a 16K prefill: the last prompt token alone looks for its chunks
        _verify("first_scores_16k", 1, _GQA8B, 16383, 16384, 1, 32, 32, _SMALL_CACHE),
        # a target without grouped heads at 8K, whose draft model is the two-layer one
        _verify("verify_mha_8k", 4, _MHA, 8201, 8448, 60, 32, 32, _SMALL_CACHE),
        # the whole verification step of the 8B-class target at 16K: 32 layers, each with its own cache
        _verify("verify_16k_32layers", 32, _GQA8B, 16384, 16384, 60, 32, 32, _EAGLE_CACHE),
        # a prefix growing in place inside a 32K buffer, at a ragged length
        _verify("verify_32k", 4, _GQA8B, 31337, 32768, 60, 32, 64, _EAGLE_CACHE),
        # the 70B-class target at 16K: 480 stacked rows per KV head, chunks of 64
        _verify("verify_70b_16k", 4, _GQA70B, 16384, 16384, 60, 64, 32, _EAGLE_CACHE),
        # the longest context: 128K, 4096 chunks to rank
        _verify("verify_128k", 2, _GQA8B, 131072, 131072, 60, 32, 64, _EAGLE_CACHE),
        # a short, ragged prompt
        _prefill("prefill_2k", _GQA8B, 1987),
        # a 16K prompt
        _prefill("prefill_16k", _GQA8B, 16384),
    ]


def _spread(rng, lo, hi):
    """A whole number, spread over the logarithm of the range."""
    return min(hi, max(lo, int(round(math.exp(rng.uniform(math.log(lo), math.log(hi)))))))


def draw(rng):
    """One more case of the same ranges, without a name."""
    kind = rng.choice(("verify", "verify", "verify", "verify", "draft", "draft", "prefill", "prefill"))
    if kind == "draft":
        heads = rng.choice((_GQA8B, _GQA8B, _SMALL_DRAFT, _MHA))
        capacity = rng.choice((16, 32, 48, 64)) * 32
        tokens = capacity - rng.choice((0, 0, rng.randint(1, 31)))
        c = _draft("", rng.choice((1, 1, 2)), heads, rng.choice((1, rng.randint(2, 20), rng.randint(20, 64))), capacity,
                   tokens)
    elif kind == "prefill":
        heads = rng.choice((_GQA8B, _GQA8B, _GQA70B, _MHA))
        c = _prefill("", heads, _spread(rng, 256, 16384 if heads[0] == 32 else 11500) - rng.randint(0, 9))
    else:
        heads = rng.choice((_GQA8B, _GQA8B, _GQA8B, _GQA70B, _MHA))
        prefix = _spread(rng, 256, 131072)
        if rng.random() < 0.7:
            prefix -= rng.randint(0, min(200, prefix // 2))            # ragged
        capacity = prefix + rng.choice((0, rng.randint(1, 1024)))
        nodes = rng.choice((1, rng.randint(2, 32), rng.randint(33, 64), 60, 60, rng.randint(65, 128)))
        layers = max(1, min(rng.choice((1, 1, 2, 4, 8)), int(1.2e9 / (capacity * heads[1] * heads[2] * 4))))
        c = _verify("", layers, heads, prefix, capacity, nodes, rng.choice((16, 32, 32, 64)), rng.choice((8, 16, 32, 32, 64)),
                    rng.choice((_EAGLE_CACHE, _SMALL_CACHE)))
    del c["name"]
    return c


# ---------------------------------------------------------------------------------------------------------
# inputs


def _levels(nodes):
    """How many tree keys each node sees: itself and one node of every level above."""
    return [i // _WIDTH + 1 for i in range(nodes)]


def _tree(nodes, gen, device):
    """parent[]: levels of 10 nodes, each node's parent anywhere in the level above (-1 = the last prefix token)."""
    i = torch.arange(nodes, device=device)
    pick = torch.randint(0, _WIDTH, (nodes,), generator=gen, device=device)
    return torch.where(i < _WIDTH, torch.full_like(i, -1), (i // _WIDTH - 1) * _WIDTH + pick).to(torch.int32)


def _randn(shape, gen, device):
    return torch.randn(shape, generator=gen, device=device, dtype=torch.bfloat16)


def _layer(c, length, gen, device, boost=None):
    """Q, cache and tree keys/values of one layer; `boost` (one value per cached token) raises the tokens' scores,
    as retrieval meets them: a few chunks of the context matter, the rest much less."""
    nodes, q, kv, dim = c["nodes"], c["q_heads"], c["kv_heads"], c["dim"]
    Q = _randn((nodes, q, dim), gen, device)
    K = _randn((length, kv, dim), gen, device)
    Kt = _randn((nodes, kv, dim), gen, device)
    if boost is not None:
        u = torch.nn.functional.normalize(torch.randn((kv, dim), generator=gen, device=device), dim=1)
        Q = (Q * dim ** -0.5 + 8 * u.repeat_interleave(q // kv, 0)).to(torch.bfloat16)
        Kt = Kt * dim ** -0.5
        K.mul_(dim ** -0.5)
        for lo in range(0, length, 16384):                            # in pieces: a long cache is a large tensor
            part = boost[lo:lo + 16384, None, None] * (u * (dim ** 0.5 / 8))
            K[lo:lo + 16384] = (K[lo:lo + 16384] + part).to(torch.bfloat16)
    return {"Q": Q, "K_prefix": K, "V_prefix": _randn((length, kv, dim), gen, device), "K_tree": Kt,
            "V_tree": _randn((nodes, kv, dim), gen, device)}


def prepare(case, seed):
    dev = torch.device("cuda", torch.cuda.current_device())
    gen = torch.Generator(device=dev)
    gen.manual_seed(seed)
    c = dict(case)
    s = {"case": c}
    if c["kind"] == "prefill":
        q, kv, dim, n = c["q_heads"], c["kv_heads"], c["dim"], c["tokens"]
        s["Q"], s["K"], s["V"] = (_randn((n, h, dim), gen, dev) for h in (q, kv, kv))
        s["O"] = torch.empty_like(s["Q"])
        s["lse"] = torch.empty((q, n), dtype=torch.float32, device=dev)
        s["status"] = torch.zeros(1, dtype=torch.int32, device=dev)
        return s
    nodes, layers = c["nodes"], c["layers"]
    s["parent"] = _tree(nodes, gen, dev)
    s["O"] = torch.empty((layers, nodes, c["q_heads"], c["dim"]), dtype=torch.bfloat16, device=dev)
    s["lse"] = torch.empty((layers, c["q_heads"], nodes), dtype=torch.float32, device=dev)
    if c["kind"] == "draft":
        s["layers"] = [_layer(c, c["capacity"], gen, dev) for _ in range(layers)]
        s["n_tokens"] = torch.full((1,), c["tokens"], dtype=torch.int32, device=dev)
        s["status"] = torch.zeros(1, dtype=torch.int32, device=dev)
        t = s["layers"][0]
        # the capacity never changes, so a program keeps the descriptor
        s["desc"] = api.make_attn_desc(t["Q"], t["K_prefix"], t["K_tree"], s["O"][0], c["capacity"], 32)
        s["ws"] = torch.empty(api.specext_verify_attn_workspace(s["desc"]), dtype=torch.uint8, device=dev)
        return s
    # which chunks matter: about 1.5 top_k of them are raised a little, top_k of those clearly, so that the ranking
    # is decided by the inputs and not by the rounding of a sum
    n_chunks = -(-c["prefix"] // c["chunk"])
    order = torch.randperm(n_chunks, generator=gen, device=dev)
    level = torch.rand(n_chunks, generator=gen, device=dev) * 0.4
    top = order[:c["top_k"]]
    level[top] = 1.0 + 2.0 * torch.rand(top.numel(), generator=gen, device=dev)
    boost = torch.zeros(c["capacity"], device=dev)
    boost[:c["prefix"]] = level.repeat_interleave(c["chunk"])[:c["prefix"]]
    s["layers"] = [_layer(c, c["capacity"], gen, dev, boost) for _ in range(layers)]
    s["hp"] = HotPath(c["q_heads"], c["kv_heads"], c["dim"], nodes, c["chunk"], c["top_k"], c["capacity"],
                      draft_layers=c["draft_layers"], draft_kv_heads=c["draft_heads"], draft_head_dim=c["draft_dim"],
                      device=dev)
    s["dK"], s["dV"] = (_randn((c["draft_layers"], c["capacity"], c["draft_heads"], c["draft_dim"]), gen, dev)
                        for _ in range(2))
    s["row"] = nodes * 5 // 8                                         # the last accepted node
    t = s["layers"][0]
    # the workspace of the layers without scores, at the cache's capacity: kept, as the HotPath keeps its own
    need = max(api.specext_verify_attn_workspace(
        api.make_attn_desc(t["Q"], t["K_prefix"], t["K_tree"], s["O"][0], n, c["chunk"])) for n in (c["capacity"], c["prefix"]))
    s["ws"] = torch.empty(need, dtype=torch.uint8, device=dev)
    return s


# ---------------------------------------------------------------------------------------------------------
# one pass


def run(s):
    c = s["case"]
    if c["kind"] == "prefill":
        api.specext_prefill_attn(s["Q"], s["K"], s["V"], s["O"], s["lse"], s["status"])
        return {"O": s["O"], "lse": s["lse"]}
    if c["kind"] == "draft":
        for i, t in enumerate(s["layers"]):
            api.specext_draft_attn(s["desc"], t["Q"], t["K_prefix"], t["V_prefix"], s["n_tokens"], t["K_tree"],
                                   t["V_tree"], s["parent"], s["O"][i], s["lse"][i], s["ws"], s["status"])
        return {"O": s["O"], "lse": s["lse"]}
    hp, L, last = s["hp"], c["prefix"], c["layers"] - 1
    if last > 0:
        # the prefix grows with every step, so the descriptor is made once per step
        t = s["layers"][0]
        desc = api.make_attn_desc(t["Q"], t["K_prefix"], t["K_tree"], s["O"][0], L, c["chunk"])
        for i in range(last):
            t = s["layers"][i]
            api.specext_verify_attn(desc, t["Q"], t["K_prefix"], t["V_prefix"], t["K_tree"], t["V_tree"], s["parent"],
                                    s["O"][i], s["lse"][i], None, s["ws"], hp.status)
    hp.verify_attn(s["layers"][last], s["parent"], L, True)
    hp.select_gather(s["row"], L, s["dK"], s["dV"])
    kept = min(c["top_k"], -(-L // c["chunk"]))
    return {"O": s["O"][:last], "lse": s["lse"][:last], "O_last": hp.O, "lse_last": hp.lse,
            "chunk_score": hp.chunk_score(L), "idx": hp.idx[:kept], "n_selected": hp.n_selected, "n_tokens": hp.n_tokens,
            "K_compact": hp.K_compact, "V_compact": hp.V_compact}


# ---------------------------------------------------------------------------------------------------------
# what a pass cannot do without, and how exact it is


def work(case):
    c = case
    q, kv, dim = c["q_heads"], c["kv_heads"], c["dim"]
    if c["kind"] == "prefill":
        n = c["tokens"]
        return {"bytes": 2 * n * dim * (2 * q + 2 * kv) + 4 * n * q, "flops": 4 * q * dim * (n * (n + 1) // 2)}
    nodes = c["nodes"]
    L = c["tokens"] if c["kind"] == "draft" else c["prefix"]
    per_layer = 4 * L * kv * dim + 4 * nodes * kv * dim + 4 * nodes * q * dim + 4 * q * nodes
    flops = c["layers"] * 4 * q * dim * (nodes * L + sum(_levels(nodes)))
    nbytes = c["layers"] * per_layer + 4 * nodes
    if c["kind"] == "verify":
        n_chunks = -(-L // c["chunk"])
        kept = min(c["top_k"], n_chunks)
        tokens = min(L, kept * c["chunk"])
        nbytes += 4 * nodes * n_chunks + 4 * n_chunks + 4 * kept + 8
        nbytes += 2 * 4 * tokens * c["draft_layers"] * c["draft_heads"] * c["draft_dim"]   # K and V, read and written
    return {"bytes": nbytes, "flops": flops}


def tolerance(case):
    """Outputs are bf16 sums of bf16-rounded probabilities: against fp64 the listed cases show rel up to 2.4e-3 and a
    largest error of 0.013 (of the root mean square or of the value); lse and scores show 2e-7.  Four times that."""
    return {"rel": 1e-2, "max": 0.05}
