"""Timed cases of the decode path: what a program that decodes images with relaxed speculative decoding has this library do.

Three kinds of case:

* ``step``     one speculative decode step on a static draft tree: the drafter's rows -> draft tokens (``sample_draft_tree``,
               over the whole tree at once or level by level as a drafter that feeds on its own tokens does) -> relaxed
               verification of every node and the walk (``verify_tree``).  Uniforms come from the library's own generator.
* ``dynamic``  one step with dynamic trees: ``expand_frontier`` per depth, ``trim_tree``, the drafted shapes read back, a
               ``Forest`` of them, and its verification with deterministic drafts.
* ``table``    the neighbour table of a codebook (``build_neighbors``), made once per codebook.

Logits are normal and the drafter's rows are noisy copies of the target's, so that some draft tokens are accepted and some
are not; codebooks are normal with 5 % exact copies in the table cases.
"""
import math
from fractions import Fraction
from itertools import product

import torch

import paper_2502_06352_b200 as L

DTYPES = {"f32": torch.float32, "bf16": torch.bfloat16}
FAN_OUT = {26: (4, 3, 2, 1, 1), 60: (4, 3, 3, 2, 2, 1, 1), 80: (4, 4, 3, 3, 2, 2, 1, 1)}   # largest number of children by depth


def step(name, batch, nodes, vocab, dtype, **more):
    case = dict(name=name, kind="step", batch=batch, nodes=nodes, vocab=vocab, dtype=dtype, guidance=0.0, temperature=1.0,
                top_k=0, std=1.5, mix=1.0, noise=0.5, codes=16384, dim=8, code_dtype="f32", offset=0, k=50, lam=2.0, delta=0.0,
                low=0, high=0, by_level=False, lazy=False)
    case.update(more)
    return case


def dynamic(name, batch, vocab, dtype, **more):
    case = dict(name=name, kind="dynamic", batch=batch, vocab=vocab, dtype=dtype, guidance=0.0, temperature=1.0, std=2.0,
                depths=6, children=8, expand=8, nodes=59, codes=8192, dim=256, code_dtype="bf16", offset=4096, k=100, lam=3.0)
    case.update(more)
    return case


def table(name, codes, dim, dtype, k):
    return dict(name=name, kind="table", codes=codes, dim=dim, dtype=dtype, k=k)


WIDE = dict(codes=8192, dim=256, code_dtype="bf16", offset=4096, k=100, lam=3.0)   # 65536 tokens, image tokens [4096, 12288)


def listed():
    return [
        # one image at a time, the drafter runs level by level: a handful of rows per call, latency and launches count
        step("one_image", 1, 26, 16384, "f32", guidance=7.5, by_level=True),
        # the same model serving 64 requests, rows of a whole tree known
        step("batched_images", 64, 26, 16384, "f32", guidance=7.5),
        # a mid-size batch with the usual top-k 1000 truncation and the extended tree
        step("top_k_1000", 8, 60, 16384, "f32", guidance=7.5, top_k=1000, std=1.2, k=100, lam=3.0),
        # a wide vocabulary of text and image tokens, all of it allowed
        step("wide_vocab", 4, 60, 65536, "f32", guidance=3.0, **WIDE),
        # the same model with its usual top-k 2000 truncation
        step("wide_top_k_2000", 4, 60, 65536, "f32", guidance=3.0, top_k=2000, **WIDE),
        # the same model inside an image: only the 8192 image tokens are allowed
        step("image_tokens_only", 4, 60, 65536, "f32", guidance=3.0, low=4096, high=12288, by_level=True, **WIDE),
        # offline generation at full batch: the largest call
        step("batch_64", 64, 80, 65536, "bf16", std=1.0, mix=0.7, noise=0.7, **dict(WIDE, k=200)),
        # sizes that divide nothing: another tokenizer, a pruned tree, an odd batch, the additive bound
        step("ragged", 5, 43, 40003, "bf16", guidance=4.0, temperature=0.9, delta=0.05, codes=10007, dim=24,
             code_dtype="bf16", offset=1, k=37),
        # dynamic trees for a full batch: six depths, trimmed to 59 nodes, every sequence its own shape
        dynamic("dynamic_trees", 64, 65536, "bf16"),
        # codebooks as they are met: small float codes, wide bfloat16 codes, and a large codebook
        table("table_16384x8", 16384, 8, "f32", 100),
        table("table_8192x256", 8192, 256, "bf16", 200),
        table("table_65536x256", 65536, 256, "bf16", 200),
    ]


def log_between(rng, low, high):
    return int(round(math.exp(rng.uniform(math.log(low), math.log(high)))))


def draw(rng):
    kind = rng.choice(["step", "step", "step", "step", "dynamic", "table"])
    if kind == "table":
        codes, dim, dtype = log_between(rng, 2048, 65536), rng.choice([8, 12, 16, 32, 64, 100, 256]), rng.choice(["bf16", "bf16", "f32"])
        if dtype == "f32" or dim % 8:       # exact distances of every pair: large tables of these take seconds
            codes, dim = min(codes, 20000), min(dim, 64)
        return table("", codes, dim, dtype, log_between(rng, 8, 200)) | {"name": "table_drawn"}
    vocab = rng.choice([4096, 16384, 65536, log_between(rng, 4000, 70000)])
    dtype = rng.choice(["f32", "bf16"])
    guidance = rng.choice([0.0, 3.0, 7.5, round(rng.uniform(1.5, 9.0), 2)])
    size = (4 if dtype == "f32" else 2) * (2 if guidance else 1)
    room = 600e6 / (vocab * size)           # rows that fit 600 MB on either side
    codes = rng.choice([1024, 4096, 8192, log_between(rng, 500, 9000)])
    codes = min(codes, vocab - 64)
    shared = dict(guidance=guidance, temperature=rng.choice([1.0, 1.0, 0.8, 1.2]), codes=codes, dim=rng.choice([8, 16, 64]),
                  code_dtype="bf16", offset=rng.choice([0, vocab - codes - 3]), k=rng.choice([10, 37, 100, 200]), lam=rng.choice([2.0, 3.0, 5.0]))
    if kind == "dynamic":
        depths, children, expand = rng.randint(3, 7), rng.choice([4, 6, 8]), rng.choice([4, 8, 10])
        nodes = rng.randint(20, 60)
        batch = max(1, min(log_between(rng, 1, 64), int(room / max(nodes, depths * expand))))
        return dynamic("dynamic_drawn", batch, vocab, dtype, **dict(shared, std=rng.choice([1.0, 2.0, 4.0]), depths=depths,
                                                                    children=children, expand=expand, nodes=nodes))
    nodes = rng.choice([26, 60, 80, rng.randint(12, 90)])
    batch = max(1, min(log_between(rng, 1, 64), int(room / nodes)))
    low, high = rng.choice([(0, 0), (0, 0), (shared["offset"], shared["offset"] + codes)])
    top_k = rng.choice([0, 0, 0, 1000, 2000, rng.randint(50, 2000)])
    top_k = 0 if vocab > 16384 and batch * nodes > 500 else top_k
    return step("step_drawn", batch, nodes, vocab, dtype, **dict(
        shared, std=rng.choice([1.0, 1.2, 1.5]), mix=rng.choice([0.7, 1.0]), noise=rng.choice([0.3, 0.5, 0.7]),
        top_k=top_k if not high or top_k < high - low else 0, delta=rng.choice([0.0, 0.0, 0.05]), low=low, high=high,
        by_level=rng.random() < 0.5, lazy=rng.random() < 0.15))


def tree_of(nodes):
    """A static tree that leans to the left: the `nodes` heaviest rank paths, weight (2/3)^depth * (1/2)^(sum of ranks), breadth first."""
    caps = FAN_OUT.get(nodes, (4, 4, 3, 3, 2, 2, 1, 1))
    paths = [(Fraction(2, 3) ** d * Fraction(1, 2) ** sum(p), p)
             for d in range(1, len(caps) + 1) for p in product(*[range(c) for c in caps[:d]])]
    paths.sort(key=lambda wp: (-wp[0], len(wp[1]), wp[1]))
    number, parent = {(): 0}, [-1]
    for p in sorted((p for _, p in paths[: nodes - 1]), key=lambda p: (len(p), p)):
        number[p] = len(parent)
        parent.append(number[p[:-1]])
    return parent


def levels_of(parent):
    """[begin, end) of the parents that one call of a level-by-level drafter expands, for each level."""
    depth = [0]
    for p in parent[1:]:
        depth.append(depth[p] + 1)
    return [(depth.index(d), depth.index(d) + depth.count(d)) for d in range(max(depth))]


def normal(gen, shape, std):
    return torch.randn(shape, generator=gen, device="cuda") * std


def rows_like(x, dtype):
    """[B][N][V] rows in `dtype`, each starting on a 16-byte boundary as a serving program lays them out."""
    B, N, V = x.shape
    out = torch.empty((B, N, -(-V // 8) * 8), dtype=dtype, device="cuda")[:, :, :V]
    out.copy_(x)
    return out


def codebook(gen, codes, dim, dtype, copies=0.0):
    cb = normal(gen, (codes, dim), 1.0)
    n = int(codes * copies)
    if n:
        order = torch.randperm(codes, generator=gen, device="cuda")
        cb[order[:n]] = cb[order[n:2 * n]]
    return cb.to(DTYPES[dtype])


def prepare(case, seed):
    gen = torch.Generator(device="cuda")
    gen.manual_seed(seed)
    if case["kind"] == "table":
        return dict(case=case, codebook=codebook(gen, case["codes"], case["dim"], case["dtype"], 0.05))
    dt, B, V = DTYPES[case["dtype"]], case["batch"], case["vocab"]
    s = dict(case=case, table=L.build_neighbors(codebook(gen, case["codes"], case["dim"], case["code_dtype"]), case["k"]))
    s["params"] = L.Params(vocab=V, cfg_scale=case["guidance"] or 1.0, temperature=case["temperature"], lam=case["lam"], k=case["k"],
                           code_offset=case["offset"], n_codes=case["codes"], seed=seed, step=1)
    sides = ("cond", "uncond") if case["guidance"] else ("cond",)
    if case["kind"] == "dynamic":
        s["params"].draft_deterministic = 1
        for side in sides:
            widths = [1] + [case["expand"]] * (case["depths"] - 1)
            s["draft_" + side] = [rows_like(normal(gen, (B, f, V), case["std"]), dt) for f in widths]
            s["target_" + side] = rows_like(normal(gen, (B, case["nodes"], V), case["std"]), dt)
        return s
    p = s["params"]
    p.top_k_target = p.top_k_draft = case["top_k"]
    p.delta, p.allowed_begin, p.allowed_end, p.lazy_walk = case["delta"], case["low"], case["high"], int(case["lazy"])
    parent = tree_of(case["nodes"])
    N = len(parent)
    s["tree"] = L.Tree(parent)
    s["levels"] = levels_of(parent) if case["by_level"] else [(0, N)]
    for side in sides:
        x = normal(gen, (B, N, V), case["std"])
        s["target_" + side] = rows_like(x, dt)
        s["draft_" + side] = rows_like(x * case["mix"] + normal(gen, (B, N, V), case["noise"]), dt)
    # buffers that a decode loop keeps
    s["tokens"] = torch.zeros((B, N), dtype=torch.int32, device="cuda")
    s["out"] = {}
    s["workspace"] = torch.empty(L.binding.lib.lantern_verify_tree_workspace(s["tree"].handle, B), dtype=torch.uint8, device="cuda")
    return s


def run(s):
    case = s["case"]
    if case["kind"] == "table":
        return L.build_neighbors(s["codebook"], case["k"], return_dist=True)
    if case["kind"] == "dynamic":
        return run_dynamic(s, case)
    for begin, end in s["levels"]:
        L.sample_draft_tree(s["params"], s["tree"], s["draft_cond"], s.get("draft_uncond"), tokens=s["tokens"],
                            parent_begin=begin, parent_end=end)
    # per-node results (acceptance statistics by depth) are asked for wherever every node is verified
    out = L.verify_tree(s["params"], s["tree"], s["table"], s["target_cond"], s.get("target_uncond"), s["draft_cond"],
                        s.get("draft_uncond"), s["tokens"], out=s["out"], debug=not case["lazy"], workspace=s["workspace"])
    return dict(out, tokens=s["tokens"])


def run_dynamic(s, case):
    pool = L.DraftPool(case["batch"], case["depths"], case["children"], case["expand"])
    for depth in range(case["depths"]):
        L.expand_frontier(s["params"], pool, s["draft_cond"][depth], s["draft_uncond"][depth] if case["guidance"] else None)
    n, parent, tokens, index, logv = L.trim_tree(pool, case["nodes"])
    forest = L.Forest(parent.tolist(), n.tolist(), case["nodes"])
    out = L.verify_tree(s["params"], forest, s["table"], s["target_cond"], s.get("target_uncond"), None, None, tokens, debug=True)
    for name in ("out_tokens", "out_nodes"):     # as wide as the deepest tree: the decode loop keeps one column per depth
        out[name] = torch.nn.functional.pad(out[name], (0, case["depths"] + 1 - out[name].shape[1]), value=-1)
    return dict(out, n_nodes=n, parent=parent, tokens=tokens, pool_index=index, logv=logv)


def work(case):
    """Every row once; per tested child its table row; per node its results.  Tables: codebook in, indices and distances out."""
    if case["kind"] == "table":
        n, d = case["codes"], case["dim"]
        return {"bytes": n * d * (4 if case["dtype"] == "f32" else 2) + 8 * n * case["k"], "flops": 2.0 * n * n * d}
    span = (case.get("high") or case["vocab"]) - (case.get("low") or 0)
    row = span * (4 if case["dtype"] == "f32" else 2) * (2 if case["guidance"] else 1)
    B, N = case["batch"], case["nodes"]
    if case["kind"] == "dynamic":
        rows = B * (1 + case["expand"] * (case["depths"] - 1)) + B * N
        return {"bytes": rows * row + B * (N - 1) * case["k"] * 4 + 40 * B * N, "flops": 4.0 * rows * span}
    parent = tree_of(N)
    inner = len(set(parent[1:]))
    if case["lazy"]:     # only the rows on the accepted path: at least the root's
        return {"bytes": B * (inner + 2) * row, "flops": 4.0 * B * (inner + 2) * span}
    rows = B * (N + 2 * inner)      # target rows, and the drafter's rows by the sampler and by verification
    return {"bytes": rows * row + B * (N - 1) * case["k"] * 4 + 20 * B * N, "flops": 4.0 * rows * span}


def tolerance(case):
    """Masses, acceptance probabilities and softmax denominators are float32 sums, and a token drawn by inverse CDF moves to
    its neighbour where the uniform lies within their rounding of a boundary.  About four times what 20 seeds showed between
    rows summed by one, four and eight thread blocks: 3.5e-6 overall, 1.2e-4 for one value (a residual mass after
    cancellation), 2.3e-3 of the drawn tokens.  Tables are ranked by exact distances: their indices agree."""
    if case["kind"] == "table":
        return {"rel": 1e-6, "max": 4e-6}
    return {"rel": 1.5e-5, "max": 5e-4, "differ": 8e-3}
