"""Parity of lantern_sample_draft_tree with the oracle (Sec. 2.1: s tokens per node drawn from
p, read as Gumbel-top-s without replacement)."""
import numpy as np
import pytest
import torch

import oracle
import workloads as W
from gpu_cases import Case, f64, small_config
from parity_util import KEY_TIE

pytestmark = pytest.mark.gpu


@pytest.fixture(scope="module")
def L():
    import paper_2502_06352_b200 as lib
    return lib


def _gpu_sample(L, case, gumbel=None, seed_step=None, parent_range=(0, None), tokens=None):
    g, par, _, _ = case.gpu_inputs(L)
    tree = L.Tree(case.parent)
    if seed_step:
        par.seed, par.step = seed_step
    prob = torch.zeros((case.B, case.N), dtype=torch.float32, device="cuda")
    status = torch.zeros(1, dtype=torch.int32, device="cuda")
    tok = L.sample_draft_tree(par, tree, g["draft_cond"], g["draft_uncond"], tokens=tokens,
                              parent_begin=parent_range[0], parent_end=parent_range[1],
                              gumbel_uniforms=None if gumbel is None else gumbel.cuda(), draft_prob=prob,
                              device_status=status)
    torch.cuda.synchronize()
    assert int(status.item()) == 0
    return tok.cpu().numpy(), prob.cpu().numpy(), tok


def _compare(case, gum, gtok, gprob):
    kids = oracle.tree_children(case.parent)
    ties = 0
    for b in range(case.B):
        du = case.logits["draft_uncond"]
        for n in range(case.N):
            if not kids[n]:
                continue
            p, _ = oracle.postprocess_row(f64(case.logits["draft_cond"][b, n]), None if du is None else f64(du[b, n]),
                                          case.params["cfg_scale"], case.params["temperature"],
                                          case.params["top_k_draft"], case.params["allowed_begin"],
                                          case.params["allowed_end"])
            want, wp, gaps = oracle.sample_children(p, gum[b, n], len(kids[n]), return_gaps=True)
            got = [int(gtok[b, c]) for c in kids[n]]
            if got != want:
                r = next(i for i in range(len(want)) if got[i] != want[i])
                assert min(gaps[max(0, r - 1): r + 1]) < KEY_TIE, ("sampler mismatch", b, n, got, want, gaps)
                ties += 1
                continue
            assert np.allclose(gprob[b, kids[n]], wp, atol=1e-5)
            real = [t for t in got if t >= 0]
            assert len(set(real)) == len(real)
    return ties


@pytest.mark.parametrize("kw", [dict(), dict(cfg_scale=None), dict(top_k=20), dict(dtype="bf16", cfg_scale=None),
                                dict(vocab=1003, codebook_size=1003), dict(n_nodes=60, temperature=0.8)])
@pytest.mark.parametrize("kernels", [1, 2])          # streaming kernel forced / excluded
def test_explicit_uniforms(L, kw, kernels):
    pad = 5 if kw.get("vocab") == 1003 else 0
    case = Case(small_config(**kw), seed=21, tokens="random", pad=pad, kernels=kernels)
    gum = W.make_gumbel_uniforms(case.B, case.N, case.V, 1234)
    gtok, gprob, _ = _gpu_sample(L, case, gumbel=gum)
    assert _compare(case, gum.numpy(), gtok, gprob) <= 1
    assert np.all(gtok[:, 0] == -1)


@pytest.mark.parametrize("cs", [1, 2, 8])
def test_cluster_sizes_and_allowed_range(L, cs):
    case = Case(small_config(vocab=2048, codebook_size=512, code_offset=256, top_k=30), seed=22,
                tokens="random", allowed=(256, 768))
    gum = W.make_gumbel_uniforms(case.B, case.N, case.V, 99)
    old = L.set_cluster_size(cs)
    try:
        gtok, gprob, _ = _gpu_sample(L, case, gumbel=gum)
    finally:
        L.set_cluster_size(old)
    assert _compare(case, gum.numpy(), gtok, gprob) <= 1
    assert np.all((gtok[:, 1:] >= 256) & (gtok[:, 1:] < 768))


@pytest.mark.parametrize("cs", [0, 1])
@pytest.mark.parametrize("kw", [dict(vocab=3001, codebook_size=3001, top_k=200),
                                dict(vocab=9000, codebook_size=2000, top_k=1000, dtype="bf16", cfg_scale=None)])
def test_topk_rows_list_and_dense_kernels(L, cs, kw):
    # cs = 0: the list-based kernel; cs = 1: the dense kernel.  Philox uniforms, so the list kernel
    # has to pick the right word of each token's counter block.
    case = Case(small_config(**kw), seed=25, tokens="random", pad=3 if kw.get("dtype", "f32") == "f32" else 8)
    seed, step = 0x5EED, 11
    gum = np.empty((case.B, case.N, case.V), dtype=np.float32)
    for b in range(case.B):
        for n in range(case.N):
            gum[b, n] = oracle.stream_uniforms(seed, step, b * case.N + n, 0, count=case.V)
    old = L.set_cluster_size(cs)
    try:
        gtok, gprob, _ = _gpu_sample(L, case, seed_step=(seed, step))
    finally:
        L.set_cluster_size(old)
    assert _compare(case, gum, gtok, gprob) <= 1


def test_topk_with_massive_ties_is_redrawn_by_the_dense_kernel(L):
    # logits on a grid of 2.0: the k-th largest value is shared by more entries than the list
    # kernel holds, so it marks every parent and the dense kernel draws them
    case = Case(small_config(vocab=8000, codebook_size=1000, top_k=300, cfg_scale=None, batch=2), seed=26,
                tokens="random")
    for v in case.padded.values():
        if v is not None:
            v.copy_(torch.round(v / 2.0) * 2.0)
    gum = W.make_gumbel_uniforms(case.B, case.N, case.V, 77)
    gtok, gprob, _ = _gpu_sample(L, case, gumbel=gum)
    assert _compare(case, gum.numpy(), gtok, gprob) <= 1
    assert np.all(gtok[:, 1:] >= 0)


def test_philox_uniforms_and_level_by_level(L):
    case = Case(small_config(batch=2), seed=23, tokens="random")
    seed, step = 0xABCDEF12345, 7
    gum = np.empty((case.B, case.N, case.V), dtype=np.float32)
    for b in range(case.B):
        for n in range(case.N):
            gum[b, n] = oracle.stream_uniforms(seed, step, b * case.N + n, 0, count=case.V)
    gtok, gprob, _ = _gpu_sample(L, case, seed_step=(seed, step))
    assert _compare(case, gum, gtok, gprob) <= 1
    # expanding one level at a time fills the same tokens
    depth = [0] * case.N
    for i in range(1, case.N):
        depth[i] = depth[case.parent[i]] + 1
    tok = None
    for d in range(max(depth) + 1):
        ids = [i for i in range(case.N) if depth[i] == d]
        _, _, tok = _gpu_sample(L, case, seed_step=(seed, step), parent_range=(ids[0], ids[-1] + 1), tokens=tok)
    assert np.array_equal(tok.cpu().numpy(), gtok)


def test_small_support_gives_minus_one(L):
    # only 2 allowed tokens but 4 children at the root
    case = Case(small_config(batch=1), seed=24, tokens="random", allowed=(10, 12))
    gum = W.make_gumbel_uniforms(case.B, case.N, case.V, 5)
    gtok, gprob, _ = _gpu_sample(L, case, gumbel=gum)
    kids = oracle.tree_children(case.parent)
    root = [int(gtok[0, c]) for c in kids[0]]
    assert sorted(root[:2]) == [10, 11] and root[2:] == [-1] * (len(root) - 2)
    assert _compare(case, gum.numpy(), gtok, gprob) == 0


def test_first_child_follows_p_chi_square(L):
    """V = 16: over many independent rows the first child is distributed as p (Philox path)."""
    V, B = 16, 4096
    cfg = small_config(vocab=V, codebook_size=V, batch=B, cfg_scale=None, k=0)
    parent = [-1, 0, 0]
    row = torch.randn(V, generator=torch.Generator().manual_seed(3)) * 1.2
    logits = row.repeat(B, 3, 1).contiguous().cuda()
    tree = L.Tree(parent)
    par = L.Params(vocab=V, seed=77, step=1)
    counts = np.zeros(V)
    pair = {}
    for step in range(8):
        par.step = step
        tok = L.sample_draft_tree(par, tree, logits, None).cpu().numpy()
        counts += np.bincount(tok[:, 1], minlength=V)
        assert np.all(tok[:, 1] != tok[:, 2])
    p = torch.softmax(row.double(), 0).numpy()
    n = counts.sum()
    chi2 = ((counts - n * p) ** 2 / (n * p)).sum()
    assert chi2 < 44.3       # 15 dof, p ~ 1e-4


@pytest.mark.parametrize("seed", [0, 1, 2, 3])
@pytest.mark.parametrize("kw", [dict(vocab=65536, codebook_size=1024, dtype="bf16", cfg_scale=None),
                                dict(vocab=16384, codebook_size=1024, temperature=0.7),
                                dict(vocab=5000, codebook_size=1024, n_nodes=26, cfg_scale=None)])
def test_streaming_kernel_over_seeds_and_row_shapes(L, seed, kw):
    """The streaming sampler (forced) on rows of the benchmark's width and smaller, several seeds: first
    threshold from the warps' best keys, the scheduled cut, the exact ranking."""
    case = Case(small_config(batch=2, **kw), seed=100 + seed, tokens="random", kernels=1)
    gum = W.make_gumbel_uniforms(case.B, case.N, case.V, 4321 + seed)
    gtok, gprob, _ = _gpu_sample(L, case, gumbel=gum)
    assert _compare(case, gum.numpy(), gtok, gprob) <= 1


@pytest.mark.parametrize("shape", ["rising", "falling", "flat"])
def test_streaming_kernel_on_monotone_and_constant_rows(L, shape):
    """Rows whose logits rise along the row keep producing keys above every earlier threshold (the candidate
    list overflows and the row is redone with a cut after every chunk); falling rows never do; constant rows
    leave everything to the uniforms.  All must agree with the oracle."""
    case = Case(small_config(batch=2, vocab=65536, codebook_size=1024, dtype="f32", cfg_scale=None), seed=77,
                tokens="random", kernels=1)
    V = case.V
    ramp = torch.linspace(-30.0, 30.0, V)
    row = {"rising": ramp, "falling": ramp.flip(0), "flat": torch.zeros(V)}[shape]
    case.padded["draft_cond"][:, :, :V] = row
    gum = W.make_gumbel_uniforms(case.B, case.N, V, 99)
    gtok, gprob, _ = _gpu_sample(L, case, gumbel=gum)
    assert _compare(case, gum.numpy(), gtok, gprob) <= 1


@pytest.mark.parametrize("kw", [dict(vocab=4096, codebook_size=512), dict(vocab=4099, codebook_size=512, cfg_scale=None),
                                dict(vocab=16384, codebook_size=512, batch=1, parent=[-1, 0]),
                                dict(vocab=20011, codebook_size=512, dtype="bf16"),
                                dict(vocab=65536, codebook_size=512, dtype="bf16", batch=1, parent=[-1, 0, 0, 0, 1], allowed=(4097, 12290)),
                                dict(vocab=33000, codebook_size=512, batch=1, parent=[-1, 0, 0, 0, 1], allowed=(32990, 33000))])
@pytest.mark.parametrize("philox", [False, True])
def test_small_calls_on_the_streaming_kernel(L, kw, philox):
    """What the library picks by itself for a handful of parents: rows that are one chunk per CTA and rows of several,
    clusters of up to eight CTAs, allowed ranges that no vector divides and one narrower than a vector per warp."""
    kw = dict(kw)
    allowed, parent = kw.pop("allowed", (0, 0)), kw.pop("parent", None)
    V = kw["vocab"]
    case = Case(small_config(**kw), parent=parent, seed=31, tokens="random", allowed=allowed, kernels=0, pad=-V % 8)
    if philox:
        seed, step = 0xBEEF, 5
        gum = np.empty((case.B, case.N, V), dtype=np.float32)
        for b in range(case.B):
            for n in range(case.N):
                gum[b, n] = oracle.stream_uniforms(seed, step, b * case.N + n, 0, count=V)
        gtok, gprob, _ = _gpu_sample(L, case, seed_step=(seed, step))
    else:
        gum = W.make_gumbel_uniforms(case.B, case.N, V, 4242).numpy()
        gtok, gprob, _ = _gpu_sample(L, case, gumbel=torch.from_numpy(gum))
    assert _compare(case, gum, gtok, gprob) <= 1


@pytest.mark.parametrize("dtype", ["f32", "bf16"])
def test_streaming_kernel_on_wide_ranges_and_nearly_empty_rows(L, dtype):
    """Logits from -250 to 250 (the exponential of the elements' test overflows and vanishes), and rows of which all
    but two elements are -inf: fewer candidates than children."""
    case = Case(small_config(batch=2, vocab=20000, codebook_size=512, dtype=dtype, cfg_scale=None), seed=41, tokens="random", kernels=1)
    rows = case.padded["draft_cond"]
    g = torch.Generator().manual_seed(6)
    rows[0] = ((torch.rand(rows[0].shape, generator=g) * 500.0) - 250.0).to(rows.dtype)
    rows[1] = -float("inf")
    rows[1, :, 17] = 1.0
    rows[1, :, 19999] = 0.5
    gum = W.make_gumbel_uniforms(case.B, case.N, case.V, 7)
    gtok, gprob, _ = _gpu_sample(L, case, gumbel=gum)
    assert _compare(case, gum.numpy(), gtok, gprob) <= 1


@pytest.mark.parametrize("kw", [dict(vocab=16385, codebook_size=500, top_k=50), dict(vocab=20001, codebook_size=500, top_k=2048, cfg_scale=None),
                                dict(vocab=65536, codebook_size=500, top_k=2000, dtype="bf16"), dict(vocab=4096, codebook_size=500, top_k=6),
                                dict(vocab=33000, codebook_size=500, top_k=1000, allowed=(4099, 12290)),
                                dict(vocab=33000, codebook_size=500, top_k=300, allowed=(32001, 32100))])
def test_topk_rows_of_every_width(L, kw):
    kw = dict(kw)
    allowed = kw.pop("allowed", (0, 0))
    case = Case(small_config(batch=1, **kw), seed=33, tokens="random", allowed=allowed, pad=-kw["vocab"] % 8)
    gum = W.make_gumbel_uniforms(case.B, case.N, case.V, 515)
    gtok, gprob, _ = _gpu_sample(L, case, gumbel=gum)
    assert _compare(case, gum.numpy(), gtok, gprob) <= 1
    again, prob, _ = _gpu_sample(L, case, gumbel=gum)
    assert np.array_equal(again, gtok) and np.array_equal(prob, gprob)          # bit for bit


@pytest.mark.parametrize("V,cs", [(4096, 0), (16384, 0), (65536, 1)])       # one chunk per CTA; the same on a cluster; sixteen chunks
@pytest.mark.parametrize("dtype", ["f32", "bf16"])
def test_supplied_uniforms_of_any_size_are_used_as_given(L, V, cs, dtype):
    """Uniforms that no 2^-23 grid holds, down to the smallest float32, on a token that dominates its row, at the row's
    start and far behind it; a second token's key lies 1e-3 above or below, so that a key that is off by more shows."""
    us = [2.0 ** -24, 1e-8, 1e-7, 1e-6, 1e-5, 3e-5, 1e-30, 1e-42, 1.0 - 2.0 ** -24]
    parent = [-1] + [0] * 4
    kw = dict(vocab=V, codebook_size=512, batch=2 * len(us), dtype=dtype, cfg_scale=None)
    case = Case(small_config(**kw), parent=parent, seed=61, tokens="random", kernels=1)
    gum = W.make_gumbel_uniforms(case.B, case.N, V, 17)
    rows = case.padded["draft_cond"]
    for i, u in enumerate(us):
        for j in range(2):
            b = 2 * i + j
            a = 5 if j == 0 else V - 99
            gum[b, 0, a] = u
            rows[b, 0, a] = 40.0
            key = float(rows[b, 0, a].float()) - np.log(-np.log(np.float64(gum[b, 0, a].item())))
            t = (a + 1234) % V                         # a token of the same height whose uniform puts its key beside that one
            rows[b, 0, t] = rows[b, 0, a]
            for step in (1e-3, -1e-3):
                want = np.exp(-np.exp(-(key + step - float(rows[b, 0, t].float()))))
                if 0.0 < np.float32(want) < 1.0:
                    gum[b, 0, t] = float(np.float32(want))
                    break
    old = L.set_cluster_size(cs)
    try:
        gtok, gprob, _ = _gpu_sample(L, case, gumbel=gum)
    finally:
        L.set_cluster_size(old)
    assert _compare(case, gum.numpy(), gtok, gprob) == 0
    dominant = [5 if b % 2 == 0 else V - 99 for b in range(case.B)]
    assert all(dominant[b] in gtok[b, 1:] for b in range(case.B))


@pytest.mark.parametrize("z", [20000.0, -300000.0])
def test_large_logits_are_ordered_by_exact_keys(L, z):
    """Logits so large that a float32 step (2e-3, 3e-2) is far above the keys' own error: two tokens of different heights whose
    float32 keys z + G + ln(ln 2) round to different sides of a half step, 1e-7 apart, so that they are a whole step apart and
    say nothing about the order.  (The kept candidates' order is that of keys in double precision, so no near-tie is excused.)"""
    V, B, parent = 4096, 512, [-1, 0, 0]
    case = Case(small_config(vocab=V, codebook_size=512, batch=B, n_nodes=3, cfg_scale=None, k=0), parent=parent, seed=62, tokens="random", kernels=1)
    rng = np.random.default_rng(12)
    step = abs(float(np.spacing(np.float32(z))))
    case.padded["draft_cond"][:] = z - 60.0 * max(1.0, step)
    gum = W.make_gumbel_uniforms(B, case.N, V, 18)
    pair = {}
    for b in range(B):
        edge = -(round(0.5 * rng.random() / step) + 0.5) * step - float(np.log(np.log(2.0)))
        t = rng.choice(V, 2, replace=False)
        lower = int(rng.integers(1, max(2, round(0.6 / step)))) * step          # the second token's logit, in whole steps
        key = []
        for i, (below, off) in enumerate(((0.0, -5e-8), (lower, 5e-8))):
            gum[b, 0, t[i]] = float(np.float32(np.exp(-np.exp(-(edge + below + off)))))
            case.padded["draft_cond"][b, 0, t[i]] = z - below
            key.append(-below - np.log(-np.log(float(gum[b, 0, t[i]]))))
        if abs(key[0] - key[1]) > 1e-9:
            pair[b] = [int(x) for x in (t if key[0] > key[1] else t[::-1])]
    assert len(pair) > B // 2
    g, par, _, _ = case.gpu_inputs(L)
    tok = L.sample_draft_tree(par, L.Tree(case.parent), g["draft_cond"], None, gumbel_uniforms=gum.cuda()).cpu().numpy()
    for b, want in pair.items():
        assert [int(tok[b, c]) for c in (1, 2)] == want, b
