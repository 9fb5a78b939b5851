"""What is measured: the work that a program using this package has it do, through the public entry points.

A case is a dict of plain sizes and options; ``kind`` says which part of the retrieve-and-verify step it is:

  draft    fc_retrieve on two stores and fc_build_tree over what it found: the drafting half of a step.  A step calls it
           once per generated batch of tokens, at batch 1 (one user) up to a few hundred.
  build    fc_datastore_build of a token corpus with its suffix keys: done when a repository is opened (a project store)
           or a general corpus is indexed.
  attn     fc_tree_attn over a filled KV cache: the verification attention of one layer.
  mlp      fc_add_rmsnorm, fc_gemm_silu_mul, fc_gemm_bf16: the MLP block of one decoder layer over the draft tree's rows.
  head     fc_add_rmsnorm, the LM head GEMM, fc_argmax_accept: from the last layer to the accepted tokens.
  decoder  TreeDecoder.forward: a whole verification forward (every layer: norms, projections, RoPE, attention, MLP, head).
  loop     PipelinedStepLoop: several whole steps (retrieval, tree, attention, acceptance, cache append), from the start
           of a generation; with the replay cache or, ``alg1``, with the CACHE and the missing table of Algorithm 1.

Sizes follow synth.WORKLOADS, the decoder shapes of decoder.py and the tests.  Ragged lengths come from the case alone
(so its work is known), values from the seed.
"""
import math

import numpy as np
import torch

import paper_2502_17139_gb300.fastcoder as fc
import paper_2502_17139_gb300.synth as synth
from paper_2502_17139_gb300.decoder import DecoderShape, TreeDecoder
from paper_2502_17139_gb300.step import PipelinedStepLoop

DEV = "cuda"
VOCAB = synth.VOCAB
D = 128
BF = torch.bfloat16


def listed():
    return [
        # one user, a store of a mid-size repository and a common one: every kernel is a latency chain
        dict(name="draft_b1", kind="draft", B=1, n_general=5_000_000, n_project=300_001, n_max=16, k=64, d=10, budget=64, n_pad=64),
        # the two-source workload at its full size: 100M + 5M tokens, 256 contexts
        dict(name="draft_b256", kind="draft", B=256, n_general=100_000_000, n_project=5_000_000, n_max=16, k=64, d=10, budget=64, n_pad=64),
        # a repository's own store, indexed when it is opened
        dict(name="build_1m", kind="build", n=1_000_003, zipf=1.3),
        # the general store
        dict(name="build_100m", kind="build", n=100_000_000, zipf=1.1),
        # the paper's own setting: batch 1, inputs of up to 2k tokens, a 7B-shaped layer
        dict(name="attn_b1", kind="attn", B=1, H=32, Hkv=32, kv=2311, n_pad=64),
        # a few users with long repository contexts, grouped heads
        dict(name="attn_b4_long", kind="attn", B=4, H=32, Hkv=8, kv=16384, n_pad=64),
        # a 7B-shaped layer at a serving batch
        dict(name="attn_b16", kind="attn", B=16, H=32, Hkv=32, kv=4096, n_pad=64),
        # the step loop's own attention: grouped heads, long caches, trees of up to 128 nodes
        dict(name="attn_b32_long", kind="attn", B=32, H=32, Hkv=8, kv=16384, n_pad=128),
        # the MLP of a 1.3B-shaped layer for one user's draft tree: the weights are read for 64 rows
        dict(name="mlp_b1", kind="mlp", B=1, n_pad=64, hidden=2048, inter=5504),
        # final norm, LM head and acceptance at a serving batch
        dict(name="head_b32", kind="head", B=32, n_pad=64, hidden=2048),
        # a whole verification forward for one user: eight layers of the 1.3B shape (each more layer repeats the same work, and
        # bf16 roundings of the first spread through all that follow)
        dict(name="decoder_b1", kind="decoder", B=1, n_pad=64, hidden=2048, layers=8, H=16, Hkv=16, inter=5504, kv=2048),
        # the whole step loop at its serving size: two stores, 32 sequences, 16k-token caches, four sub-batches
        dict(name="loop_b32", kind="loop", B=32, n_split=4, steps=8, n_general=100_000_000, n_project=5_000_000, n_max=16, k=64, d=10,
             budget=128, n_pad=128, H=32, Hkv=8, kv=16384, alg1=False),
    ]


def _log(rng, lo, hi):
    return int(round(math.exp(rng.uniform(math.log(lo), math.log(hi)))))


def draw(rng):
    kind = rng.choice(["draft", "build", "attn", "attn", "mlp", "head", "decoder", "loop"])
    n_pad = rng.choice([64, 128])
    if kind == "draft":
        k = rng.choice([16, 64])
        return dict(kind=kind, B=_log(rng, 1, 256), n_general=_log(rng, 300_000, 50_000_000), n_project=_log(rng, 50_000, 5_000_000),
                    n_max=rng.choice([16, 24]), k=k, d=rng.choice([8, 10, 12]), budget=rng.randint(n_pad // 2, n_pad), n_pad=n_pad)
    if kind == "build":
        return dict(kind=kind, n=_log(rng, 100_000, 60_000_000), zipf=rng.choice([1.1, 1.3]))
    if kind == "attn":
        H, Hkv = rng.choice([(32, 32), (32, 8), (16, 16), (32, 4)])
        B, kv = _log(rng, 1, 32), _log(rng, 200, 16384)
        while B * Hkv * kv > 32 * 8 * 16384:
            B = max(1, B // 2)
        return dict(kind=kind, B=B, H=H, Hkv=Hkv, kv=kv, n_pad=n_pad)
    if kind in ("mlp", "head"):
        hidden, inter = rng.choice([(2048, 5504), (4096, 11008), (1024, 2816)])
        c = dict(kind=kind, B=_log(rng, 1, 32), n_pad=n_pad, hidden=hidden)
        return dict(c, inter=inter) if kind == "mlp" else c
    if kind == "decoder":
        hidden, H, Hkv, inter = rng.choice([(2048, 16, 16, 5504), (2048, 16, 4, 5504), (4096, 32, 8, 11008)])
        return dict(kind=kind, B=_log(rng, 1, 8), n_pad=n_pad, hidden=hidden, layers=rng.randint(2, 8), H=H, Hkv=Hkv, inter=inter,
                     kv=_log(rng, 200, 4096))
    B = _log(rng, 1, 32)
    return dict(kind=kind, B=B, n_split=rng.randint(1, min(4, B)), steps=rng.choice([4, 8]), n_general=_log(rng, 300_000, 20_000_000),
                n_project=_log(rng, 50_000, 2_000_000), n_max=16, k=64, d=10, budget=n_pad, n_pad=n_pad, H=32, Hkv=8, kv=_log(rng, 500, 16384),
                alg1=rng.random() < 0.5)


# ---------------------------------------------------------------- inputs
def _gen(seed, stream):
    g = torch.Generator(device=DEV)
    g.manual_seed((int(seed) * 1000003 + stream) & ((1 << 62) - 1))
    return g


def _randn(g, *shape):
    return torch.randn(shape, generator=g, device=DEV, dtype=BF)


_CDF = {}


def _zipf(g, n, s):
    """n Zipf(s) token ids, as code has them."""
    if s not in _CDF:
        _CDF[s] = torch.from_numpy(synth.zipf_cdf(s, VOCAB)).to(DEV)
    out = torch.empty(n, dtype=torch.int32, device=DEV)
    step = 1 << 25
    for lo in range(0, n, step):
        u = torch.rand(min(step, n - lo), generator=g, device=DEV, dtype=torch.float64)
        out[lo:lo + len(u)] = torch.searchsorted(_CDF[s], u, right=True).clamp_(max=VOCAB - 1).to(torch.int32)
    return out


def _corpus(g, n, s):
    """A Zipf stream in which 6 percent of the 64-token slots begin with 8 to 64 tokens copied from elsewhere: the repeats
    of code."""
    t = _zipf(g, n, s)
    slots = n // 64 - 1
    m = max(1, slots * 6 // 100)
    dst = torch.randperm(slots, generator=g, device=DEV)[:m] * 64
    src = torch.randint(0, n - 64, (m,), generator=g, device=DEV)
    ln = torch.randint(8, 65, (m,), generator=g, device=DEV)
    at = torch.arange(64, device=DEV)
    keep = (at[None, :] < ln[:, None]).reshape(-1)
    frm, to = (src[:, None] + at).reshape(-1)[keep], (dst[:, None] + at).reshape(-1)[keep]
    t[to] = t[frm]
    return t


def _stores_and_contexts(case, seed, ctx_len, stride):
    """A project store and a general store, and contexts whose last 16 tokens come from the project (half of them), the
    general store (a quarter) or neither."""
    g = _gen(seed, 1)
    corpora = [_corpus(g, case["n_project"], 1.3), _corpus(g, case["n_general"], 1.1)]
    B = case["B"]
    ctx = _zipf(g, B * ctx_len, 1.1).view(B, ctx_len)
    kind = torch.randint(0, 4, (B,), generator=g, device=DEV)
    at = torch.arange(16, device=DEV)
    for t, hit in ((corpora[0], kind < 2), (corpora[1], kind == 2)):
        p = torch.randint(0, len(t) - 32, (B,), generator=g, device=DEV)
        tail = t[p[:, None] + at]
        ctx[:, ctx_len - 16:] = torch.where(hit[:, None], tail, ctx[:, ctx_len - 16:])
    full = torch.zeros((B, stride), dtype=torch.int32, device=DEV)
    full[:, :ctx_len] = ctx
    return corpora, full, torch.full((B,), ctx_len, dtype=torch.int32, device=DEV)


def _sizes(case):
    """Tree sizes and cache lengths of a batch: a quarter of the trees are small, most are near the budget (the step loop's
    own mix); caches are between 60 percent of ``kv`` and all of it."""
    B, n_pad = case["B"], case["n_pad"]
    r = np.random.RandomState(B * 131071 + n_pad * 8191 + case.get("kv", 0) * 17 + 5)
    small = r.rand(B) < 0.3
    n = np.where(small, r.randint(1, n_pad // 2 + 1, B), r.randint(n_pad * 3 // 4, n_pad + 1, B))
    n[0] = min(n_pad, max(int(n[0]), n_pad * 3 // 4))
    kv = case.get("kv", 1)
    return n.astype(np.int32), r.randint(max(1, kv * 6 // 10), kv + 1, B).astype(np.int32)


def _trees(case, seed):
    """Random draft trees: tokens and parents, [B, n_pad]."""
    n, _ = _sizes(case)
    rng = np.random.default_rng([int(seed), 77])
    tok = np.full((case["B"], case["n_pad"]), -1, np.int32)
    par = np.full((case["B"], case["n_pad"]), -1, np.int32)
    for b, nb in enumerate(n):
        t, p = synth.random_tree(rng, int(nb), 10, 4, VOCAB)
        tok[b, :nb], par[b, :nb] = t.view(np.int32), p
    return tok, par


def _dev(a):
    return torch.from_numpy(np.ascontiguousarray(a)).to(DEV)


def _tree_inputs(case, seed):
    n, kv = _sizes(case)
    tok, par = _trees(case, seed)
    return dict(tok=_dev(tok), parent=_dev(par), n_nodes=_dev(n), kv_len=_dev(kv))


def _attn_inputs(case, seed):
    g = _gen(seed, 2)
    B, H, Hkv, n_pad = case["B"], case["H"], case["Hkv"], case["n_pad"]
    return dict(_tree_inputs(case, seed), q=_randn(g, B, n_pad, H, D), kc=_randn(g, B, Hkv, case["kv"], D), vc=_randn(g, B, Hkv, case["kv"], D),
                kt=_randn(g, B, Hkv, n_pad, D), vt=_randn(g, B, Hkv, n_pad, D))


def _mat(g, k, n):
    return (torch.randn((k, n), generator=g, device=DEV) * k ** -0.5).to(BF)


def _norm_w(g, n):
    return (1 + 0.1 * torch.randn(n, generator=g, device=DEV)).to(BF)


def _block_inputs(case, seed):
    g = _gen(seed, 3)
    T, hidden = case["B"] * case["n_pad"], case["hidden"]
    s = dict(x=_randn(g, T, hidden), w=_norm_w(g, hidden))
    if case["kind"] == "mlp":
        s.update(wgu=_mat(g, hidden, 2 * case["inter"]), wd=_mat(g, case["inter"], hidden))
    else:
        s.update(lm=_mat(g, hidden, VOCAB), **_tree_inputs(case, seed))
    return s


def _decoder_inputs(case, seed):
    W = synth.decoder_weights(case["hidden"], case["layers"], case["H"], case["Hkv"], D, case["inter"], VOCAB, int(seed) + 9, DEV)
    g = _gen(seed, 4)
    caches = [tuple(_randn(g, case["B"], case["Hkv"], case["kv"] + 64, D) for _ in range(2)) for _ in range(case["layers"])]
    return dict(_tree_inputs(case, seed), W=W, caches=caches)


def prepare(case, seed):
    s = {"case": case}
    kind, B = case["kind"], case["B"] if "B" in case else 0
    if kind == "draft":
        corpora, s["ctx"], s["ctx_len"] = _stores_and_contexts(case, seed, 64, 64)
        s["stores"] = [fc.fc_datastore_build(t, VOCAB) for t in corpora]
        s["p"] = fc.params(case["n_max"], 2, case["k"], case["d"])
        s["root"] = s["ctx"][:, -1].contiguous()
        s["kv_len"] = torch.full((B,), 1000, dtype=torch.int32, device=DEV)
        s["res"], s["tree"] = fc.retrieve_outputs(2, B, s["p"], DEV), fc.tree_outputs(B, case["n_pad"], DEV)
    elif kind == "build":
        s["tokens"] = _corpus(_gen(seed, 1), case["n"], case["zipf"])
    elif kind == "attn":
        s.update(_attn_inputs(case, seed))
        s["mask"] = fc.fc_tree_mask(s["parent"], s["n_nodes"], s["kv_len"])["mask"]
        s["out"] = torch.empty_like(s["q"])
    elif kind in ("mlp", "head"):
        s.update(_block_inputs(case, seed))
        s["h"] = torch.empty_like(s["x"])
        T = s["x"].shape[0]
        if kind == "mlp":
            s["wgu"] = fc.fc_interleave_gate_up(s["wgu"])
            s["act"] = torch.empty((T, case["inter"]), dtype=BF, device=DEV)
            s["o"] = torch.empty_like(s["x"])
        else:
            s["logits"] = torch.empty((T, VOCAB), dtype=BF, device=DEV)
    elif kind == "decoder":
        s.update(_decoder_inputs(case, seed))
        m = fc.fc_tree_mask(s["parent"], s["n_nodes"], s["kv_len"])
        s["mask"], s["pos"] = m["mask"], m["pos"]
        shape = DecoderShape(hidden=case["hidden"], layers=case["layers"], H=case["H"], Hkv=case["Hkv"], inter=case["inter"], vocab=VOCAB)
        s["dec"] = TreeDecoder(shape, s["W"], B, case["n_pad"], case["kv"] + 64, DEV, caches=s["caches"])
    else:
        steps, n_pad, H, Hkv = case["steps"], case["n_pad"], case["H"], case["Hkv"]
        grow = steps * (case["d"] + 1)
        corpora, ctx, ctx_len = _stores_and_contexts(case, seed, 128, 128 + grow)
        stores = [fc.fc_datastore_build(t, VOCAB) for t in corpora]
        g = _gen(seed, 5)
        cap = case["kv"] + grow
        kc, vc = _randn(g, B, Hkv, cap, D), _randn(g, B, Hkv, cap, D)
        seq = dict(capacity=4096, min_size=4, chunk=20) if case["alg1"] else None
        s["loop"] = PipelinedStepLoop(case["n_split"], stores, ctx, ctx_len, fc.params(case["n_max"], 2, case["k"], case["d"]), case["budget"],
                                      n_pad, [1, 1], H, Hkv, D, cap, _sizes(case)[1], VOCAB, k_cache=kc, v_cache=vc, seq_cache=seq)
        q = [_randn(g, B, n_pad, H, D) for _ in range(2)]
        kv = [[_randn(g, B, Hkv, n_pad, D) for _ in range(2)] for _ in range(2)]
        rnd = lambda hi, *shape: torch.randint(0, hi, shape, generator=g, device=DEV, dtype=torch.int32)  # noqa: E731
        # a target model that follows the tree for 0 to 8 tokens, and half of the queries may be served from the replay cache
        s["steps"] = [(q[t % 2], kv[t % 2][0], kv[t % 2][1], rnd(2, B), rnd(9, B), _zipf(g, B * n_pad, 1.1).view(B, n_pad)) for t in range(steps)]
    return s


# ---------------------------------------------------------------- one pass
def run(s):
    kind = s["case"]["kind"]
    if kind == "draft":
        fc.fc_retrieve(s["stores"], s["ctx"], s["ctx_len"], s["p"], out=s["res"])
        c = s["case"]
        fc.fc_build_tree(s["res"], [1, 1], s["root"], s["kv_len"], c["budget"], c["n_pad"], out=s["tree"])
        return dict(res=s["res"], tree=s["tree"])
    if kind == "build":
        ds = fc.fc_datastore_build(s["tokens"], VOCAB)
        return [ds.sa, ds.bucket, ds.lcp, ds.keys]
    if kind == "attn":
        return fc.fc_tree_attn(s["q"], s["kc"], s["vc"], s["kv_len"], s["kt"], s["vt"], s["mask"], s["n_nodes"], out=s["out"])
    if kind == "mlp":
        fc.fc_add_rmsnorm(s["x"], None, s["w"], s["h"])
        fc.fc_gemm_silu_mul(s["h"], s["wgu"], s["act"])
        fc.fc_gemm_bf16(s["act"], s["wd"], out=s["o"])
        return [s["act"], s["o"]]
    if kind == "head":
        fc.fc_add_rmsnorm(s["x"], None, s["w"], s["h"])
        fc.fc_gemm_bf16(s["h"], s["lm"], out=s["logits"])
        c = s["case"]
        acc = fc.fc_argmax_accept(s["logits"].view(c["B"], c["n_pad"], VOCAB), s["tok"], s["parent"], s["n_nodes"], 12)
        return dict(logits=s["logits"], acc=acc)
    if kind == "decoder":
        dec = s["dec"]
        logits = dec.forward(s["tok"], s["n_nodes"], s["mask"], s["pos"], s["kv_len"])
        return dict(logits=logits, k=dec.k_rot, v=dec.v_heads)
    loop = s["loop"]
    loop.reset()
    for step in s["steps"]:
        loop.step(*step)
    loop.join()
    return dict(attn=loop.attn_out, acc=loop.acc, tree=loop.tree, ctx=loop.ctx, ctx_len=loop.ctx_len_now, kv_len=loop.kv_len_now)


# ---------------------------------------------------------------- what a pass cannot do without
def _attn_work(B, H, Hkv, n_pad, n, kv):
    n, kv = n.astype(np.float64), kv.astype(np.float64)
    byt = 2 * 2 * Hkv * D * (kv.sum() + n.sum()) + 2 * H * D * (n.sum() + B * n_pad) + (n * n_pad / 8).sum()
    return byt, 4 * D * H * (n * (kv + 5)).sum()


def _draft_bytes(c, sources=2):
    B, k, d, n_pad = c["B"], c["k"], c["d"], c["n_pad"]
    found = sources * B * (k * (d + 2) + 2) * 4
    return B * 256 + 2 * found + B * n_pad * (16 + n_pad / 8)


def work(case):
    c, kind = case, case["kind"]
    if kind == "draft":
        return {"bytes": _draft_bytes(c), "flops": 0.0}
    if kind == "build":
        return {"bytes": c["n"] * (4 + 4 + 1 + 32) + 4 * (VOCAB + 1), "flops": 0.0}
    n, kv = _sizes(c)
    if kind == "attn":
        byt, fl = _attn_work(c["B"], c["H"], c["Hkv"], c["n_pad"], n, kv)
        return {"bytes": byt, "flops": fl}
    if kind == "loop":
        byt, fl = _attn_work(c["B"], c["H"], c["Hkv"], c["n_pad"], np.full(c["B"], 0.7 * c["n_pad"]), kv)
        append = 4 * 5 * c["B"] * c["Hkv"] * D * 2
        return {"bytes": c["steps"] * (byt + _draft_bytes(c) + append), "flops": c["steps"] * fl}
    T, hid = c["B"] * c["n_pad"], c["hidden"]
    if kind == "mlp":
        inter = c["inter"]
        return {"bytes": 2 * (3 * hid * inter + 2 * T * hid + hid + T * inter), "flops": 6.0 * T * hid * inter}
    if kind == "head":
        return {"bytes": 2 * (hid * VOCAB + T * hid + hid + T * VOCAB), "flops": 2.0 * T * hid * VOCAB}
    H, Hkv, inter, L = c["H"], c["Hkv"], c["inter"], c["layers"]
    per = 2 * hid * H * D + 2 * hid * Hkv * D + 3 * hid * inter
    abyt, afl = _attn_work(c["B"], H, Hkv, c["n_pad"], n, kv)
    return {"bytes": 2 * (L * per + hid * VOCAB + T * hid + T * VOCAB) + L * (abyt - 4 * H * D * T + 4 * T * Hkv * D),
            "flops": 2.0 * T * (L * per + hid * VOCAB) + L * afl}


def tolerance(case):
    kind = case["kind"]
    if kind in ("draft", "build"):
        return "exact"
    if kind == "attn":
        return {"rel": 1e-2}  # bf16 probabilities and results: about 2.3e-3 from 64 bits
    if kind == "mlp":
        return {"rel": 1e-2}  # bf16 activations and results: about 3e-3
    if kind == "head":
        return {"rel": 1e-2, "differ": 0.005}  # two logits that tie in bf16 change places
    if kind == "decoder":
        return {"rel": 3e-2}  # bf16 between all operations of all layers
    return {"rel": 1e-2}


# ---------------------------------------------------------------- the same in 64 bits
def _ancestors(par):
    """[n_pad, n_pad] truth values: row i may see column j."""
    n = len(par)
    m = np.zeros((n, n), bool)
    for i in range(n):
        if i and par[i] < 0:
            continue
        j = i
        while j >= 0:
            m[i, j] = True
            j = par[j]
    return m


def _attn64(q, kc, vc, kv, kt, vt, par, n):
    """q [B, n_pad, H, D] -> the same shape, float64; rows past a tree's nodes are zero."""
    B, n_pad, H, _ = q.shape
    Hkv = kc.shape[1]
    G = H // Hkv
    out = torch.zeros(q.shape, dtype=torch.float64, device=DEV)
    for b in range(B):
        nb, L = int(n[b]), int(kv[b])
        see = _dev(_ancestors(par[b])[:nb, :nb])
        for g in range(Hkv):
            qq = q[b, :nb, g * G:(g + 1) * G].double().transpose(0, 1) * D ** -0.5  # [G, nb, D]
            k = torch.cat([kc[b, g, :L], kt[b, g, :nb]]).double()
            v = torch.cat([vc[b, g, :L], vt[b, g, :nb]]).double()
            sc = qq @ k.T
            sc[:, :, L:] = sc[:, :, L:].masked_fill(~see, -math.inf)
            out[b, :nb, g * G:(g + 1) * G] = (torch.softmax(sc, -1) @ v).transpose(0, 1)
    return out


def _rms64(x, w, eps=1e-6):
    return x * torch.rsqrt(x.square().mean(-1, keepdim=True) + eps) * w.double()


def _rope64(x, pos, base=10000.0):
    """x [..., rows, D] with pos [..., rows]: dimension i turns with i + D/2; rows of negative positions stay."""
    f = base ** (-2 * torch.arange(D // 2, device=DEV, dtype=torch.float64) / D)
    a = pos.clamp(min=0).double()[..., None] * f
    lo, hi = x[..., :D // 2], x[..., D // 2:]
    return torch.cat([lo * a.cos() - hi * a.sin(), hi * a.cos() + lo * a.sin()], -1)


def exact(case, seed):
    kind = case["kind"]
    if kind in ("draft", "build", "loop"):
        return None  # whole numbers; the loop's attention is the attention cases'
    if kind == "attn":
        s = _attn_inputs(case, seed)
        n, kv = _sizes(case)
        return _attn64(s["q"], s["kc"], s["vc"], kv, s["kt"], s["vt"], s["parent"].cpu().numpy(), n)
    if kind in ("mlp", "head"):
        s = _block_inputs(case, seed)
        h = _rms64(s["x"].double(), s["w"])
        if kind == "head":
            return dict(logits=torch.cat([h @ w.double() for w in s["lm"].split(8192, 1)], 1), acc=None)
        gu = h @ s["wgu"].double()
        gate, up = gu.split(case["inter"], 1)
        act = gate * torch.sigmoid(gate) * up
        return [act, act @ s["wd"].double()]
    s = _decoder_inputs(case, seed)
    n, kv = _sizes(case)
    B, n_pad, H, Hkv = case["B"], case["n_pad"], case["H"], case["Hkv"]
    tok, par = s["tok"], s["parent"].cpu().numpy()
    depth = np.full(par.shape, -1)
    for b in range(B):
        for i in range(int(n[b])):
            depth[b, i] = 0 if i == 0 else depth[b, par[b, i]] + 1
    pos = _dev(np.where(depth >= 0, kv[:, None] + depth, -1))
    W = s["W"]
    x = torch.where((tok >= 0).reshape(-1, 1), W["embed"][tok.clamp(min=0).long().reshape(-1)].double(), 0.0)
    ks, vs = [], []
    for lw, (kc, vc) in zip(W["layers"], s["caches"]):
        h = _rms64(x, lw["attn_norm"])
        q = (h @ lw["wq"].double()).view(B, n_pad, H, D)
        kk, vv = (h @ lw["wkv"].double()).view(B, n_pad, 2, Hkv, D).permute(2, 0, 3, 1, 4)
        q = _rope64(q, pos[:, :, None].expand(B, n_pad, H))
        kk = _rope64(kk, pos[:, None, :].expand(B, Hkv, n_pad))
        ks.append(kk)
        vs.append(vv)
        a = _attn64(q, kc, vc, kv, kk, vv, par, n)
        x = x + a.reshape(B * n_pad, H * D) @ lw["wo"].double()
        gate, up = (_rms64(x, lw["mlp_norm"]) @ lw["wgu"].double()).split(case["inter"], 1)
        x = x + (gate * torch.sigmoid(gate) * up) @ lw["wd"].double()
    h = _rms64(x, W["final_norm"])
    return dict(logits=torch.cat([h @ w.double() for w in W["lm_head"].split(8192, 1)], 1).view(B, n_pad, VOCAB), k=ks, v=vs)
