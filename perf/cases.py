"""The work a user of this framework has it do, as cases that can be timed.

Every case goes through the framework's public entry points (``VerifyRound``,
``BlockPrefill`` and the calls of ``paper_2605_24793_gb300.cospec``).  Sizes are those of
the workloads in ``workload.CONFIGS``, of the tests and of the benchmark: the Qwen3-8B,
Qwen3-32B and Llama-3-8B shapes at their batch sizes, the tiny round, the paper's
default draft length K = 25 and the arbitrator's regions.  The seven kinds of case:

  round    one whole verify / arbitrate / commit round replayed as a CUDA graph
  attn     the verify attention of one layer (decode direction)
  region   the arbitrator's attention of one layer (the draft/target region, full mask)
  prefill  the causal prefill of a context: pack, commit and attend every layer
  lmhead   the fused LM head, greedy or sampled at T = 1
  sps      the exact-match baseline's step: LM-head logits, acceptance, commit
  rl       rewards, advantages and objective of a batch of rollouts
"""
from __future__ import annotations

import math

import numpy as np
import torch

from paper_2605_24793_gb300 import cospec as C
from paper_2605_24793_gb300 import workload as W
from paper_2605_24793_gb300.prefill import BlockPrefill
from paper_2605_24793_gb300.round import VerifyRound

DEV = "cuda"
PAGE = 16


def listed():
    qwen8 = dict(q_heads=32, kv_heads=8, head_dim=128)
    return [
        # The smallest round there is: one layer, batch 1, vocabulary 4096.  Latency and
        # launches are all of it.
        dict(name="round_tiny", kind="round", batch=1, ctx_lo=256, ctx_hi=256, k=4, layers=1,
             hidden=512, vocab=4096, q_heads=8, kv_heads=2, head_dim=64, mlp=64),
        # One user being served: every layer of a Qwen3-8B-shaped target at batch 1.
        dict(name="round_qwen8b_b1", kind="round", batch=1, ctx_lo=4096, ctx_hi=4096, k=5, layers=36,
             hidden=4096, vocab=151936, mlp=256, **qwen8),
        # A serving batch of ragged contexts over a shuffled page table, one layer.
        dict(name="attn_b16_k7", kind="attn", batch=16, ctx_lo=2048, ctx_hi=8192, k=7, **qwen8),
        # The same batch at the paper's default draft length.
        dict(name="attn_b16_k25", kind="attn", batch=16, ctx_lo=2048, ctx_hi=8192, k=25, **qwen8),
        # Long reasoning: one layer of the Llama-3-8B-shaped batch-64 workload, the largest.
        dict(name="attn_llama_b64_k7", kind="attn", batch=64, ctx_lo=8192, ctx_hi=32768, k=7, **qwen8),
        # The arbitrator's look at a K = 25 block: 53 region rows over the cached context.
        dict(name="region_k25_b4", kind="region", batch=4, ctx_lo=4096, ctx_hi=4096, k=25, **qwen8),
        # A new request's context enters the arbitrator's cache.
        dict(name="prefill_4096", kind="prefill", batch=1, context=4096, layers=4, **qwen8),
        # The LM head of the Qwen3-32B batch-32 round (256 rows) and of the Llama batch-64
        # round (512 rows).
        dict(name="lmhead_qwen32b_256", kind="lmhead", rows=256, hidden=5120, vocab=151936, k=7, sample=False),
        dict(name="lmhead_llama_512", kind="lmhead", rows=512, hidden=4096, vocab=128256, k=7, sample=False),
        # Stochastic decoding at T = 1, Qwen3-8B shape, batch 16.
        dict(name="lmhead_sample_128", kind="lmhead", rows=128, hidden=4096, vocab=151936, k=7, sample=True),
        # The distribution-preserving baseline's decision step at batch 16, with the commit of 32 layers.
        dict(name="sps_b16_k7", kind="sps", batch=16, ctx_lo=128, ctx_hi=512, k=7, layers=32, hidden=4096,
             vocab=151936, kv_heads=8, head_dim=128),
        # The RL stage on 256 prompts x 8 rollouts of up to 64 rounds.
        dict(name="rl_256x8x64_k25", kind="rl", groups=256, rollouts=8, rounds=64, k=25),
    ]


def _log_int(rng, lo, hi):
    """An integer in [lo, hi], uniform in the logarithm."""
    return max(lo, min(hi, int(round(math.exp(rng.uniform(math.log(lo), math.log(hi)))))))


_HEADS = [(32, 8, 128), (32, 8, 128), (64, 8, 128), (8, 2, 64), (16, 8, 64), (12, 4, 128)]


def draw(rng):
    kind = rng.choice(["round", "attn", "attn", "region", "prefill", "lmhead", "sps", "rl"])
    hq, hkv, d = rng.choice(_HEADS)
    heads = dict(q_heads=hq, kv_heads=hkv, head_dim=d)
    if kind == "round":
        hi = _log_int(rng, 100, 6000)
        return dict(kind=kind, batch=rng.randint(1, 4), ctx_lo=max(1, hi // 2), ctx_hi=hi, k=rng.randint(1, 15),
                    layers=rng.randint(1, 24), hidden=64 * rng.randint(8, 64), vocab=_log_int(rng, 4000, 60000),
                    mlp=rng.randint(32, 256), **heads)
    if kind == "attn":
        batch, hi = _log_int(rng, 1, 64), _log_int(rng, 200, 32768)
        return dict(kind=kind, batch=batch, ctx_lo=max(1, hi // 4), ctx_hi=hi, k=rng.randint(0, 25), **heads)
    if kind == "region":
        hi = _log_int(rng, 500, 8192)
        return dict(kind=kind, batch=_log_int(rng, 1, 16), ctx_lo=max(1, hi // 2), ctx_hi=hi, k=rng.randint(1, 29), **heads)
    if kind == "prefill":
        return dict(kind=kind, batch=rng.randint(1, 2), context=_log_int(rng, 200, 4096), layers=rng.randint(1, 3), **heads)
    if kind == "lmhead":
        return dict(kind=kind, rows=_log_int(rng, 1, 512), hidden=64 * rng.randint(8, 72),
                    vocab=_log_int(rng, 4000, 128256), k=rng.randint(0, 15), sample=rng.random() < 0.4)
    if kind == "sps":
        return dict(kind=kind, batch=_log_int(rng, 1, 24), ctx_lo=64, ctx_hi=_log_int(rng, 128, 512), k=rng.randint(1, 9),
                    layers=rng.randint(1, 32), hidden=64 * rng.randint(8, 64), vocab=_log_int(rng, 4000, 128256),
                    kv_heads=hkv, head_dim=d)
    return dict(kind="rl", groups=_log_int(rng, 8, 512), rollouts=rng.randint(1, 8), rounds=_log_int(rng, 2, 64), k=rng.randint(3, 31))


# ---------------------------------------------------------------- inputs (plain torch, from the seed alone)
def _gen(seed):
    g = torch.Generator(device=DEV)
    g.manual_seed(int(seed) * 7919 + 13)
    return g


def _normal(g, shape, std=1.0):
    return torch.empty(shape, dtype=torch.bfloat16, device=DEV).normal_(0.0, std, generator=g)


def _contexts(case, seed):
    """Ragged context lengths spread evenly over [ctx_lo, ctx_hi], in an order of the seed."""
    B, lo, hi = case["batch"], case["ctx_lo"], case["ctx_hi"]
    rng = np.random.default_rng(int(seed))
    ctx = lo + np.floor((hi - lo + 1) * (np.arange(B) + rng.random(B)) / B).astype(np.int64)
    return np.minimum(rng.permutation(ctx), hi).astype(np.int32)


def _pages(case, ctx, rows, seed):
    """A shuffled page table with room for the context and one block, over a pool whose size
    is the same for every seed."""
    B, lo, hi = case["batch"], case["ctx_lo"], case["ctx_hi"]
    most = np.minimum(lo + (hi - lo + 1) * np.arange(1, B + 1) // B, hi)
    total = int(((most + rows + PAGE - 1) // PAGE).sum())
    need = (ctx.astype(np.int64) + rows + PAGE - 1) // PAGE
    order = np.random.default_rng(int(seed) + 1).permutation(total)
    table = np.full((B, (hi + rows + PAGE - 1) // PAGE), -1, dtype=np.int32)
    at = 0
    for b, n in enumerate(need):
        table[b, :n] = order[at:at + n]
        at += int(n)
    return table, total


def _cache_inputs(case, seed, layers, rows, q_heads):
    g = _gen(seed)
    B, Hkv, D = case["batch"], case["kv_heads"], case["head_dim"]
    ctx = _contexts(case, seed)
    table, n = _pages(case, ctx, rows, seed)
    s = dict(ctx_np=ctx, table=torch.from_numpy(table).to(DEV), ctx=torch.from_numpy(ctx).to(DEV), table_np=table, num_pages=n)
    if q_heads:
        s["q"] = _normal(g, (layers, B, rows, q_heads, D))
    s["kb"] = _normal(g, (layers, B, rows, Hkv, D))
    s["vb"] = _normal(g, (layers, B, rows, Hkv, D))
    s["kp"] = _normal(g, (layers, n, Hkv, PAGE, D))
    s["vp"] = _normal(g, (layers, n, Hkv, PAGE, D))
    return s, g


def _head_inputs(case, g, rows):
    return _normal(g, (rows, case["hidden"])), _normal(g, (case["vocab"], case["hidden"]), 0.02)


def _drafts(g, hidden, w, batch, k, rate=0.3):
    """The target's first choice with probability 1 - rate, else one of its next seven."""
    V = w.shape[0]
    top = torch.cat([torch.topk(hidden[i:i + 64].float() @ w.float().T, min(8, V), dim=1).indices
                     for i in range(0, hidden.shape[0], 64)]).view(batch, k + 1, -1)[:, :k]
    pick = torch.randint(1, top.shape[2], (batch, k, 1), generator=g, device=DEV)
    keep = torch.rand((batch, k, 1), generator=g, device=DEV) >= rate
    return torch.gather(top, 2, torch.where(keep, torch.zeros_like(pick), pick)).view(batch, k).to(torch.int32)


def _mlp(seed, H):
    r = np.random.default_rng(int(seed) + 5)
    a1, a2 = 1.0 / math.sqrt(8), 1.0 / math.sqrt(H)
    u = lambda n, a: torch.from_numpy(r.uniform(-a, a, n).astype(np.float32))  # noqa: E731
    return u((H, 8), a1), u(H, a1), u(H, a2), u((), a2)


def _round_inputs(case, seed):
    s, g = _cache_inputs(case, seed, case["layers"], case["k"] + 1, case["q_heads"])
    s["hidden"], s["w"] = _head_inputs(case, g, case["batch"] * (case["k"] + 1))
    s["draft"] = _drafts(g, s["hidden"], s["w"], case["batch"], case["k"])
    s["mlp"] = _mlp(seed, case["mlp"])
    return s


def _region_rows(case):
    return 2 * case["k"] + 3 if case["kind"] == "region" else case["k"] + 1


def _prefill_inputs(case, seed):
    g = _gen(seed)
    L, B, T, D = case["layers"], case["batch"], case["context"], case["head_dim"]
    return dict(q=_normal(g, (L, B, T, case["q_heads"], D)), k=_normal(g, (L, B, T, case["kv_heads"], D)),
                v=_normal(g, (L, B, T, case["kv_heads"], D)))


def _lmhead_inputs(case, seed):
    g = _gen(seed)
    s = {}
    s["hidden"], s["w"] = _head_inputs(case, g, case["rows"])
    draft = torch.randint(0, case["vocab"], (case["rows"],), generator=g, device=DEV, dtype=torch.int32)
    draft[case["k"]::case["k"] + 1] = -1          # the bonus row of every block scores no draft
    s["draft"] = draft
    return s


def _sps_inputs(case, seed):
    R, K, B, V = case["k"] + 1, case["k"], case["batch"], case["vocab"]
    s, g = _cache_inputs(case, seed, case["layers"], R, 0)
    s["hidden"], s["w"] = _head_inputs(case, g, B * R)
    wf = s["w"].float()
    q = torch.empty((B, K, V), device=DEV)
    for b in range(B):                            # a draft that roughly agrees with the target
        x = s["hidden"][b * R:b * R + K].float() @ wf.T
        q[b] = torch.softmax(x + torch.empty_like(x).normal_(generator=g), dim=1)
    s["dq"] = q
    s["draft"] = torch.multinomial(q.view(B * K, V), 1, generator=g).view(B, K).to(torch.int32)
    s["seed"] = int(seed) * 0x9E3779B97F4A7C15 % (1 << 63)
    return s


def _rl_inputs(case, seed):
    g = _gen(seed)
    G, M, K = case["groups"], case["groups"] * case["rollouts"], case["k"]
    r = np.random.default_rng(int(seed))
    nr = r.permutation(1 + np.arange(M) % case["rounds"])
    off = np.concatenate([[0], np.cumsum(nr)]).astype(np.int32)
    R = int(off[-1])
    u = lambda: torch.rand((R, K), generator=g, device=DEV)  # noqa: E731
    match = (u() >= 0.3).to(torch.uint8)
    return dict(group_off=torch.arange(0, M + 1, case["rollouts"], dtype=torch.int32, device=DEV), round_off=torch.from_numpy(off).to(DEV),
                correct=torch.from_numpy((r.random(M) < 0.5).astype(np.uint8)).to(DEV), match=match,
                accept=match | (u() < 0.6).to(torch.uint8), ell=torch.log1p(-u()) * 1.5,
                ratio=torch.exp(0.2 * torch.empty((R, K), device=DEV).normal_(generator=g)),
                p_new=u() * 0.9 + 0.05, p_ref=u() * 0.9 + 0.05)


# ---------------------------------------------------------------- what a user's program has in hand
def prepare(case, seed):
    kind = case["kind"]
    if kind == "round":
        s = _round_inputs(case, seed)
        cfg = W.RoundConfig("round", 0, batch=case["batch"], ctx_lo=case["ctx_lo"], ctx_hi=case["ctx_hi"], k=case["k"],
                            layers=case["layers"], hidden=case["hidden"], q_heads=case["q_heads"], kv_heads=case["kv_heads"],
                            head_dim=case["head_dim"], vocab=case["vocab"], mlp_hidden=case["mlp"], mismatch_rate=0.3,
                            mismatch_topk=8, shuffled_pages=True)
        inp = dict(cfg=cfg, ctx_len_np=s["ctx_np"], page_table_np=s["table_np"], num_pages=s["num_pages"], q=s["q"], k_blk=s["kb"],
                   v_blk=s["vb"], k_pages=s["kp"], v_pages=s["vp"], hidden=s["hidden"], w=s["w"], mlp=s["mlp"],
                   page_table=s["table"], ctx_len=s["ctx"])
        rnd = VerifyRound(inp, s["draft"].cpu().numpy(), keep_attn=True)
        rnd.capture()
        return dict(kind=kind, rnd=rnd)
    if kind in ("attn", "region"):
        s, _ = _cache_inputs(case, seed, 1, _region_rows(case), case["q_heads"])
        return dict(kind=kind, args=(s["q"][0], s["kb"][0], s["vb"][0], s["kp"][0], s["vp"][0], s["table"], s["ctx"],
                                     torch.empty_like(s["q"][0]), int(s["ctx_np"].max())))
    if kind == "prefill":
        s = _prefill_inputs(case, seed)
        return dict(kind=kind, pf=BlockPrefill(case["layers"], case["batch"], case["context"], case["q_heads"], case["kv_heads"],
                                               case["head_dim"]), **s)
    if kind == "lmhead":
        s = _lmhead_inputs(case, seed)
        M = case["rows"]
        s.update(kind=kind, sample=case["sample"], ids=torch.empty(M, dtype=torch.int32, device=DEV),
                 stats=torch.empty((M, 5), device=DEV), ws=C.new_lmhead_workspace(M, case["hidden"], case["vocab"]),
                 seed=torch.tensor([int(seed) * 0x9E3779B97F4A7C15 % (1 << 63)], dtype=torch.int64, device=DEV))
        return s
    if kind == "sps":
        s = _sps_inputs(case, seed)
        B, K, V = case["batch"], case["k"], case["vocab"]
        M = B * (K + 1)
        i32 = dict(dtype=torch.int32, device=DEV)
        row_ids = torch.full((B, K + 1), -1, **i32)
        row_ids[:, :K] = s["draft"]
        s.update(kind=kind, ctx0=s["ctx"].clone(), row_ids=row_ids.view(-1), seed=torch.tensor([s["seed"]], dtype=torch.int64, device=DEV),
                 argmax=torch.empty(M, **i32), stats=torch.empty((M, 5), device=DEV), logits=torch.empty((M, V), device=DEV),
                 target=torch.empty(M, **i32), accept=torch.empty((B, K), dtype=torch.uint8, device=DEV),
                 ratio=torch.empty((B, K), device=DEV), s=torch.empty(B, **i32), emitted=torch.empty((B, K + 1), **i32),
                 ws_lm=C.new_lmhead_workspace(M, case["hidden"], V), ws_sps=C.new_sps_workspace(B))
        return s
    s = _rl_inputs(case, seed)
    s["kind"] = kind
    return s


def run(state):
    kind = state["kind"]
    if kind == "round":
        r = state["rnd"]
        r.replay()
        return dict(attn=r.attn_out, argmax=r.argmax, stats=r.stats, p=r.p, accept=r.accept, s=r.accept_len, emitted=r.emitted,
                    ctx=r.ctx_len, k_pages=r.k_pages, v_pages=r.v_pages)
    if kind in ("attn", "region"):
        return C.verify_attn(*state["args"], block_full=kind == "region")
    if kind == "prefill":
        pf = state["pf"]
        out = pf.run(state["q"], state["k"], state["v"])
        return dict(out=out, ctx=pf.ctx_len, k_pages=pf.k_pages, v_pages=pf.v_pages)
    if kind == "lmhead":
        a = state
        if a["sample"]:
            return C.lmhead_sample_features(a["hidden"], a["w"], a["draft"], 1.0, a["seed"], a["ids"], a["stats"], a["ws"])
        return C.lmhead_argmax_features(a["hidden"], a["w"], a["draft"], a["ids"], a["stats"], a["ws"])
    if kind == "sps":
        a = state
        a["ctx"].copy_(a["ctx0"])
        C.lmhead_logits_features(a["hidden"], a["w"], a["row_ids"], 1.0, a["argmax"], a["stats"], a["logits"], a["ws_lm"])
        C.sps_accept(a["draft"], a["stats"], a["logits"], a["dq"], a["seed"], a["target"], a["accept"], a["ratio"], a["ws_sps"])
        C.accept_commit(a["draft"], a["target"], a["accept"], a["kb"], a["vb"], a["kp"], a["vp"], a["table"], a["ctx"], a["s"],
                        a["emitted"])
        return dict(argmax=a["argmax"], stats=a["stats"], logits=a["logits"], target=a["target"], accept=a["accept"],
                    ratio=a["ratio"], s=a["s"], emitted=a["emitted"], ctx=a["ctx"], k_pages=a["kp"], v_pages=a["vp"])
    a = state
    return C.rl_advantages(a["group_off"], a["correct"], a["round_off"], a["match"], a["accept"], a["ell"], None, a["ratio"],
                           a["p_new"], a["p_ref"])


# ---------------------------------------------------------------- what a pass cannot do without
def _attn_work(case, rows):
    B, Hq, Hkv, D = case["batch"], case["q_heads"], case["kv_heads"], case["head_dim"]
    keys = B * (case["ctx_lo"] + case["ctx_hi"]) / 2
    seen = rows if case["kind"] == "region" else (rows + 1) / 2
    return (4.0 * keys * Hkv * D + 4.0 * B * rows * (Hq + Hkv) * D, 4.0 * Hq * D * rows * (keys + B * seen))


def _head_work(case, rows):
    d, V = case["hidden"], case["vocab"]
    return 2.0 * V * d + 2.0 * rows * d + 24.0 * rows, 2.0 * rows * d * V


def work(case):
    kind = case["kind"]
    if kind == "lmhead":
        b, f = _head_work(case, case["rows"])
    elif kind in ("attn", "region"):
        b, f = _attn_work(case, _region_rows(case))
    elif kind == "round":
        R, B, L = case["k"] + 1, case["batch"], case["layers"]
        b, f = (x + L * y for x, y in zip(_head_work(case, B * R), _attn_work(case, R)))
        b += 8.0 * L * B * R * case["kv_heads"] * case["head_dim"]        # the block's K/V into the cache
    elif kind == "prefill":
        n = case["layers"] * case["batch"] * case["context"] * case["head_dim"]
        b = 4.0 * n * (case["q_heads"] + 2 * case["kv_heads"])
        f = 2.0 * n * case["q_heads"] * (case["context"] + 1)
    elif kind == "sps":
        R, B, V = case["k"] + 1, case["batch"], case["vocab"]
        b, f = _head_work(case, B * R)
        b += 4.0 * B * R * V + 8.0 * B * V + 8.0 * case["layers"] * B * R * case["kv_heads"] * case["head_dim"] / 2
    else:
        n = case["groups"] * case["rollouts"] * (case["rounds"] + 1) / 2 * case["k"]
        b, f = 27.0 * n, 60.0 * n
    return dict(bytes=b, flops=f)


def tolerance(case):
    kind = case["kind"]
    # bf16 attention outputs whose probabilities are rounded to bf16 at another scale
    if kind in ("attn", "region", "prefill"):
        return dict(rel=1e-2, max=0.1)
    # the round holds such attention outputs beside 32-bit statistics; ids may differ at ties
    if kind == "round":
        return dict(rel=1e-2, max=0.1, differ=0.004)
    # 32-bit sums of bf16 products; a near tie may turn one id
    if kind in ("lmhead", "sps"):
        return dict(rel=2e-5, max=2e-3, differ=0.004)
    # 64-bit arithmetic, 32-bit results
    return dict(rel=1e-6, max=1e-5)


# ---------------------------------------------------------------- 64-bit results, without this repository's code
def _attend64(q, kb, vb, kp, vp, table, ctx, full):
    out = torch.empty(q.shape, dtype=torch.float64, device=DEV)
    B, R, Hq, D = q.shape
    Hkv = kb.shape[2]
    G = Hq // Hkv
    mask = torch.zeros((R, R), dtype=torch.float64, device=DEV)
    if not full:
        mask.masked_fill_(torch.ones((R, R), dtype=torch.bool, device=DEV).triu(1), -math.inf)
    for b in range(B):
        n = int(ctx[b])
        ids = torch.from_numpy(table[b, :(n + PAGE - 1) // PAGE].astype(np.int64)).to(DEV)
        k, v = (torch.cat([p[ids].permute(1, 0, 2, 3).reshape(Hkv, -1, D)[:, :n], x[b].transpose(0, 1)], 1).double()
                for p, x in ((kp, kb), (vp, vb)))
        qq = q[b].view(R, Hkv, G, D).permute(1, 2, 0, 3).reshape(Hkv, G * R, D).double()
        x = qq @ k.transpose(1, 2) / math.sqrt(D)
        x[:, :, n:] += mask.repeat(G, 1)
        o = torch.softmax(x, 2) @ v
        out[b] = o.view(Hkv, G, R, D).permute(2, 0, 1, 3).reshape(R, Hq, D)
    return out


def _stats64(hidden, w, draft):
    """[M, 5]: max, second, log-sum-exp, entropy, the draft's logit; the argmax; the logits."""
    w64 = w.double()
    x = torch.cat([hidden[i:i + 64].double() @ w64.T for i in range(0, hidden.shape[0], 64)])
    st = torch.full((x.shape[0], 5), math.nan, dtype=torch.float64, device=DEV)
    top = torch.topk(x, 2, dim=1)
    st[:, :2] = top.values
    st[:, 2] = torch.logsumexp(x, 1)
    for i in range(0, x.shape[0], 64):
        st[i:i + 64, 3] = st[i:i + 64, 2] - (torch.softmax(x[i:i + 64], 1) * x[i:i + 64]).sum(1)
    has = draft >= 0
    st[has, 4] = x[has, draft[has].long()]
    return st, top.indices[:, 0].to(torch.int32), x


def _policy64(st, argmax, draft, mlp, batch, k):
    st, argmax = st.view(batch, k + 1, 5), argmax.view(batch, k + 1)
    match = draft == argmax[:, :k]
    a, n = st[:, :k], st[:, 1:]
    i = torch.arange(1, k + 1, dtype=torch.float64, device=DEV)
    f = torch.stack([a[..., 4] - a[..., 2], a[..., 0] - a[..., 2], a[..., 0] - a[..., 1], a[..., 3], n[..., 0] - n[..., 2],
                     torch.nan_to_num(n[..., 4] - n[..., 2], nan=0.0), (i / k).expand(batch, k),
                     (match.double().cumsum(1) - match.double()) / k], 2)
    w1, b1, w2, b2 = (t.to(DEV).double() for t in mlp)
    z = torch.relu(f @ w1.T + b1) @ w2 + b2
    return torch.where(match, torch.ones_like(z), torch.sigmoid(z))


def _rl64(s):
    alpha, beta, eta_fail, eps, ce, bh, bk = 1.0, 0.25, 0.5, float(np.float32(1e-6)), float(np.float32(0.2)), float(np.float32(0.01)), float(np.float32(0.02))
    R, K = s["match"].shape
    i = torch.arange(1, K + 1, device=DEV)
    mism = s["match"] == 0
    rej = mism & (s["accept"] == 0)
    first = lambda m: torch.where(m.any(1), m.to(torch.uint8).argmax(1) + 1, torch.full((R,), K + 1, device=DEV))  # noqa: E731
    stop, istar = first(rej), first(mism)
    has = mism.any(1)
    rho = torch.where(has, (stop - istar).double() / (K + 1 - istar).clamp(min=1).double(), torch.zeros(R, dtype=torch.float64, device=DEV))
    eff = mism & (i <= stop.clamp(max=K)[:, None])
    M = s["correct"].numel()
    of = torch.repeat_interleave(torch.arange(M, device=DEV), (s["round_off"][1:] - s["round_off"][:-1]).long())
    corr = s["correct"].bool()
    cr = corr[of][:, None]
    bad = -alpha * s["ell"].double().abs() * (i < stop[:, None]) - beta * (i == stop[:, None])
    zero = torch.zeros((), dtype=torch.float64, device=DEV)
    g = torch.where(eff, torch.where(cr, rho[:, None].expand(R, K), bad), zero)
    seg = lambda x: torch.zeros(M, dtype=torch.float64, device=DEV).index_add_(0, of, x)  # noqa: E731
    J, A = seg(g.sum(1)), seg(g.abs().sum(1))
    per = M // (s["group_off"].numel() - 1)
    Jg, cg = J.view(-1, per), corr.view(-1, per)
    pos, neg = (Jg * cg).sum(1), (Jg * ~cg).abs().sum(1)
    mixed = cg.any(1) & ~cg.all(1)
    gamma = torch.where(mixed, neg / (pos + eps), torch.ones_like(pos))
    Jb = torch.where(cg, gamma[:, None] * Jg, Jg)
    mu = Jb.mean(1, keepdim=True)
    sd = (Jb - mu).square().mean(1, keepdim=True).sqrt()
    eta = torch.where(cg.any(1, keepdim=True), 1.0, eta_fail)
    adv = (eta * (Jb - mu) / (sd + eps)).view(-1)
    share = torch.where(A[of][:, None] > 0, g.abs() / A[of][:, None], zero)
    dec = torch.where(eff, torch.where(cr, rho[:, None], share) * adv[of][:, None], zero)
    rt, p, q = (s[n].double() for n in ("ratio", "p_new", "p_ref"))
    surr = (torch.minimum(rt * dec, rt.clamp(1 - ce, 1 + ce) * dec) * eff).sum()
    ent = ((-p * p.log() - (1 - p) * (1 - p).log()) * eff).sum()
    kl = ((p * (p / q).log() + (1 - p) * ((1 - p) / (1 - q)).log()) * eff).sum()
    return dict(g=g, eff=None, rho=torch.where(has, rho, torch.full_like(rho, math.nan)), J=J, Jbar=Jb.view(-1), adv=adv, adv_dec=dec,
                loss=torch.stack([surr, ent, kl, -surr - bh * ent + bk * kl]))


def exact(case, seed):
    kind = case["kind"]
    if kind in ("attn", "region"):
        s, _ = _cache_inputs(case, seed, 1, _region_rows(case), case["q_heads"])
        return _attend64(s["q"][0], s["kb"][0], s["vb"][0], s["kp"][0], s["vp"][0], s["table_np"], s["ctx_np"], kind == "region")
    if kind == "prefill":
        s = _prefill_inputs(case, seed)
        L, B, T, Hq, D = s["q"].shape
        G = Hq // case["kv_heads"]
        out = torch.empty(s["q"].shape, dtype=torch.float64, device=DEV)
        hide = torch.ones((T, T), dtype=torch.bool, device=DEV).triu(1)
        for l in range(L):
            for b in range(B):
                for h in range(Hq):
                    x = s["q"][l, b, :, h].double() @ s["k"][l, b, :, h // G].double().T / math.sqrt(D)
                    out[l, b, :, h] = torch.softmax(x.masked_fill_(hide, -math.inf), 1) @ s["v"][l, b, :, h // G].double()
        return dict(out=out, ctx=None, k_pages=None, v_pages=None)
    if kind == "lmhead":
        s = _lmhead_inputs(case, seed)
        st, ids, _ = _stats64(s["hidden"], s["w"], s["draft"])
        return [None if case["sample"] else ids, st]
    if kind == "round":
        s = _round_inputs(case, seed)
        B, K = case["batch"], case["k"]
        rows = torch.full((B, K + 1), -1, dtype=torch.int32, device=DEV)
        rows[:, :K] = s["draft"]
        st, ids, _ = _stats64(s["hidden"], s["w"], rows.view(-1))
        attn = torch.stack([_attend64(s["q"][l], s["kb"][l], s["vb"][l], s["kp"][l], s["vp"][l], s["table_np"], s["ctx_np"], False)
                            for l in range(case["layers"])])
        return dict(attn=attn, argmax=ids, stats=st, p=_policy64(st, ids, s["draft"], s["mlp"], B, K), accept=None, s=None,
                    emitted=None, ctx=None, k_pages=None, v_pages=None)
    if kind == "sps":
        s = _sps_inputs(case, seed)
        B, K = case["batch"], case["k"]
        rows = torch.full((B, K + 1), -1, dtype=torch.int32, device=DEV)
        rows[:, :K] = s["draft"]
        st, ids, x = _stats64(s["hidden"], s["w"], rows.view(-1))
        p = torch.exp(st[:, 4] - st[:, 2]).view(B, K + 1)[:, :K]
        q = torch.gather(s["dq"], 2, s["draft"].long()[..., None])[..., 0].double()
        return dict(argmax=ids, stats=st, logits=x, target=None, accept=None, ratio=(p / q).clamp(max=1.0), s=None, emitted=None,
                    ctx=None, k_pages=None, v_pages=None)
    return _rl64(_rl_inputs(case, seed))
