"""Parity of the CUDA path (through the C ABI) with the CPU oracle on seeded
inputs small enough for the oracle, spanning several tiles, ragged tails and
the degenerate cases (empty context, K = 0, single / many KV splits)."""
import math

import numpy as np
import pytest
import torch

from oracle import cospec_oracle as O
from paper_2605_24793_gb300 import build as BLD
from paper_2605_24793_gb300 import cospec as C
from paper_2605_24793_gb300 import workload as W
from paper_2605_24793_gb300.round import VerifyRound

from .parity_util import assert_close, report_ties, tie_positions

pytestmark = pytest.mark.gpu


@pytest.fixture(scope="module", autouse=True)
def lib():
    C.load_library(BLD.build())
    torch.cuda.set_device(0)
    assert C.get_device_error() == 0
    yield
    assert C.get_device_error() == 0


def bf16(a: np.ndarray) -> torch.Tensor:
    return torch.from_numpy(np.ascontiguousarray(a, dtype=np.float32)).to(torch.bfloat16).cuda()


def host(t: torch.Tensor) -> np.ndarray:
    return t.detach().float().cpu().numpy().astype(np.float64)


def _paged_case(rng, B, R, Hq, Hkv, D, ctx, shuffled, std=1.0, spare_pages=0):
    P = 16
    need = [(c + R + P - 1) // P for c in ctx]
    num = sum(need) + spare_pages
    order = rng.permutation(num) if shuffled else np.arange(num)
    table = np.full((B, max(need)), -1, dtype=np.int32)
    s = 0
    for b in range(B):
        table[b, :need[b]] = order[s:s + need[b]]
        s += need[b]
    mk = lambda *shape: rng.standard_normal(shape).astype(np.float32) * std
    return dict(q=bf16(mk(B, R, Hq, D)), k_blk=bf16(mk(B, R, Hkv, D)), v_blk=bf16(mk(B, R, Hkv, D)),
                k_pages=bf16(mk(num, Hkv, P, D)), v_pages=bf16(mk(num, Hkv, P, D)),
                page_table=torch.from_numpy(table).cuda(),
                ctx_len=torch.tensor(ctx, dtype=torch.int32).cuda(), table_np=table,
                ctx_np=np.array(ctx))


ATTN_CASES = [
    # B, R, Hq, Hkv, D, contexts, shuffled pages
    (1, 6, 32, 8, 128, [4096], False),              # Qwen3-8B-like, many KV splits
    (4, 8, 64, 8, 128, [0, 17, 1000, 3333], True),  # G*R = 64 rows, empty and ragged contexts
    (1, 5, 8, 2, 64, [256], False),                 # head_dim 64
    (3, 3, 4, 4, 128, [5, 64, 65], True),           # G = 1, R = 3 -> 3 rows (one 16-row tile)
    (2, 16, 64, 8, 128, [100, 2000], True),         # G*R = 128 rows: one full row group
    (2, 8, 128, 8, 64, [31, 700], False),           # G = 16 -> 128 rows at head_dim 64
    (2, 1, 32, 8, 128, [0, 1], False),              # K = 0: one row per sequence
    (5, 4, 32, 8, 128, [8191, 40, 63, 64, 2049], True),
    (1, 26, 32, 8, 128, [4096], False),             # K = 25 (the paper's default): 104 rows, one group
    (2, 32, 128, 8, 64, [300, 1500], True),         # 512 rows per KV head: 4 row groups of 128
    (2, 2, 128, 1, 128, [500, 1200], True),         # G = 128 (one KV head): 256 rows, mma.sync
]


def expected_kernel(R, Hq, Hkv, D):
    """More than 32 query rows per KV head (G <= 64, head_dim 64 or 128):
    the tcgen05 kernel (row groups of up to 128 rows); otherwise the
    mma.sync kernel."""
    G = Hq // Hkv
    if G > 64 or D not in (64, 128):
        return C.ATTN_MMA_SYNC
    jb = 128 // G
    return C.ATTN_TCGEN05 if G * min(R, jb) > 32 else C.ATTN_MMA_SYNC

# Batches with a (sequence, KV head, row group) per SM and more than 32 query
# rows per group select the tcgen05 kernel.
_ctx = lambda n, seed: list(np.random.default_rng(seed).integers(0, 700, n))
# Batches above 64 sequences are taken in index order, not longest first.
ATTN_CASES += [
    (80, 6, 32, 8, 128, _ctx(80, 12), True),        # 24 rows: mma.sync kernel
    (70, 16, 32, 8, 128, _ctx(70, 13), True),       # 64 rows: tcgen05 kernel
    (64, 4, 32, 8, 128, _ctx(64, 15), True),        # 64 sequences: the largest batch ranked
    (65, 4, 32, 8, 128, _ctx(65, 16), True),        # 65: the smallest taken in index order
]
ATTN_TC_CASES = [
    (24, 8, 64, 8, 128, [0, 1, 63, 64, 65, 127, 128, 129] + _ctx(16, 1), True),  # G = 8: 64 rows
    (20, 4, 128, 8, 64, _ctx(20, 2), True),         # head_dim 64, G = 16: 64 rows
    (10, 8, 128, 8, 128, _ctx(10, 3), True),        # 128 rows: one full row group
    (20, 8, 40, 8, 128, _ctx(20, 4), False),        # G = 5: 40 rows
    (20, 16, 32, 8, 128, [2000] + _ctx(19, 5), True),  # G = 4, 16 block rows: 64 rows, longer context
    (3, 64, 8, 8, 128, [0, 100, 1500], True),        # R = 64, the largest block: 64 rows
    (2, 64, 16, 8, 64, [50, 700], True),             # R = 64, G = 2: 128 rows, head_dim 64
    (16, 26, 32, 8, 128, _ctx(16, 11), True),        # K = 25 at batch 16: 104 rows, one group
    (2, 32, 32, 8, 128, [600, 129], True),           # K = 31: exactly 128 rows
    (2, 33, 32, 8, 128, [300, 50], True),            # 132 rows: groups of 32 and 1 block rows
    (1, 16, 32, 8, 64, [2000], False),               # head_dim 64 at batch 1: a split of 8
    (2, 3, 64, 1, 128, [400, 1000], True),           # G = 64, the largest: row groups of 2 and 1 block rows
    (3, 11, 24, 8, 128, [129, 700, 0], True),        # G = 3: 33 rows, one past the mma.sync kernel
    (64, 8, 64, 8, 128, _ctx(64, 14), True),         # 64 sequences, ranked longest first
]


@pytest.mark.parametrize("case", ATTN_CASES, ids=lambda c: f"B{c[0]}R{c[1]}G{c[2]//c[3]}D{c[4]}")
def test_verify_attention_matches_oracle(case):
    B, R, Hq, Hkv, D, ctx, shuffled = case
    rng = np.random.default_rng(B * 1000 + R * 100 + Hq + D + sum(ctx))
    t = _paged_case(rng, B, R, Hq, Hkv, D, ctx, shuffled)
    max_ctx = max(ctx)
    assert C.verify_attn_plan(t["q"], t["k_pages"], t["page_table"], max_ctx)[0] == \
        expected_kernel(R, Hq, Hkv, D)
    out = torch.empty_like(t["q"])
    C.verify_attn(t["q"], t["k_blk"], t["v_blk"], t["k_pages"], t["v_pages"], t["page_table"],
                  t["ctx_len"], out, max_ctx)
    ref = O.verify_attention(host(t["q"]), host(t["k_blk"]), host(t["v_blk"]), host(t["k_pages"]),
                             host(t["v_pages"]), t["table_np"], t["ctx_np"], 16)
    assert_close(host(out), ref, "attention")
    # a second call gives the same bits
    out2 = torch.empty_like(out)
    C.verify_attn(t["q"], t["k_blk"], t["v_blk"], t["k_pages"], t["v_pages"], t["page_table"],
                  t["ctx_len"], out2, max_ctx)
    assert torch.equal(out, out2)


@pytest.mark.parametrize("case", ATTN_TC_CASES, ids=lambda c: f"B{c[0]}R{c[1]}G{c[2] // c[3]}D{c[4]}")
def test_verify_attention_tcgen05_matches_oracle(case):
    B, R, Hq, Hkv, D, ctx, shuffled = case
    rng = np.random.default_rng(B * 1000 + R * 100 + Hq + D + int(sum(ctx)))
    t = _paged_case(rng, B, R, Hq, Hkv, D, ctx, shuffled)
    max_ctx = int(max(ctx))
    assert C.verify_attn_plan(t["q"], t["k_pages"], t["page_table"], max_ctx)[0] == C.ATTN_TCGEN05
    out = torch.empty_like(t["q"])
    C.verify_attn(t["q"], t["k_blk"], t["v_blk"], t["k_pages"], t["v_pages"], t["page_table"],
                  t["ctx_len"], out, max_ctx)
    ref = O.verify_attention(host(t["q"]), host(t["k_blk"]), host(t["v_blk"]), host(t["k_pages"]),
                             host(t["v_pages"]), t["table_np"], t["ctx_np"], 16)
    assert_close(host(out), ref, "attention (tcgen05)")
    out2 = torch.empty_like(out)
    C.verify_attn(t["q"], t["k_blk"], t["v_blk"], t["k_pages"], t["v_pages"], t["page_table"],
                  t["ctx_len"], out2, max_ctx)
    assert torch.equal(out, out2)


# The tcgen05 kernel splits a (sequence, head, row group)'s KV range over a
# cluster when the batch has fewer units than SMs, and when a context passes
# 256 tiles of 128 keys: 2, 4 and 8 splits merged through distributed shared
# memory, with most sequences far shorter than the split.
ATTN_TC_SPLIT_CASES = [
    # B, R, Hq, Hkv, D, contexts, shuffled, expected splits
    (12, 8, 64, 8, 128, [6000] + _ctx(11, 8), True, 2),           # 96 units
    (6, 8, 64, 8, 128, [9000, 3000] + _ctx(4, 9), True, 4),       # 48 units
    (1, 8, 64, 8, 128, [6000], False, 12),                        # one wave of 12-CTA clusters
    (20, 8, 64, 8, 128, [33000, 9000] + _ctx(18, 10), False, 2),  # a context past 256 tiles
    # the halves' maxima swapped (D = 128, up to three tiles per CTA) or not, clusters of eight and more or not
    (2, 9, 16, 2, 128, [500, 300], True, 2),                      # two tiles per CTA
    (1, 17, 8, 2, 128, [1537], True, 6),                          # 13 tiles over six
    (2, 17, 8, 2, 64, [2048, 0], True, 8),                        # head_dim 64, two tiles per CTA
    (1, 33, 4, 2, 64, [4000], True, 16),                          # the same, clusters of 16
    (1, 9, 16, 2, 128, [8000], False, 16),                        # four tiles per CTA
]


@pytest.mark.parametrize("case", ATTN_TC_SPLIT_CASES, ids=lambda c: f"B{c[0]}R{c[1]}S{c[7]}")
def test_verify_attention_tcgen05_split_matches_oracle(case):
    B, R, Hq, Hkv, D, ctx, shuffled, splits = case
    rng = np.random.default_rng(B * 1000 + R * 100 + Hq + D + int(sum(ctx)))
    t = _paged_case(rng, B, R, Hq, Hkv, D, ctx, shuffled)
    max_ctx = int(max(ctx))
    assert C.verify_attn_plan(t["q"], t["k_pages"], t["page_table"], max_ctx) == (C.ATTN_TCGEN05, splits)
    out = torch.empty_like(t["q"])
    C.verify_attn(t["q"], t["k_blk"], t["v_blk"], t["k_pages"], t["v_pages"], t["page_table"],
                  t["ctx_len"], out, max_ctx)
    ref = O.verify_attention(host(t["q"]), host(t["k_blk"]), host(t["v_blk"]), host(t["k_pages"]),
                             host(t["v_pages"]), t["table_np"], t["ctx_np"], 16)
    assert_close(host(out), ref, "attention (tcgen05, split)")


# Contexts around the edges of pages, 64-key softmax steps and 128-key tiles.
EDGE_CTX = [0, 1, 15, 16, 63, 64, 65, 100, 127, 128, 129, 191, 192, 193, 255, 300]


@pytest.mark.parametrize("full", [False, True], ids=["causal", "full"])
@pytest.mark.parametrize("R,Hq,Hkv,D,variant", [
    (33, 32, 8, 128, C.ATTN_TWO_TILES),     # 132 rows: the second row tile has four
    (53, 32, 8, 128, C.ATTN_TWO_TILES),     # 212 rows
    (64, 32, 8, 64, C.ATTN_TWO_TILES),      # 256 rows, head_dim 64
    (64, 24, 8, 128, C.ATTN_TWO_TILES),     # G = 3: row tiles of 42 block rows (126 query rows)
    (40, 64, 8, 128, C.ATTN_TWO_TILES),     # G = 8: a group of two row tiles and one of a single tile
    (40, 64, 8, 64, C.ATTN_TWO_TILES),      # the same, head_dim 64
    (20, 32, 8, 128, C.ATTN_ONE_TILE),      # 80 rows, unsplit
    (32, 16, 8, 64, C.ATTN_ONE_TILE),       # 64 rows, head_dim 64
])
def test_verify_attention_tile_edges(R, Hq, Hkv, D, variant, full):
    """One and two row tiles per CTA at every key remainder (more than 128 rows on 128 or more
    (sequence, head) units of a few tiles take two).  bf16 outputs of probabilities rounded to bf16:
    the usual tolerance."""
    B = len(EDGE_CTX)
    rng = np.random.default_rng(R * 100 + Hq + D)
    t = _paged_case(rng, B, R, Hq, Hkv, D, EDGE_CTX, True)
    assert C.verify_attn_plan(t["q"], t["k_pages"], t["page_table"], max(EDGE_CTX)) == (C.ATTN_TCGEN05, 1)
    assert C.verify_attn_variant(t["q"], t["k_pages"], t["page_table"], max(EDGE_CTX)) == variant
    out = torch.empty_like(t["q"])
    C.verify_attn(t["q"], t["k_blk"], t["v_blk"], t["k_pages"], t["v_pages"], t["page_table"],
                  t["ctx_len"], out, max(EDGE_CTX), block_full=full)
    ref = O.verify_attention(host(t["q"]), host(t["k_blk"]), host(t["v_blk"]), host(t["k_pages"]),
                             host(t["v_pages"]), t["table_np"], t["ctx_np"], 16,
                             **({"block_mask": "full"} if full else {}))
    assert_close(host(out), ref, "attention (tile edges)")
    assert C.get_device_error() == 0


@pytest.mark.parametrize("R", [20, 53])
def test_verify_attention_moving_maximum(R):
    """Scores that grow along the context move the reference maximum (and rescale the outputs) tile
    after tile, in one half of the keys and not the other."""
    B, Hq, Hkv, D = 16, 32, 8, 128
    ctx = [40 * (i + 1) for i in range(B)]
    rng = np.random.default_rng(R)
    t = _paged_case(rng, B, R, Hq, Hkv, D, ctx, False)
    table = t["table_np"]
    for b in range(B):
        for pos in range(ctx[b]):
            scale = 0.2 + 0.02 * pos if (pos // 64) % 2 == 0 else 0.1
            t["k_pages"][int(table[b, pos // 16]), :, pos % 16] *= scale
    t["q"] *= 2
    out = torch.empty_like(t["q"])
    C.verify_attn(t["q"], t["k_blk"], t["v_blk"], t["k_pages"], t["v_pages"], t["page_table"],
                  t["ctx_len"], out, max(ctx))
    ref = O.verify_attention(host(t["q"]), host(t["k_blk"]), host(t["v_blk"]), host(t["k_pages"]),
                             host(t["v_pages"]), t["table_np"], t["ctx_np"], 16)
    assert_close(host(out), ref, "attention (moving maximum)")


# The arbitrator's draft/target region (Sec. 3.3): 2K+3 block rows that see
# the whole block; K = 7 gives 17 rows, K = 25 (the paper's default) 53.
ATTN_FULL_CASES = [
    # B, R, Hq, Hkv, D, contexts, shuffled, expected kernel
    (1, 17, 32, 8, 128, [4096], False, 1),          # K = 7 region on a Qwen3-4B-like arbitrator
    (3, 53, 32, 8, 128, [0, 300, 2500], True, 1),   # K = 25 region: 212 rows in groups of 128 and 84
    (2, 4, 128, 1, 128, [700, 90], True, 0),        # G = 128: 512 rows in 64-row groups, mma.sync
    (2, 9, 16, 8, 64, [100, 33], True, 0),          # head_dim 64, K = 3 region
    (20, 53, 8, 8, 128, _ctx(20, 6), True, 1),      # G = 1, 53 rows per group: tcgen05 kernel
    (24, 17, 32, 8, 128, _ctx(24, 7), True, 1),     # G = 4, 68 rows in one group: tcgen05 kernel
    (2, 64, 8, 8, 128, [300, 0], True, 1),          # a 64-row region, the largest block
]


@pytest.mark.parametrize("case", ATTN_FULL_CASES, ids=lambda c: f"B{c[0]}R{c[1]}G{c[2] // c[3]}D{c[4]}")
def test_verify_attention_full_block_matches_oracle(case):
    B, R, Hq, Hkv, D, ctx, shuffled, kernel = case
    rng = np.random.default_rng(B * 1000 + R * 100 + Hq + D + int(sum(ctx)) + 77)
    t = _paged_case(rng, B, R, Hq, Hkv, D, ctx, shuffled)
    max_ctx = int(max(ctx))
    assert C.verify_attn_plan(t["q"], t["k_pages"], t["page_table"], max_ctx)[0] == kernel
    out = torch.empty_like(t["q"])
    C.verify_attn(t["q"], t["k_blk"], t["v_blk"], t["k_pages"], t["v_pages"], t["page_table"],
                  t["ctx_len"], out, max_ctx, block_full=True)
    ref = O.verify_attention(host(t["q"]), host(t["k_blk"]), host(t["v_blk"]), host(t["k_pages"]),
                             host(t["v_pages"]), t["table_np"], t["ctx_np"], 16, block_mask="full")
    assert_close(host(out), ref, "attention (full block)")
    # the causal call on the same inputs still matches the causal oracle
    C.verify_attn(t["q"], t["k_blk"], t["v_blk"], t["k_pages"], t["v_pages"], t["page_table"],
                  t["ctx_len"], out, max_ctx)
    ref_c = O.verify_attention(host(t["q"]), host(t["k_blk"]), host(t["v_blk"]), host(t["k_pages"]),
                               host(t["v_pages"]), t["table_np"], t["ctx_np"], 16)
    assert_close(host(out), ref_c, "attention (causal, long block)")


def test_verify_attention_split_count_does_not_change_result_beyond_tolerance():
    rng = np.random.default_rng(3)
    t = _paged_case(rng, 2, 6, 32, 8, 128, [3000, 5000], True)
    ref = O.verify_attention(host(t["q"]), host(t["k_blk"]), host(t["v_blk"]), host(t["k_pages"]),
                             host(t["v_pages"]), t["table_np"], t["ctx_np"], 16)
    for max_ctx in (5000, t["table_np"].shape[1] * 16):     # different split plans
        out = torch.empty_like(t["q"])
        C.verify_attn(t["q"], t["k_blk"], t["v_blk"], t["k_pages"], t["v_pages"], t["page_table"],
                      t["ctx_len"], out, max_ctx)
        assert_close(host(out), ref, f"attention max_ctx={max_ctx}")


def test_verify_attention_constant_values():
    # closed form: constant V gives that constant whatever the scores
    rng = np.random.default_rng(4)
    t = _paged_case(rng, 2, 6, 32, 8, 128, [777, 3], True)
    t["v_pages"].fill_(0.375)
    t["v_blk"].fill_(0.375)
    out = torch.empty_like(t["q"])
    C.verify_attn(t["q"], t["k_blk"], t["v_blk"], t["k_pages"], t["v_pages"], t["page_table"],
                  t["ctx_len"], out, 777)
    assert torch.all(out.float() == 0.375)


def test_verify_attention_concurrent_host_threads():
    # Calls from several host threads (ctypes releases the GIL), each on its
    # own stream and with its own block size, so that first launches race to
    # set each variant's shared-memory limit: every result equals the same
    # call made alone.
    import threading
    rng = np.random.default_rng(11)
    shapes = [(2, 4, 32, 8, 128, [900, 40]), (1, 20, 32, 8, 128, [1500]),
              (2, 40, 16, 8, 128, [300, 700]), (3, 8, 64, 8, 128, [100, 2000, 5])]
    cases = [_paged_case(rng, *sh, True) for sh in shapes]
    refs = []
    for sh, t in zip(shapes, cases):
        out = torch.empty_like(t["q"])
        C.verify_attn(t["q"], t["k_blk"], t["v_blk"], t["k_pages"], t["v_pages"], t["page_table"],
                      t["ctx_len"], out, max(sh[5]))
        refs.append(out)
    torch.cuda.synchronize()
    outs = [torch.empty_like(t["q"]) for t in cases]
    errors = []

    def worker(i):
        try:
            s = torch.cuda.Stream()
            t = cases[i]
            for _ in range(20):
                C.verify_attn(t["q"], t["k_blk"], t["v_blk"], t["k_pages"], t["v_pages"], t["page_table"],
                              t["ctx_len"], outs[i], max(shapes[i][5]), stream=s)
            s.synchronize()
        except Exception as e:  # noqa: BLE001 - reported below
            errors.append(e)

    threads = [threading.Thread(target=worker, args=(i,)) for i in range(len(cases))]
    for th in threads:
        th.start()
    for th in threads:
        th.join()
    assert not errors, errors
    for ref, out in zip(refs, outs):
        assert torch.equal(ref, out)


LM_CASES = [
    # M, d, V, weight std
    (1, 64, 128, 0.1),
    (5, 512, 4096, 0.02),
    (6, 4096, 151936, 0.02),      # Qwen3-8B LM head, batch 1, K = 5
    (17, 256, 1000, 0.1),         # vocabulary not a multiple of the 128-row tile
    (128, 1024, 3000, 0.05),
    (300, 128, 2048, 0.1),        # two passes of 160 and 140 rows
    (256, 5120, 1280, 0.02),
    (384, 256, 3000, 0.05),       # two equal passes of 192 rows (the Llama K = 5 round)
    (512, 256, 2000, 0.05),       # two full 256-row passes
    (520, 128, 1500, 0.1),        # three passes of 176, 176 and 168 rows
]


@pytest.mark.parametrize("case", LM_CASES, ids=lambda c: f"M{c[0]}d{c[1]}V{c[2]}")
def test_lmhead_matches_oracle(case):
    M, d, V, wstd = case
    rng = np.random.default_rng(M * 7 + d + V)
    hidden = bf16(rng.standard_normal((M, d)))
    w = bf16(rng.standard_normal((V, d)) * wstd)
    dfr = rng.integers(0, V, M).astype(np.int32)
    dfr[::3] = -1
    dfr_t = torch.from_numpy(dfr).cuda()
    am = torch.empty(M, dtype=torch.int32, device="cuda")
    st = torch.empty((M, 5), dtype=torch.float32, device="cuda")
    ws = C.new_lmhead_workspace(M, d, V)
    C.lmhead_argmax_features(hidden, w, dfr_t, am, st, ws)
    ref_am, ref_st = O.lmhead_stats(host(hidden), host(w), dfr)
    assert_close(st.cpu().numpy(), ref_st, "lm-head stats")
    margin = ref_st[:, 0] - ref_st[:, 1]
    clear = margin >= 1e-3
    assert np.array_equal(am.cpu().numpy()[clear], ref_am[clear])
    print(f"lm-head {case}: tie rows {(~clear).sum()}")


@pytest.mark.parametrize("M,d,V", [
    (2, 64, 1),            # one id: no second logit
    (31, 64, 100),         # the second CTA of the pair has no vocabulary row
    (33, 128, 129),        # a second 32-column chunk; one id for the second CTA
    (65, 192, 257),        # three chunks; a second vocabulary tile of one id
    (257, 64, 300),        # two row slices sharing one launch
    (1030, 64, 513),       # five slices: two launches of three and two
])
def test_lmhead_tile_and_slice_edges(M, d, V):
    """Statistics, ids, logits and samples at the edges of the 256-id tiles, the 32-row chunks and the
    row slices.  The logits are 32-bit sums of exact products (error below d ulps of the largest term
    sum, far under the usual tolerance), so ids are compared outside near ties."""
    rng = np.random.default_rng(M + d + V)
    hidden, w = bf16(rng.standard_normal((M, d))), bf16(rng.standard_normal((V, d)) * 0.2)
    dfr = rng.integers(-1, V, M).astype(np.int32)
    dfr_t = torch.from_numpy(dfr).cuda()
    ids = torch.empty(M, dtype=torch.int32, device="cuda")
    st = torch.empty((M, 5), dtype=torch.float32, device="cuda")
    ws = C.new_lmhead_workspace(M, d, V)
    x = O.lmhead_logits(host(hidden), host(w))
    with np.errstate(all="ignore"):
        ref_am, ref_st = O.lmhead_stats(host(hidden), host(w), dfr)
    if V == 1:
        ref_st[:, 1] = -np.inf
        ref_st[:, 3] = 0.0
    clear = ref_st[:, 0] - ref_st[:, 1] >= 1e-3
    logits = torch.empty((M, V), dtype=torch.float32, device="cuda")
    for mode in ("greedy", "logits"):
        if mode == "greedy":
            C.lmhead_argmax_features(hidden, w, dfr_t, ids, st, ws)
        else:
            C.lmhead_logits_features(hidden, w, dfr_t, 1.0, ids, st, logits, ws)
            assert_close(logits.cpu().numpy(), x, "logits")
        got = st.cpu().numpy()
        assert np.array_equal(np.isinf(got[:, 1]), np.isinf(ref_st[:, 1]))
        fin = ref_st.copy()
        fin[:, 1] = np.where(np.isinf(fin[:, 1]), 0, fin[:, 1])
        got[:, 1] = np.where(np.isinf(got[:, 1]), 0, got[:, 1])
        assert_close(got, fin, f"{mode} stats")
        assert np.array_equal(ids.cpu().numpy()[clear], ref_am[clear])
    seed = 0x5DEECE66D1234567
    C.lmhead_sample_features(hidden, w, dfr_t, 1.0, torch.tensor([seed], dtype=torch.int64, device="cuda"), ids, st, ws)
    keys = O.gumbel_keys(x, seed, 1.0)
    sure = np.ones(M, bool) if V == 1 else np.diff(np.sort(keys, axis=1)[:, -2:], axis=1)[:, 0] >= 1e-3
    assert np.array_equal(ids.cpu().numpy()[sure], np.argmax(keys, axis=1)[sure])
    assert C.get_device_error() == 0


def test_lmhead_extreme_logits():
    """Equal logits and a logit near the largest float keep well-defined statistics; NaN is passed on."""
    M, d, V = 40, 64, 700
    hidden = np.zeros((M, d), np.float32)
    w = np.zeros((V, d), np.float32)
    w[:, 0] = 1.0
    w[7, 1] = 1.0                       # the only id that sees column 1
    hidden[1, 0] = 3.0                  # all logits 3
    hidden[2, 1] = 1e38                 # one huge logit: the others underflow
    hidden[3, 1] = np.inf               # inf * 0: NaN logits beside an infinite one
    hidden[4, 2] = 1e38
    w[650, 2] = 1e38                    # overflows to one infinite logit in row 4
    hidden_t, w_t = bf16(hidden), bf16(w)
    ids = torch.empty(M, dtype=torch.int32, device="cuda")
    st = torch.empty((M, 5), dtype=torch.float32, device="cuda")
    C.lmhead_argmax_features(hidden_t, w_t, torch.full((M,), 7, dtype=torch.int32, device="cuda"), ids, st,
                             C.new_lmhead_workspace(M, d, V))
    ids, st = ids.cpu().numpy(), st.cpu().numpy()
    assert ids[0] == 0 and ids[1] == 0 and ids[2] == 7
    np.testing.assert_allclose(st[0, :4], [0, 0, np.log(V), np.log(V)], rtol=1e-6)
    np.testing.assert_allclose(st[1], [3, 3, 3 + np.log(V), np.log(V), 3], rtol=1e-6)
    np.testing.assert_allclose(st[2], [st[2, 4], 0, st[2, 4], 0, st[2, 4]], rtol=1e-6)
    assert np.isnan(st[3, 2])           # NaN logits reach the log-sum-exp
    assert ids[4] == 650 and st[4, 0] == np.inf and st[4, 2] == np.inf
    assert C.get_device_error() == 0


def test_lmhead_exact_ties_pick_lowest_id():
    rng = np.random.default_rng(11)
    M, d, V = 8, 256, 700
    hidden = rng.standard_normal((M, d))
    w = rng.standard_normal((V, d)) * 0.01
    w[[3, 130, 699]] = hidden[0] * 0.5          # three identical top rows for row 0
    w[[257, 258]] = hidden[1] * 0.5             # two identical top rows for row 1
    hidden_t, w_t = bf16(hidden), bf16(w)
    am = torch.empty(M, dtype=torch.int32, device="cuda")
    st = torch.empty((M, 5), dtype=torch.float32, device="cuda")
    C.lmhead_argmax_features(hidden_t, w_t, torch.full((M,), -1, dtype=torch.int32, device="cuda"),
                             am, st, C.new_lmhead_workspace(M, d, V))
    am = am.cpu().numpy()
    st = st.cpu().numpy()
    assert am[0] == 3 and am[1] == 257
    assert st[0, 0] == st[0, 1] and st[1, 0] == st[1, 1]      # second == max on a tie
    assert np.all(np.isnan(st[:, 4]))


def _stats_case(rng, B, K, V=64):
    x = rng.standard_normal((B * (K + 1), V)) * 2.0
    top1 = np.argmax(x, axis=1).reshape(B, K + 1)
    draft = np.where(rng.random((B, K)) < 0.5, top1[:, :K], rng.integers(0, V, (B, K))).astype(np.int32)
    dfr = np.full((B, K + 1), -1)
    dfr[:, :K] = draft
    am, st = O.row_stats(x, dfr.reshape(-1))
    return draft, am.reshape(B, K + 1).astype(np.int32), st.reshape(B, K + 1, 5)


@pytest.mark.parametrize("K", [1, 3, 7, 31])
@pytest.mark.parametrize("mode", [0, 1, 2])
@pytest.mark.parametrize("lam", [0.4, 0.6, 0.8])
def test_arbitrate_matches_oracle(K, mode, lam):
    rng = np.random.default_rng(K * 100 + mode * 10 + int(lam * 10))
    B, H = 37, 256
    draft, am, st = _stats_case(rng, B, K)
    w1 = (rng.random((H, 8)) * 2 - 1) / math.sqrt(8)
    b1 = (rng.random(H) * 2 - 1) / math.sqrt(8)
    w2 = (rng.random(H) * 2 - 1) / math.sqrt(H)
    b2 = 0.05
    ref_p, ref_a = O.arbitrate(draft, am, st, w1, b1, w2, b2, lam, mode)
    p = torch.empty((B, K), dtype=torch.float32, device="cuda")
    a = torch.empty((B, K), dtype=torch.uint8, device="cuda")
    f32 = lambda v: torch.tensor(np.asarray(v, dtype=np.float32)).cuda()
    C.arbitrate(torch.from_numpy(draft).cuda(), torch.from_numpy(am).cuda(),
                f32(st), f32(w1), f32(b1), f32(w2), b2, lam, mode, p, a)
    p = p.cpu().numpy()
    a = a.cpu().numpy()
    assert_close(p, ref_p, "policy probability")
    clear = np.abs(ref_p - lam) >= 1e-3
    assert np.array_equal(a[clear], ref_a[clear])
    assert np.all(a[draft == am[:, :K]] == 1)


def test_features_feed_the_mlp_as_the_oracle_builds_them():
    # a one-hot first layer exposes each feature in turn through z
    rng = np.random.default_rng(21)
    B, K = 9, 7
    draft, am, st = _stats_case(rng, B, K)
    feats = O.arbitration_features(draft, am, st)
    mism = draft != am[:, :K]
    for k in range(8):
        w1 = np.zeros((2, 8)); w1[0, k] = 1.0; w1[1, k] = -1.0
        b1 = np.zeros(2); w2 = np.array([1.0, -1.0])           # z = relu(f) - relu(-f) = f_k
        p = torch.empty((B, K), dtype=torch.float32, device="cuda")
        a = torch.empty((B, K), dtype=torch.uint8, device="cuda")
        f32 = lambda v: torch.tensor(np.asarray(v, dtype=np.float32)).cuda()
        C.arbitrate(torch.from_numpy(draft).cuda(), torch.from_numpy(am).cuda(), f32(st), f32(w1),
                    f32(b1), f32(w2), 0.0, 0.5, 0, p, a)
        z = -np.log(1.0 / np.clip(p.cpu().numpy().astype(np.float64), 1e-30, 1 - 1e-7) - 1.0)
        assert_close(z[mism], feats[..., k][mism], f"feature F{k}", abs_tol=1e-3, rel_tol=1e-3)


@pytest.mark.parametrize("K,L,B", [(0, 3, 6), (1, 3, 6), (5, 3, 6), (7, 3, 6), (7, 64, 32)])
def test_accept_commit_matches_oracle(K, L, B):
    # (7, 64, 32): the commit grid of the Qwen3-32B-shaped round (64 layers x
    # 32 sequences, one CTA each), with short contexts
    rng = np.random.default_rng(40 + K + L)
    R, Hkv, D, P = K + 1, 8, 128, 16
    ctx = rng.integers(0, 200, B).astype(np.int32)
    need = (ctx + R + P - 1) // P
    num = int(need.sum())
    perm = rng.permutation(num)
    table = np.full((B, need.max()), -1, dtype=np.int32)
    s0 = 0
    for b in range(B):
        table[b, :need[b]] = perm[s0:s0 + need[b]]
        s0 += need[b]
    V = 50
    am = rng.integers(0, V, (B, R)).astype(np.int32)
    draft = np.where(rng.random((B, K)) < 0.6, am[:, :K], rng.integers(0, V, (B, K))).astype(np.int32)
    acc = (rng.random((B, K)) < 0.5).astype(np.uint8)
    acc[draft == am[:, :K]] = 1
    kb = bf16(rng.standard_normal((L, B, R, Hkv, D)))
    vb = bf16(rng.standard_normal((L, B, R, Hkv, D)))
    kp = bf16(rng.standard_normal((L, num, Hkv, P, D)))
    vp = bf16(rng.standard_normal((L, num, Hkv, P, D)))
    bits = lambda t: t.cpu().view(torch.int16).numpy()
    kp0, vp0 = bits(kp), bits(vp)
    ctx_t = torch.from_numpy(ctx).cuda()
    alen = torch.empty(B, dtype=torch.int32, device="cuda")
    em = torch.empty((B, R), dtype=torch.int32, device="cuda")
    C.accept_commit(torch.from_numpy(draft.reshape(B, K)).cuda(), torch.from_numpy(am).cuda(),
                    torch.from_numpy(acc.reshape(B, K)).cuda(), kb, vb, kp, vp,
                    torch.from_numpy(table).cuda(), ctx_t, alen, em)
    s, emitted = O.accept_scan(draft.reshape(B, K), am, acc.reshape(B, K))
    kp_ref, vp_ref, ctx_ref = O.commit_kv(bits(kb), bits(vb), kp0, vp0, table, ctx, s, P)
    assert np.array_equal(alen.cpu().numpy(), s)
    assert np.array_equal(em.cpu().numpy(), emitted)
    assert np.array_equal(ctx_t.cpu().numpy(), ctx_ref)
    assert np.array_equal(bits(kp), kp_ref) and np.array_equal(bits(vp), vp_ref)


def _tiny_round(mode, lam, cfg_name="tiny", **over):
    cfg = W.CONFIGS[cfg_name].replace(**over) if over else W.CONFIGS[cfg_name]
    inp = W.make_round_inputs(cfg, device="cuda")
    hostinp = {k: (v.cpu() if torch.is_tensor(v) else v) for k, v in inp.items()}
    x = O.lmhead_logits(hostinp["hidden"], hostinp["w"])
    draft = W.synth_drafts(cfg, O.topk_ids(x, 8).reshape(cfg.batch, cfg.rows, 8))
    ref = O.cospec_round(hostinp, draft, lam, mode)
    rnd = VerifyRound(inp, draft, lam, mode, keep_attn=True)
    rnd.run(restore=False)
    torch.cuda.synchronize()
    return cfg, draft, ref, rnd


def _check_round(cfg, draft, ref, rnd, lam):
    for l in range(cfg.layers):
        assert_close(host(rnd.attn_out[l]), ref["attn"][l], f"attention layer {l}")
    B, R, K = cfg.batch, cfg.rows, cfg.k
    st = rnd.stats.cpu().numpy().reshape(B, R, 5)
    assert_close(st, ref["stats"], "lm-head stats")
    s_gpu = rnd.accept_len.cpu().numpy()
    ties = tie_positions(ref["stats"], draft, ref["argmax"], ref["p"], ref["s"], s_gpu, lam)
    report_ties("round parity", f"{cfg.name} K={K} lambda={lam}", ties)
    tie = ties > 0
    ok = ~tie
    am = rnd.argmax.cpu().numpy().reshape(B, R)
    assert np.array_equal(am[ok], ref["argmax"][ok])
    if K > 0:
        assert_close(rnd.p.cpu().numpy()[ok], ref["p"][ok], "policy probability")
        assert np.array_equal(rnd.accept.cpu().numpy()[ok], ref["a"][ok])
    assert np.array_equal(s_gpu[ok], ref["s"][ok])
    assert np.array_equal(rnd.emitted.cpu().numpy()[ok], ref["emitted"][ok])
    assert np.array_equal(rnd.ctx_len.cpu().numpy()[ok], ref["ctx_len"][ok])
    kp = rnd.k_pages.cpu().view(torch.int16).numpy()
    vp = rnd.v_pages.cpu().view(torch.int16).numpy()
    table = rnd.inp["page_table_np"]
    for b in np.nonzero(ok)[0]:
        pages = table[b][table[b] >= 0]
        assert np.array_equal(kp[:, pages], ref["k_pages"][:, pages])
        assert np.array_equal(vp[:, pages], ref["v_pages"][:, pages])
    return int(tie.sum())


@pytest.mark.parametrize("mode", [0, 1, 2])
def test_tiny_round_matches_oracle(mode):
    cfg, draft, ref, rnd = _tiny_round(mode, 0.6)
    assert _check_round(cfg, draft, ref, rnd, 0.6) == 0
    if mode == 1:
        assert np.array_equal(ref["s"], O.strict_spd_length(draft, ref["argmax"]))
    if mode == 2:
        assert np.all(ref["s"] == cfg.k + 1)


def test_small_batched_round_with_n01_inputs():
    # several sequences, three layers, shuffled pages, N(0,1) attention inputs
    cfg, draft, ref, rnd = _tiny_round(0, 0.6, batch=6, ctx_lo=0, ctx_hi=700, layers=3,
                                       qkv_std=1.0, shuffled_pages=True, k=7, mismatch_rate=0.5)
    ties = _check_round(cfg, draft, ref, rnd, 0.6)
    print(f"tie-affected sequences: {ties} of {cfg.batch}")


def test_packed_step_buffers_give_the_same_round():
    # The packed host-facing buffers rebind the inputs and results as views;
    # a replayed graph over them must reproduce the unpacked round bit for bit.
    cfg = W.CONFIGS["tiny"].replace(batch=5, ctx_lo=0, ctx_hi=900, layers=2, k=7,
                                    shuffled_pages=True, mismatch_rate=0.5)
    inp_ref = W.make_round_inputs(cfg, device="cuda")
    x = O.lmhead_logits(inp_ref["hidden"].cpu(), inp_ref["w"].cpu())
    draft = W.synth_drafts(cfg, O.topk_ids(x, 8).reshape(cfg.batch, cfg.rows, 8))
    plain = VerifyRound(inp_ref, draft, 0.6, 0, keep_attn=True)
    plain.replay()
    packed = VerifyRound(W.make_round_inputs(cfg, device="cuda"), draft, 0.6, 0, keep_attn=True)
    packed.pack_step_io()
    assert packed.q.data_ptr() == packed.io_in.data_ptr()
    for name in ("q", "k_blk", "v_blk", "hidden", "draft", "draft_for_row"):
        t = getattr(packed, name)
        assert t.data_ptr() % 256 == 0 and torch.equal(t.cpu(), getattr(plain, name).cpu())
    packed.replay()
    packed.replay()         # the graph restores the context: a second replay is the same round
    torch.cuda.synchronize()
    assert packed.accept_len.data_ptr() == packed.io_out.data_ptr()
    for name in ("accept_len", "emitted", "argmax", "stats", "p", "accept", "ctx_len",
                 "attn_out", "k_pages", "v_pages"):
        a, b = getattr(plain, name).cpu(), getattr(packed, name).cpu()
        assert torch.equal(a.view(torch.uint8) if a.is_floating_point() else a,
                           b.view(torch.uint8) if b.is_floating_point() else b), name
    B, R = cfg.batch, cfg.rows
    lead = (B + 63) // 64 * 64
    out = packed.io_out.cpu()
    assert torch.equal(out[:B], plain.accept_len.cpu())
    assert torch.equal(out[lead:].view(B, R), plain.emitted.cpu())


def test_block_size_one_round_is_greedy():
    cfg, draft, ref, rnd = _tiny_round(0, 0.6, k=0, batch=3, ctx_lo=10, ctx_hi=300)
    assert np.all(rnd.accept_len.cpu().numpy() == 1)
    em = rnd.emitted.cpu().numpy()
    x = O.lmhead_logits(rnd.hidden.cpu(), rnd.w.cpu())
    assert np.array_equal(em[:, 0], np.argmax(x, axis=1))
    _check_round(cfg, draft, ref, rnd, 0.6)


def test_device_checks_set_error_bits_without_faulting():
    rng = np.random.default_rng(5)
    t = _paged_case(rng, 2, 6, 32, 8, 128, [100, 200], False)
    out = torch.empty_like(t["q"])
    bad = t["page_table"].clone()
    bad[1, 3] = 10 ** 6                                    # page id outside the pool
    C.verify_attn(t["q"], t["k_blk"], t["v_blk"], t["k_pages"], t["v_pages"], bad, t["ctx_len"],
                  out, 200)
    assert C.get_device_error() & C.DEVERR_PAGE
    long_ctx = torch.tensor([100, t["table_np"].shape[1] * 16 + 1], dtype=torch.int32, device="cuda")
    C.verify_attn(t["q"], t["k_blk"], t["v_blk"], t["k_pages"], t["v_pages"], t["page_table"],
                  long_ctx, out, 200)
    assert C.get_device_error() & C.DEVERR_CTX
    M, d, V = 4, 128, 256
    C.lmhead_argmax_features(bf16(rng.standard_normal((M, d))), bf16(rng.standard_normal((V, d))),
                             torch.tensor([0, V, -1, 5], dtype=torch.int32, device="cuda"),
                             torch.empty(M, dtype=torch.int32, device="cuda"),
                             torch.empty((M, 5), dtype=torch.float32, device="cuda"),
                             C.new_lmhead_workspace(M, d, V))
    assert C.get_device_error() == C.DEVERR_TOKEN
    assert C.get_device_error() == 0                       # reading clears the word


def test_tcgen05_attention_device_checks_skip_only_the_bad_sequence():
    # 64 query rows per KV head: the tcgen05 kernel.  A page id outside the
    # pool (clamped to page 0 for the copy) and a context past the page table
    # (no tiles at all) each set their bit; the other sequence's rows still
    # match the oracle.
    rng = np.random.default_rng(6)
    t = _paged_case(rng, 2, 16, 32, 8, 128, [700, 300], True)
    assert C.verify_attn_plan(t["q"], t["k_pages"], t["page_table"], 700)[0] == C.ATTN_TCGEN05
    ref = O.verify_attention(host(t["q"]), host(t["k_blk"]), host(t["v_blk"]), host(t["k_pages"]),
                             host(t["v_pages"]), t["table_np"], t["ctx_np"], 16)
    out = torch.empty_like(t["q"])
    bad = t["page_table"].clone()
    bad[1, 5] = 10 ** 6
    C.verify_attn(t["q"], t["k_blk"], t["v_blk"], t["k_pages"], t["v_pages"], bad, t["ctx_len"],
                  out, 700)
    assert C.get_device_error() == C.DEVERR_PAGE
    assert_close(host(out)[0], ref[0], "attention (tcgen05), the sequence with valid pages")
    long_ctx = torch.tensor([700, t["table_np"].shape[1] * 16 + 1], dtype=torch.int32, device="cuda")
    out.fill_(1.0)
    C.verify_attn(t["q"], t["k_blk"], t["v_blk"], t["k_pages"], t["v_pages"], t["page_table"],
                  long_ctx, out, 700)
    assert C.get_device_error() == C.DEVERR_CTX
    assert_close(host(out)[0], ref[0], "attention (tcgen05), the sequence with a valid context")
    assert torch.all(out[1] == 0)                          # the skipped sequence attends nothing


# Both sides of the rule for one launch or two: clusters of 1, 3, 8 and 8 (of two layers each) CTAs, the same
# with too many CTAs or layers.
@pytest.mark.parametrize("B,L,K,Hkv,launches", [
    (3, 1, 4, 2, 1), (5, 3, 31, 8, 1), (4, 8, 7, 2, 1), (8, 16, 3, 2, 1), (2, 11, 0, 2, 1),
    (9, 9, 3, 2, 2), (2, 17, 7, 2, 2), (110, 3, 2, 2, 2)])
def test_accept_commit_launches_one_kernel_or_two(B, L, K, Hkv, launches):
    rng = np.random.default_rng(B * 100 + L)
    D, P, R, V = 64, 16, K + 1, 9
    pages = 3
    num = B * pages
    table = rng.permutation(num).astype(np.int32).reshape(B, pages)
    ctx = rng.integers(0, pages * P - R + 1, B).astype(np.int32)
    am = rng.integers(0, V, (B, R)).astype(np.int32)
    draft = np.where(rng.random((B, K)) < 0.6, am[:, :K], rng.integers(0, V, (B, K))).astype(np.int32)
    acc = rng.integers(0, 2, (B, K)).astype(np.uint8)
    kb, vb = bf16(rng.standard_normal((L, B, R, Hkv, D))), bf16(rng.standard_normal((L, B, R, Hkv, D)))
    kp, vp = bf16(rng.standard_normal((L, num, Hkv, P, D))), bf16(rng.standard_normal((L, num, Hkv, P, D)))
    bits = lambda x: x.cpu().view(torch.int16).numpy()
    kp0, vp0 = bits(kp), bits(vp)
    dims = C.AttnDims(B, R, Hkv, Hkv, D, P, pages, num, 0.0, 0)
    assert C.accept_commit_launches(dims, L) == launches
    ctx_t, alen = torch.from_numpy(ctx).cuda(), torch.empty(B, dtype=torch.int32, device="cuda")
    am_t = torch.from_numpy(am).cuda()
    # the emitted tokens may take the place of the target's
    C.accept_commit(torch.from_numpy(draft).cuda(), am_t, torch.from_numpy(acc).cuda(), kb, vb, kp, vp,
                    torch.from_numpy(table).cuda(), ctx_t, alen, am_t)
    s, emitted = O.accept_scan(draft, am, acc)
    kp_ref, vp_ref, ctx_ref = O.commit_kv(bits(kb), bits(vb), kp0, vp0, table, ctx, s, P)
    assert np.array_equal(alen.cpu().numpy(), s) and np.array_equal(am_t.cpu().numpy(), emitted)
    assert np.array_equal(ctx_t.cpu().numpy(), ctx_ref)
    assert np.array_equal(bits(kp), kp_ref) and np.array_equal(bits(vp), vp_ref)
    assert C.get_device_error() == 0


def test_accept_commit_without_layers_takes_any_batch():
    B, K = 70000, 3
    z = lambda *sh: torch.zeros(sh, dtype=torch.int32, device="cuda")
    kv, pool = (torch.zeros(sh, dtype=torch.bfloat16, device="cuda") for sh in ((0, B, K + 1, 2, 64), (1, 1, 2, 16, 64)))
    ctx, alen, em = z(B), z(B), z(B, K + 1)
    accept = torch.ones((B, K), dtype=torch.uint8, device="cuda")
    accept[B - 1, 1] = 0
    draft = z(B, K)
    draft[B - 1, 1] = 5
    C.accept_commit(draft, z(B, K + 1), accept, kv, kv.clone(), pool, pool.clone(), z(B, 1), ctx, alen, em)
    assert C.get_device_error() == 0
    assert (ctx[:-1] == K + 1).all() and int(ctx[-1]) == 2 and torch.equal(ctx, alen)
    assert em[-1].tolist() == [0, 0, -1, -1]


def test_accept_commit_device_checks_skip_only_the_bad_sequence():
    # Sequence 1 would run past its page table (ctx + s > capacity): its
    # context stays, nothing of it is written.  Sequence 2's commit page is
    # outside the pool: those cells are skipped.  Sequence 0 commits exactly
    # as the oracle does.
    rng = np.random.default_rng(41)
    B, K, L, Hkv, D, P = 3, 3, 2, 8, 128, 16
    R = K + 1
    pages_per_seq = 4
    table = rng.permutation(B * pages_per_seq).astype(np.int32).reshape(B, pages_per_seq)
    ctx = np.array([37, pages_per_seq * P - 2, 21], dtype=np.int32)
    table_bad = table.copy()
    table_bad[2, ctx[2] // P] = 10 ** 6
    V = 50
    am = rng.integers(0, V, (B, R)).astype(np.int32)
    draft = am[:, :K].copy()                               # every draft matches: s = K + 1
    acc = np.ones((B, K), dtype=np.uint8)
    num = B * pages_per_seq
    kb = bf16(rng.standard_normal((L, B, R, Hkv, D)))
    vb = bf16(rng.standard_normal((L, B, R, Hkv, D)))
    kp = bf16(rng.standard_normal((L, num, Hkv, P, D)))
    vp = bf16(rng.standard_normal((L, num, Hkv, P, D)))
    bits = lambda x: x.cpu().view(torch.int16).numpy()
    kp0, vp0 = bits(kp), bits(vp)
    ctx_t = torch.from_numpy(ctx).cuda()
    alen = torch.empty(B, dtype=torch.int32, device="cuda")
    em = torch.empty((B, R), dtype=torch.int32, device="cuda")
    C.accept_commit(torch.from_numpy(draft).cuda(), torch.from_numpy(am).cuda(),
                    torch.from_numpy(acc).cuda(), kb, vb, kp, vp, torch.from_numpy(table_bad).cuda(),
                    ctx_t, alen, em)
    assert C.get_device_error() == C.DEVERR_CTX | C.DEVERR_PAGE
    s, emitted = O.accept_scan(draft, am, acc)
    assert np.array_equal(alen.cpu().numpy(), s) and np.array_equal(em.cpu().numpy(), emitted)
    got_ctx = ctx_t.cpu().numpy()
    assert got_ctx[0] == ctx[0] + R and got_ctx[1] == ctx[1]
    # the oracle commit of sequence 0 alone
    only0 = np.array([R, 0, 0], dtype=np.int64)
    kp_ref, vp_ref, _ = O.commit_kv(bits(kb), bits(vb), kp0, vp0, table, ctx, only0, P)
    kp_got, vp_got = bits(kp), bits(vp)
    for b in range(B):                                     # sequence 2 wrote nothing either
        pages = table[b]
        assert np.array_equal(kp_got[:, pages], kp_ref[:, pages])
        assert np.array_equal(vp_got[:, pages], vp_ref[:, pages])


@pytest.mark.parametrize("mode", ["greedy", "sampled", "logits"])
@pytest.mark.parametrize("M,V", [(3, 300), (40, 257), (300, 1000)])
def test_lmhead_infinite_and_nan_rows(mode, M, V):
    """Rows whose logits are all -inf, or all NaN, still name an id of the vocabulary; one infinite
    logit takes all the weight; the other rows are as without them."""
    rng = np.random.default_rng(M + V)
    d = 64
    hidden = bf16(rng.standard_normal((M, d)))
    w = bf16(rng.random((V, d)) + 0.5)
    bad = hidden.clone()
    w[17, 9] = -1.0
    bad[0, 5], bad[M - 1, 7] = -math.inf, math.nan
    bad[M // 2, 9] = -math.inf           # id 17: +inf, all others -inf

    def run(h):
        ids = torch.empty(M, dtype=torch.int32, device="cuda")
        st = torch.empty((M, 5), dtype=torch.float32, device="cuda")
        dfr, ws = torch.full((M,), -1, dtype=torch.int32, device="cuda"), C.new_lmhead_workspace(M, d, V)
        if mode == "greedy":
            C.lmhead_argmax_features(h, w, dfr, ids, st, ws)
        elif mode == "sampled":
            C.lmhead_sample_features(h, w, dfr, 1.0, torch.tensor([5], device="cuda"), ids, st, ws)
        else:
            C.lmhead_logits_features(h, w, dfr, 1.0, ids, st, torch.empty((M, V), device="cuda"), ws)
        return ids.cpu().numpy(), st[:, :4].cpu().numpy()

    ids, st = run(bad)
    ref_ids, ref_st = run(hidden)
    rows = [0, M // 2, M - 1]
    assert ids[rows].tolist() == [0, 17, 0] and st[0, 0] == -math.inf and math.isnan(st[M - 1, 2])
    assert st[M // 2].tolist() == [math.inf, -math.inf, math.inf, 0.0]
    keep = np.setdiff1d(np.arange(M), rows)
    assert np.array_equal(ids[keep], ref_ids[keep]) and np.array_equal(st[keep], ref_st[keep])
    assert C.get_device_error() == 0



# ---------------------------------------------------------------------------
# Stochastic decoding: temperature sampling in the LM-head epilogue (Sec. 3.1)
# ---------------------------------------------------------------------------

def _key_margin(keys: np.ndarray) -> np.ndarray:
    top2 = np.sort(keys, axis=1)[:, -2:]
    return top2[:, 1] - top2[:, 0]


SAMPLE_CASES = [
    # M, d, V, weight std, temperature, seed
    (1, 64, 128, 0.1, 1.0, 0),
    (6, 4096, 151936, 0.02, 1.0, 0x0123456789ABCDEF),   # Qwen3-8B LM head, batch 1, K = 5
    (17, 256, 1000, 0.1, 0.5, 7),                      # ragged vocabulary tile, rows not 4-aligned
    (300, 128, 2048, 0.1, 1.0, 2 ** 40 + 3),           # two passes (160 + 140 rows)
    (64, 512, 4096, 0.3, 2.0, 99),
]


@pytest.mark.parametrize("case", SAMPLE_CASES, ids=lambda c: f"M{c[0]}V{c[2]}T{c[4]}")
def test_lmhead_sampling_matches_oracle(case):
    M, d, V, wstd, T, seed = case
    rng = np.random.default_rng(M * 13 + V)
    hidden = bf16(rng.standard_normal((M, d)))
    w = bf16(rng.standard_normal((V, d)) * wstd)
    dfr = rng.integers(-1, V, M).astype(np.int32)
    smp = torch.empty(M, dtype=torch.int32, device="cuda")
    st = torch.empty((M, 5), dtype=torch.float32, device="cuda")
    seed_t = torch.tensor([seed], dtype=torch.int64, device="cuda")
    C.lmhead_sample_features(hidden, w, torch.from_numpy(dfr).cuda(), T, seed_t, smp, st,
                             C.new_lmhead_workspace(M, d, V))
    x = O.lmhead_logits(host(hidden), host(w))
    ref_s, ref_st = O.row_stats_sampled(x, dfr, seed, T)
    assert_close(st.cpu().numpy(), ref_st, "sampled lm-head stats")
    clear = _key_margin(O.gumbel_keys(x, seed, T)) >= 1e-3
    got = smp.cpu().numpy()
    assert np.array_equal(got[clear], ref_s[clear])
    assert np.all((got >= 0) & (got < V))
    # with this much noise the sample is often not the argmax
    if M >= 17:
        assert np.mean(got != np.argmax(x, axis=1)) > 0.2
    print(f"sampled lm-head {case}: tie rows {(~clear).sum()}")


def test_lmhead_sampling_reads_the_seed_when_the_graph_runs():
    M, d, V = 12, 256, 3000
    rng = np.random.default_rng(5)
    hidden = bf16(rng.standard_normal((M, d)))
    w = bf16(rng.standard_normal((V, d)) * 0.05)
    dfr = torch.full((M,), -1, dtype=torch.int32, device="cuda")
    smp = torch.empty(M, dtype=torch.int32, device="cuda")
    st = torch.empty((M, 5), dtype=torch.float32, device="cuda")
    seed_t = torch.tensor([1], dtype=torch.int64, device="cuda")
    ws = C.new_lmhead_workspace(M, d, V)
    s = torch.cuda.Stream()
    with torch.cuda.stream(s):
        C.lmhead_sample_features(hidden, w, dfr, 1.0, seed_t, smp, st, ws)
    torch.cuda.synchronize()
    g = torch.cuda.CUDAGraph()
    with torch.cuda.graph(g):
        C.lmhead_sample_features(hidden, w, dfr, 1.0, seed_t, smp, st, ws)
    x = O.lmhead_logits(host(hidden), host(w))
    seen = []
    for seed in (3, 2 ** 33 + 5, 12345):
        seed_t.fill_(seed)
        g.replay()
        torch.cuda.synchronize()
        got = smp.cpu().numpy()
        ref, _ = O.row_stats_sampled(x, np.full(M, -1), seed, 1.0)
        clear = _key_margin(O.gumbel_keys(x, seed, 1.0)) >= 1e-3
        assert np.array_equal(got[clear], ref[clear])
        seen.append(got)
    assert not np.array_equal(seen[0], seen[1]) and not np.array_equal(seen[1], seen[2])


def test_lmhead_sampling_at_tiny_temperature_is_the_argmax():
    M, d, V = 40, 512, 5000
    rng = np.random.default_rng(8)
    hidden = bf16(rng.standard_normal((M, d)))
    w = bf16(rng.standard_normal((V, d)) * 0.05)
    dfr = torch.full((M,), -1, dtype=torch.int32, device="cuda")
    ws = C.new_lmhead_workspace(M, d, V)
    am = torch.empty(M, dtype=torch.int32, device="cuda")
    smp = torch.empty(M, dtype=torch.int32, device="cuda")
    st0 = torch.empty((M, 5), dtype=torch.float32, device="cuda")
    st1 = torch.empty((M, 5), dtype=torch.float32, device="cuda")
    C.lmhead_argmax_features(hidden, w, dfr, am, st0, ws)
    C.lmhead_sample_features(hidden, w, dfr, 1e-5, torch.tensor([77], dtype=torch.int64,
                             device="cuda"), smp, st1, ws)
    x = O.lmhead_logits(host(hidden), host(w))
    top2 = np.sort(x, axis=1)[:, -2:]
    clear = (top2[:, 1] - top2[:, 0]) >= 1e-3
    assert np.array_equal(smp.cpu().numpy()[clear], am.cpu().numpy()[clear])
    # the statistics do not depend on the sampling (up to the summation order on exact ties)
    torch.testing.assert_close(st0, st1, rtol=1e-6, atol=1e-6, equal_nan=True)


@pytest.mark.parametrize("T", [1.0, 0.6])
def test_tiny_sampled_round_matches_oracle(T):
    cfg = W.CONFIGS["tiny"].replace(batch=3, k=6, mismatch_rate=0.5, ctx_lo=30, ctx_hi=200,
                                    shuffled_pages=True)
    inp = W.make_round_inputs(cfg, device="cuda")
    hostd = {kk: (v.cpu() if torch.is_tensor(v) else v) for kk, v in inp.items()}
    x = O.lmhead_logits(hostd["hidden"], hostd["w"])
    ranked = O.topk_ids(x, 8).reshape(cfg.batch, cfg.rows, 8)
    draft = W.synth_drafts(cfg, ranked)
    seed = W.sample_seed(cfg, 0)
    rnd = VerifyRound(inp, draft, cfg.lam, C.POLICY_MLP, temperature=T, seed=seed)
    rnd.run()
    torch.cuda.synchronize()
    ref = O.cospec_round(hostd, draft, cfg.lam, with_attention=False, with_commit=False,
                         sample_seed=seed, temperature=T)
    s_gpu = rnd.accept_len.cpu().numpy()
    ties = tie_positions(ref["stats"], draft, ref["argmax"], ref["p"], ref["s"], s_gpu, cfg.lam,
                         margin=ref["key_margin"])
    report_ties("sampled round parity", f"{cfg.name} T={T}", ties)
    tie = ties > 0
    ok = ~tie
    assert np.array_equal(s_gpu[ok], ref["s"][ok])
    assert np.array_equal(rnd.emitted.cpu().numpy().reshape(cfg.batch, -1)[ok], ref["emitted"][ok])
    clear = ref["key_margin"] >= 1e-3
    assert np.array_equal(rnd.argmax.cpu().numpy().reshape(cfg.batch, -1)[clear],
                          ref["argmax"][clear])
    print(f"sampled round T={T}: s {s_gpu.tolist()} ties {int(tie.sum())}")


def test_lmhead_sampling_noise_only_at_huge_temperature():
    """At T = 1e6 the keys are the Gumbel noise alone (|x / T| < 1e-5), so each
    row's sample is the position of the largest of V noise values: the
    generator, the counter layout and the upper tail of g are checked against
    the oracle's float64 noise directly."""
    M, d, V, T, seed = 64, 256, 20000, 1e6, 0xDEADBEEF12345
    rng = np.random.default_rng(21)
    hidden = bf16(rng.standard_normal((M, d)))
    w = bf16(rng.standard_normal((V, d)) * 0.01)
    smp = torch.empty(M, dtype=torch.int32, device="cuda")
    st = torch.empty((M, 5), dtype=torch.float32, device="cuda")
    C.lmhead_sample_features(hidden, w, torch.full((M,), -1, dtype=torch.int32, device="cuda"), T,
                             torch.tensor([seed], dtype=torch.int64, device="cuda"), smp, st,
                             C.new_lmhead_workspace(M, d, V))
    x = O.lmhead_logits(host(hidden), host(w))
    keys = O.gumbel_keys(x, seed, T)
    clear = _key_margin(keys) >= 1e-3
    assert clear.sum() >= M - 2
    assert np.array_equal(smp.cpu().numpy()[clear], np.argmax(keys, axis=1)[clear])


@pytest.mark.parametrize("R,Hkv,G", [(40, 2, 1), (48, 1, 1), (20, 2, 4), (53, 1, 4)])
@pytest.mark.parametrize("ctx2", [0, 100, 300])
def test_verify_attn_stable_cache_waits_for_the_block(R, Hkv, G, ctx2):
    """With the stable-cache promise the block's own K/V may still come from the
    launch before: a long attention whose output is the short one's block keys
    and values, back to back, gives what it gives with a synchronisation between."""
    import torch
    D, P = 128, 16
    g = torch.Generator(device="cuda")
    g.manual_seed(R * 1000 + ctx2)
    rnd = lambda *sh: torch.randn(*sh, generator=g, device="cuda").to(torch.bfloat16)
    ctx1 = 16384
    pages = ctx1 // P
    kp, vp = rnd(pages, Hkv, P, D), rnd(pages, Hkv, P, D)
    table = torch.arange(pages, dtype=torch.int32, device="cuda").view(1, pages)
    c1 = torch.tensor([ctx1], dtype=torch.int32, device="cuda")
    c2 = torch.tensor([ctx2], dtype=torch.int32, device="cuda")
    q1, k1, v1 = rnd(1, R, Hkv, D), rnd(1, R, Hkv, D), rnd(1, R, Hkv, D)
    q2 = rnd(1, R, Hkv * G, D)

    def both(sync):
        blk = torch.full((1, R, Hkv, D), 3.0, dtype=torch.bfloat16, device="cuda")
        out = torch.empty_like(q2)
        torch.cuda.synchronize()
        C.verify_attn(q1, k1, v1, kp, vp, table, c1, blk, ctx1)
        if sync:
            torch.cuda.synchronize()
        C.verify_attn(q2, blk, blk, kp, vp, table, c2, out, ctx1, kv_stable=True)
        torch.cuda.synchronize()
        assert C.get_device_error() == 0
        return out

    ref = both(True)
    for _ in range(5):
        assert torch.equal(both(False), ref)


# 200 units of 640 keys and more go to the CTA pairs: row groups whose second CTA has 4, 84 or
# 128 rows, two row groups, block keys padded to 32 and 64, contexts at every tile edge, more
# units per cluster than two, a batch above the ranked ones and one of more clusters than fit.
PAIR_CTX = [0, 1, 15, 16, 17, 63, 64, 65, 127, 128, 129, 191, 192, 255, 256, 257, 383, 384, 511, 512, 513, 639, 640]


@pytest.mark.parametrize("full", [False, True], ids=["causal", "full"])
@pytest.mark.parametrize("B,R,Hq,Hkv", [
    (100, 33, 8, 2), (100, 53, 8, 2), (100, 64, 8, 2), (100, 17, 16, 2), (120, 64, 16, 2), (420, 33, 8, 2),
    (420, 33, 32, 8),
])
def test_verify_attention_pair_edges(B, R, Hq, Hkv, full):
    D = 128
    rng = np.random.default_rng(B + R * 100 + Hq)
    ctx = [PAIR_CTX[(i * 7) % len(PAIR_CTX)] for i in range(B)]
    t = _paged_case(rng, B, R, Hq, Hkv, D, ctx, True)
    assert C.verify_attn_plan(t["q"], t["k_pages"], t["page_table"], max(ctx)) == (C.ATTN_TCGEN05, 1)
    assert C.verify_attn_variant(t["q"], t["k_pages"], t["page_table"], max(ctx)) == C.ATTN_CTA_PAIR
    out = torch.empty_like(t["q"])
    for b in range(B):                   # the rest of each last page is NaN
        if ctx[b] % 16:
            page = int(t["table_np"][b, ctx[b] // 16])
            t["k_pages"][page, :, ctx[b] % 16:] = float("nan")
            t["v_pages"][page, :, ctx[b] % 16:] = float("nan")
    C.verify_attn(t["q"], t["k_blk"], t["v_blk"], t["k_pages"], t["v_pages"], t["page_table"],
                  t["ctx_len"], out, max(ctx), block_full=full)
    sub = np.arange(B) if B * Hq <= 1600 else np.sort(rng.permutation(B)[:40])
    pick = lambda x: host(x[torch.from_numpy(sub).cuda()])
    ref = O.verify_attention(pick(t["q"]), pick(t["k_blk"]), pick(t["v_blk"]),
                             np.nan_to_num(host(t["k_pages"])), np.nan_to_num(host(t["v_pages"])),
                             t["table_np"][sub], t["ctx_np"][sub], 16, **({"block_mask": "full"} if full else {}))
    assert_close(pick(out), ref, "attention (CTA pairs)")
    # a second call on other contexts gives the same where the context is the same
    ctx2 = t["ctx_len"].clone()
    ctx2[::3] = 0
    out2 = torch.full_like(out, float("nan"))
    C.verify_attn(t["q"], t["k_blk"], t["v_blk"], t["k_pages"], t["v_pages"], t["page_table"],
                  ctx2, out2, max(ctx), block_full=full)
    keep = torch.arange(B, device="cuda") % 3 != 0
    assert torch.equal(out2[keep], out[keep])
    assert not torch.isnan(out2).any()
    assert C.get_device_error() == 0


def test_verify_attention_pair_skips_only_the_bad_sequence():
    B, R, Hq, Hkv, D = 100, 53, 8, 2, 128
    rng = np.random.default_rng(53)
    ctx = [640 - 3 * i for i in range(B)]
    t = _paged_case(rng, B, R, Hq, Hkv, D, ctx, True)
    assert C.verify_attn_variant(t["q"], t["k_pages"], t["page_table"], 640) == C.ATTN_CTA_PAIR
    call = lambda c, o: C.verify_attn(t["q"], t["k_blk"], t["v_blk"], t["k_pages"], t["v_pages"],
                                      t["page_table"], c, o, 640)
    good, out = torch.empty_like(t["q"]), torch.full_like(t["q"], float("nan"))
    call(t["ctx_len"], good)
    assert C.get_device_error() == 0
    bad = t["ctx_len"].clone()
    bad[5], bad[70] = -1, t["page_table"].shape[1] * 16 + 1
    call(bad, out)
    torch.cuda.synchronize()
    assert C.get_device_error() == C.DEVERR_CTX
    skip = torch.zeros(B, dtype=torch.bool, device="cuda")
    skip[[5, 70]] = True
    assert torch.equal(out[~skip], good[~skip]) and (out[skip] == 0).all()


@pytest.mark.parametrize("batch,k,ctx,layers", [(1, 4, 40, 12), (2, 7, 100, 12), (3, 15, 300, 8)])
def test_rounds_queued_without_a_restore_read_the_round_before(monkeypatch, batch, k, ctx, layers):
    """Three rounds on a growing context, captured back to back and replayed, give what the
    same launches give with a synchronisation after each, bit for bit: the second layer of a round
    starts early, but not before the commit of the round before is done."""
    cfg = W.CONFIGS["tiny"].replace(batch=batch, k=k, ctx_lo=ctx, ctx_hi=ctx, layers=layers, mismatch_rate=0.3)

    def new_round():
        inp = W.make_round_inputs(cfg, device="cuda", extra_tokens=3 * (k + 1))
        draft = W.synth_drafts(cfg, O.topk_ids(O.lmhead_logits(inp["hidden"].cpu(), inp["w"].cpu()), 8)
                               .reshape(cfg.batch, cfg.rows, 8))
        return VerifyRound(inp, draft, max_ctx=ctx + 3 * (k + 1), keep_attn=True)

    def restart(rnd, seed):
        g = torch.Generator(device="cuda")
        g.manual_seed(seed)
        for t in (rnd.k_blk, rnd.v_blk, rnd.q):
            t.normal_(generator=g)
        rnd.restore_context()

    def state(rnd):
        return [t.clone() for t in (rnd.attn_out, rnd.k_pages, rnd.v_pages, rnd.ctx_len, rnd.emitted)]

    rnd, ref = new_round(), new_round()
    restart(rnd, 0)
    rnd.run(restore=False)
    torch.cuda.synchronize()
    graph = torch.cuda.CUDAGraph()
    with torch.cuda.graph(graph):
        for _ in range(3):
            rnd.run(restore=False)
    got = []
    for seed in (1, 2, 3):
        restart(rnd, seed)
        graph.replay()
        got.append(state(rnd))
    torch.cuda.synchronize()
    for name in ("verify_attn", "accept_commit"):
        call = getattr(C, name)
        monkeypatch.setattr(C, name, lambda *a, _call=call, **kw: (_call(*a, **kw), torch.cuda.synchronize())[0])
    restart(ref, 0)
    ref.run(restore=False)
    for seed, have in zip((1, 2, 3), got):
        restart(ref, seed)
        for _ in range(3):
            ref.run(restore=False)
        for a, b in zip(have, state(ref)):
            assert torch.equal(a, b)
    assert C.get_device_error() == 0
