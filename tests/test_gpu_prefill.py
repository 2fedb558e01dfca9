"""The arbitrator's attention for one request on the device: its context
prefilled causally in chunks (verify attention + commit), then its
draft/target region attended with the full block mask, against the oracle's
dense attention under the paper's hybrid mask (Sec. 3.3)."""
import numpy as np
import pytest
import torch

from oracle import cospec_oracle as O
from paper_2605_24793_gb300 import build as BLD
from paper_2605_24793_gb300 import cospec as C
from paper_2605_24793_gb300.prefill import BlockPrefill, ChunkedPrefill

from .parity_util import assert_close

pytestmark = pytest.mark.gpu


@pytest.fixture(scope="module", autouse=True)
def lib():
    C.load_library(BLD.build())
    torch.cuda.set_device(0)


def _bf16(rng, shape):
    return torch.from_numpy(rng.standard_normal(shape, dtype=np.float32)).to(torch.bfloat16).cuda()


@pytest.mark.parametrize("method", [BlockPrefill, ChunkedPrefill], ids=["block", "chunked"])
@pytest.mark.parametrize("L,B,T,Hq,Hkv,D,region", [
    (2, 2, 200, 8, 2, 64, 9),        # ragged last chunk (200 = 6 x 32 + 8), K = 3 region
    (1, 1, 33, 32, 8, 128, 17),      # one full chunk and one row, K = 7 region
    (1, 3, 96, 16, 8, 128, 53),      # three full chunks, K = 25 region (53 rows)
    (1, 1, 1000, 8, 2, 128, 17),     # 32 chunks, the last of 8 rows
    (2, 3, 704, 4, 2, 64, 9),        # whole chunks, read where they lie: 66 chunk sequences, two layers
    (1, 2, 256, 2, 2, 64, 9),        # one query head per KV head, whole blocks of 64
    (1, 2, 200, 2, 2, 64, 9),        # the same, ragged and an odd number of chunks
])
def test_prefill_then_region_matches_dense_hybrid_attention(method, L, B, T, Hq, Hkv, D, region):
    rng = np.random.default_rng(T * 7 + region)
    G = Hq // Hkv
    q = _bf16(rng, (L, B, T, Hq, D))
    k = _bf16(rng, (L, B, T, Hkv, D))
    v = _bf16(rng, (L, B, T, Hkv, D))
    pf = method(L, B, T, Hq, Hkv, D, extra_tokens=region)
    out = pf.run(q, k, v)
    torch.cuda.synchronize()
    assert C.get_device_error() == 0
    assert np.array_equal(pf.ctx_len.cpu().numpy(), np.full(B, T))
    # the region: 2K+3 rows over the prefilled context, bidirectional among themselves
    qr = _bf16(rng, (L, B, region, Hq, D))
    kr = _bf16(rng, (L, B, region, Hkv, D))
    vr = _bf16(rng, (L, B, region, Hkv, D))
    outr = torch.empty((L, B, region, Hq, D), dtype=torch.bfloat16, device="cuda")
    for l in range(L):
        C.verify_attn(qr[l], kr[l], vr[l], pf.k_pages[l], pf.v_pages[l], pf.page_table, pf.ctx_len,
                      outr[l], T, block_full=True)
    torch.cuda.synchronize()
    assert C.get_device_error() == 0
    vis = O.hybrid_mask(T, region)
    f = lambda t: t.float().cpu().numpy()
    for l in range(L):
        for b in range(B):
            for h in range(Hq):
                kv = h // G
                qq = np.concatenate([f(q[l, b, :, h]), f(qr[l, b, :, h])])
                kk = np.concatenate([f(k[l, b, :, kv]), f(kr[l, b, :, kv])])
                vv = np.concatenate([f(v[l, b, :, kv]), f(vr[l, b, :, kv])])
                ref = O.dense_masked_attention(qq, kk, vv, vis)
                assert_close(f(out[l, b, :, h]), ref[:T], f"context rows l={l} b={b} h={h}")
                assert_close(f(outr[l, b, :, h]), ref[T:], f"region rows l={l} b={b} h={h}")
    # the cache holds the context's keys and values, position by position
    kp = pf.k_pages.cpu().view(torch.int16).numpy()
    table = pf.page_table.cpu().numpy()
    kb = k.cpu().view(torch.int16).numpy()
    for b in range(B):
        t = np.arange(T)
        np.testing.assert_array_equal(kp[:, table[b, t // 16], :, t % 16].transpose(1, 0, 2, 3), kb[:, b])


@pytest.mark.parametrize("form", ["host", "float32", "strided", "long_v", "shared_v"])
def test_block_prefill_takes_every_form_of_the_projections(form):
    """Whole-chunk contexts whose projections cannot be read where they lie give
    what the in-place path gives for the same values, bit for bit."""
    L, B, T, Hq, Hkv, D = 2, 2, 96, 4, 2, 64
    rng = np.random.default_rng(96)
    q, k, v = _bf16(rng, (L, B, T, Hq, D)), _bf16(rng, (L, B, T, Hkv, D)), _bf16(rng, (L, B, T, Hkv, D))
    if form == "shared_v":
        v = v[:1].expand(L, B, T, Hkv, D).contiguous()
    plain = BlockPrefill(L, B, T, Hq, Hkv, D)
    ref = plain.run(q, k, v)
    if form == "host":
        q2, k2, v2 = q.cpu(), k.cpu(), v.cpu()
    elif form == "float32":
        q2, k2, v2 = q.float(), k.float(), v.float()
    elif form == "strided":
        q2, k2, v2 = (t.transpose(1, 2).contiguous().transpose(1, 2) for t in (q, k, v))
    elif form == "long_v":
        q2, k2, v2 = q, k, torch.cat([v, v[:, :, :5]], dim=2)
    else:
        q2, k2, v2 = q, k, v[:1]
    other = BlockPrefill(L, B, T, Hq, Hkv, D)
    other.step()                         # without a load: zero projections
    out = other.run(q2, k2, v2)
    torch.cuda.synchronize()
    assert C.get_device_error() == 0
    assert out.device == q2.device and out.dtype == q2.dtype and out.stride() == torch.empty_like(q2).stride()
    assert torch.equal(out.to("cuda", torch.bfloat16), ref)
    assert torch.equal(other.k_pages, plain.k_pages) and torch.equal(other.v_pages, plain.v_pages)


def _synchronised(monkeypatch, name):
    """The binding's call `name`, waited for before it returns."""
    call = getattr(C, name)

    def synced(*args, **kw):
        out = call(*args, **kw)
        torch.cuda.synchronize()
        return out

    monkeypatch.setattr(C, name, synced)


@pytest.mark.parametrize("L,T,Hq,Hkv,D", [(12, 64, 8, 2, 128), (12, 128, 32, 8, 128), (6, 256, 8, 2, 64), (12, 40, 4, 2, 128)])
def test_block_prefill_layers_read_what_the_commit_wrote(monkeypatch, L, T, Hq, Hkv, D):
    """Replays on changing projections (so that a stale cache would show) give what the same
    launches give with a synchronisation after each, bit for bit: layers after the first start
    early, but not before the commit two launches back is done."""
    rng = np.random.default_rng(L * 1000 + T)
    inputs = [[_bf16(rng, (L, 1, T, h, D)) for h in (Hq, Hkv, Hkv)] for _ in range(3)]
    pf = BlockPrefill(L, 1, T, Hq, Hkv, D)
    pf.load(*inputs[-1])
    pf.step()
    torch.cuda.synchronize()
    graph = torch.cuda.CUDAGraph()
    with torch.cuda.graph(graph):
        pf.step()
    got = []
    for x in inputs:
        pf.load(*x)
        graph.replay()
        got.append([t.clone() for t in (pf.outp, pf.k_pages, pf.v_pages)])
    torch.cuda.synchronize()
    _synchronised(monkeypatch, "accept_commit")
    _synchronised(monkeypatch, "verify_attn")
    ref = BlockPrefill(L, 1, T, Hq, Hkv, D)
    for x, have in zip(inputs, got):
        ref.load(*x)
        ref.step()
        for a, b in zip(have, (ref.outp, ref.k_pages, ref.v_pages)):
            assert torch.equal(a, b)
    assert C.get_device_error() == 0


@pytest.mark.parametrize("T", [64, 72])
def test_block_prefill_step_captured_before_any_load(T):
    """A step captured first, projections loaded afterwards: each replay takes those."""
    L, Hq, Hkv, D = 2, 4, 2, 64
    rng = np.random.default_rng(T)
    pf, ref = BlockPrefill(L, 1, T, Hq, Hkv, D), BlockPrefill(L, 1, T, Hq, Hkv, D)
    graph = torch.cuda.CUDAGraph()
    with torch.cuda.graph(graph):
        pf.step()
    for _ in range(2):
        x = [_bf16(rng, (L, 1, T, h, D)) for h in (Hq, Hkv, Hkv)]
        pf.load(*x)
        graph.replay()
        out = ref.run(*x)
        torch.cuda.synchronize()
        assert torch.equal(pf.outp[:, :, :T], out)
        assert torch.equal(pf.k_pages, ref.k_pages) and torch.equal(pf.v_pages, ref.v_pages)
    assert C.get_device_error() == 0


@pytest.mark.parametrize("T", [64, 72])
def test_block_prefill_run_leaves_its_projections_loaded(T):
    """A step() after run() is the same prefill again, whatever became of the inputs."""
    L, Hq, Hkv, D = 2, 4, 2, 64
    rng = np.random.default_rng(T + 1)
    pf = BlockPrefill(L, 1, T, Hq, Hkv, D)
    x = [_bf16(rng, (L, 1, T, h, D)) for h in (Hq, Hkv, Hkv)]
    out = pf.run(*x)
    kp, vp = pf.k_pages.clone(), pf.v_pages.clone()
    for t in x:
        t.zero_()
    pf.step()
    torch.cuda.synchronize()
    assert torch.equal(pf.outp[:, :, :T], out)
    assert torch.equal(pf.k_pages, kp) and torch.equal(pf.v_pages, vp)
    assert C.get_device_error() == 0
