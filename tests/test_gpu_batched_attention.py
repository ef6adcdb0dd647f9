"""Batched attention at the edges of its tiles: 16-token copies, 64-token blocks, 256-token items, four rows per item."""
from dataclasses import replace

import numpy as np
import pytest
import torch

from oracle import fastmtp_oracle as O
from paper_2509_18362_b200 import binding as Bd
from paper_2509_18362_b200 import inputs as I
from tests.gpu_util import close, copy_kv
from tests.test_gpu_target import GpuTarget

pytestmark = pytest.mark.gpu

EDGES = [0, 1, 14, 15, 16, 47, 63, 64, 250, 255, 256, 257, 511, 530]


@pytest.mark.parametrize("page,dh,M", [
    (16, 64, 1), (16, 64, 4), (16, 128, 3), (48, 128, 4),      # one row; a full row set; a set with a row missing; tiles inside a page
    (64, 64, 6),                                               # two row sets per sequence
    (8, 128, 1), (5, 64, 4),                                   # pages that are not whole 16-token tiles: the 16-byte copies
])
def test_batched_attention_edges(page, dh, M, monkeypatch):
    """One layer over contexts at every tile edge. Cache slots that nothing has written hold NaN: they must not reach any
    result. Tolerances: gpu_util."""
    monkeypatch.setenv("FMTP_BATCHED_MIN", "1")
    s = replace(I.TINY, head_dim=dh, page_size=page, n_layers=1)
    L = EDGES[:64 // M]
    kv = I.paged_kv(s, L, M, 41)
    for b, n in enumerate(L):
        for i, p in enumerate(kv["block_table"][b]):
            if p >= 0 and (i + 1) * page > n:
                kv["k_pages"][p, :, max(0, n - i * page):] = 0x7FC0
                kv["v_pages"][p, :, max(0, n - i * page):] = 0x7FC0
    Wt = I.target_weights(s, 42)
    gpu = GpuTarget(s, Wt, [kv], max(L) + M)
    gpu.ctx.close()
    gpu.ctx = Bd.Context(s, max_rows=64, max_K=1, max_ctx=max(L) + M)
    t = I.token_ids(43, (len(L), M), s.vocab)
    h, l, _ = gpu.step(t)
    okv = [copy_kv(kv)]
    rh, rl = O.target_forward(s, Wt, t, okv)
    close(h.float().cpu().numpy(), rh, "hidden states")
    close(l.float().cpu().numpy(), rl, "logits")
    for k in ("k_pages", "v_pages"):                           # the appended rows, and nothing else, changed
        got, want = Bd.bf16_bits(gpu.dkvs[0][k]), kv[k].copy()
        for b, n in enumerate(L):
            for i in range(M):
                at = (kv["block_table"][b, (n + i) // page], slice(None), (n + i) % page)
                close(O.bf16_to_f64(got[at]), O.bf16_to_f64(okv[0][k][at]), k)
                want[at] = got[at]
        assert np.array_equal(got, want)
    if M > 1:                                                  # rows one by one: the same bits
        one = GpuTarget(s, Wt, [kv], max(L) + M)
        one.ctx.close()
        one.ctx = Bd.Context(s, max_rows=64, max_K=1, max_ctx=max(L) + M)
        for i in range(M):
            h1, l1, _ = one.step(np.ascontiguousarray(t[:, i:i + 1]))
            assert np.array_equal(Bd.bf16_bits(h1[:, 0]), Bd.bf16_bits(h[:, i]))
            assert np.array_equal(Bd.bf16_bits(l1[:, 0]), Bd.bf16_bits(l[:, i]))
            one.advance(1)
        one.close()
    gpu.close()


def test_merge_of_few_and_many_chunks(monkeypatch):
    """Contexts around 8 and 32 items of 256 tokens, where the chunk merge changes its group size and starts a second group."""
    s = replace(I.TINY, n_layers=1)
    L, M = [2040, 2047, 2300, 8185, 8191, 8500], 2
    kv = I.paged_kv(s, L, M, 51)
    Wt = I.target_weights(s, 52)
    gpu = GpuTarget(s, Wt, [kv], max(L) + M)
    gpu.ctx.close()
    monkeypatch.setenv("FMTP_BATCHED_MIN", "1")
    gpu.ctx = Bd.Context(s, max_rows=64, max_K=1, max_ctx=max(L) + M)
    t = I.token_ids(53, (len(L), M), s.vocab)
    h, l, _ = gpu.step(t)
    rh, rl = O.target_forward(s, Wt, t, [copy_kv(kv)])
    close(h.float().cpu().numpy(), rh, "hidden states")
    close(l.float().cpu().numpy(), rl, "logits")
    gpu.close()


@pytest.mark.parametrize("batched", [True, False])
@pytest.mark.parametrize("bits", [0x7FC0, 0x7F80])               # NaN, infinity
@pytest.mark.parametrize("dh,M", [(64, 4), (128, 3), (64, 6)])
def test_a_row_does_not_see_what_later_rows_hold(dh, M, bits, batched, monkeypatch):
    """The last row's token has an embedding that is not finite, and so are its keys and values: the rows before it, which share
    its K/V blocks, give the bits they give beside a finite one."""
    monkeypatch.setenv("FMTP_BATCHED_MIN", "1" if batched else "99")
    s = replace(I.TINY, head_dim=dh, n_layers=1)
    L = [0, 3, 14, 30, 63, 250] if batched else [14 if M < 6 else 60]
    kv = I.paged_kv(s, L, M, 61)
    Wt = I.target_weights(s, 62)
    t = I.token_ids(63, (len(L), M), s.vocab - 1)
    t_odd = t.copy()
    t_odd[:, -1] = s.vocab - 1
    Wt["embed"][s.vocab - 1] = bits
    got = []
    for tokens in (t, t_odd):
        gpu = GpuTarget(s, Wt, [kv], max(L) + M)
        gpu.ctx.close()
        gpu.ctx = Bd.Context(s, max_rows=64, max_K=1, max_ctx=max(L) + M)
        h = torch.zeros((len(L), M, s.d), dtype=torch.bfloat16, device="cuda")
        gpu.ctx.fastmtp_target_step(gpu.w, torch.from_numpy(tokens).cuda(), [Bd.kv(k) for k in gpu.dkvs], len(L), M, h)
        torch.cuda.synchronize()
        got.append(Bd.bf16_bits(h))
        gpu.close()
    assert np.isnan(O.bf16_to_f64(got[1][:, -1])).any()
    assert np.array_equal(got[0][:, :-1], got[1][:, :-1])
