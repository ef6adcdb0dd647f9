"""Batched draft calls at the edges of the GEMM's tiles, items and operand widths, against the oracle."""
import pytest
import torch

from oracle import fastmtp_oracle as O
from paper_2509_18362_b200 import inputs as I
from tests.gpu_util import close, copy_kv
from tests.test_gpu_draft import check_draft, run_draft_case
from tests.test_gpu_target import GpuTarget

pytestmark = pytest.mark.gpu

# q, k and v rows end inside a 128-row tile; d, q_dim and ffn leave a K block short of a ring stage or of 64 elements
ODD = I.Shape(d=320, n_q_heads=5, n_kv_heads=1, head_dim=64, ffn=1072, vocab=700, n_layers=1)
# enough head rows that an item has two tiles (more than 128 per SM)
WIDE = I.Shape(d=128, n_q_heads=2, n_kv_heads=1, head_dim=64, ffn=144, vocab=40000, n_layers=1)


@pytest.mark.parametrize("shape,B,N", [
    (ODD, 3, 1), (ODD, 8, 127), (ODD, 9, 129), (ODD, 16, 256), (ODD, 17, 257), (ODD, 33, 700), (ODD, 40, None), (ODD, 64, 640),
    (WIDE, 4, 18944), (WIDE, 4, 18945), (WIDE, 20, 30011), (WIDE, 64, 37889), (WIDE, 12, None),
])
def test_gemm_edges(shape, B, N, monkeypatch):
    """One to 64 activation rows (every width class of the operand), subsets around tile and item sizes."""
    monkeypatch.setenv("FMTP_BATCHED_MIN", "1")
    got, ref = run_draft_case(shape, 70 + B, B, [5 * b % 90 for b in range(B)], 2, N, want_logits=False)
    check_draft(got, ref, f"B={B} N={N}")


@pytest.mark.parametrize("d,V,B", [(64, 75900, 17), (128, 75900, 64), (64, 152064, 64), (128, 152064, 17), (64, 152064, 5)])
def test_head_of_three_and_more_items_per_cta(d, V, B, monkeypatch):
    """So few K blocks that a CTA's ring holds its last items before the first one's MMAs have begun: whoever joins for the
    last item's epilogue has to wait for that item, not for an earlier one in the same accumulator buffer."""
    monkeypatch.setenv("FMTP_BATCHED_MIN", "1")
    s = I.Shape(d=d, n_q_heads=2, n_kv_heads=1, head_dim=64, ffn=144, vocab=V, n_layers=1)
    got, ref = run_draft_case(s, 60 + B, B, [3 * b % 50 for b in range(B)], 1, None, want_logits=True)
    check_draft(got, ref, f"d={d} V={V} B={B}")
    for b in range(B):
        close(got["logits"][b, 0], O.head_logits(ref["h_out"][b, 0], ref["W"]["lm_head"]), f"logits b={b}")


@pytest.mark.parametrize("d", [64, 4096, 4160, 8192, 8256])
def test_row_kernels_by_width(d, monkeypatch):
    """Widths at which a thread of the row-wise kernels owns one, two or more groups of columns."""
    monkeypatch.setenv("FMTP_BATCHED_MIN", "1")
    s = I.Shape(d=d, n_q_heads=2, n_kv_heads=1, head_dim=64, ffn=80, vocab=300, n_layers=2)
    B, M = 3, 2
    kvs = [I.paged_kv(s, [0, 7, 20], M, 91 + l) for l in range(2)]
    Wt = I.target_weights(s, 90)
    gpu = GpuTarget(s, Wt, kvs, 32)
    t = I.token_ids(93, (B, M), s.vocab)
    h, l, _ = gpu.step(t)
    rh, rl = O.target_forward(s, Wt, t, [copy_kv(kv) for kv in kvs])
    close(h.float().cpu().numpy(), rh, "hidden states")
    close(l.float().cpu().numpy(), rl, "logits")
    gpu.close()
    if d <= 4160:                                  # the draft's first kernel too
        got, ref = run_draft_case(s, 95, 2, [3, 40], 2, 200, want_logits=False)
        check_draft(got, ref, f"d={d}")


@pytest.mark.parametrize("B", [1, 2, 3])
def test_target_path_by_sequences(B):
    """A model with more than 256 MB of weights per layer: target calls of three and more sequences take the batched path. On
    either path the bits do not depend on the rows per call."""
    s = I.Shape(d=2560, n_q_heads=2, n_kv_heads=1, head_dim=128, ffn=16384, vocab=300, n_layers=1)
    M, L = 2, [40, 0, 70][:B]
    kv = I.paged_kv(s, L, M, 94)
    Wt = I.target_weights(s, 95)
    gpu, one = GpuTarget(s, Wt, [kv], max(L) + M), GpuTarget(s, Wt, [kv], max(L) + M)
    t = I.token_ids(96, (B, M), s.vocab)
    n0 = gpu.ctx.launch_count
    h, l, _ = gpu.step(t)
    assert (gpu.ctx.launch_count - n0 == 1) == (B < 3)
    rh, rl = O.target_forward(s, Wt, t, [copy_kv(kv)])
    close(h.float().cpu().numpy(), rh, "hidden states")
    close(l.float().cpu().numpy(), rl, "logits")
    for i in range(M):
        h1, l1, _ = one.step(t[:, i:i + 1].copy())
        assert torch.equal(h1[:, 0], h[:, i]) and torch.equal(l1[:, 0], l[:, i])
        one.advance(1)
    gpu.close()
    one.close()
