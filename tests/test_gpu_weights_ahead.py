"""Gate/up weights that are asked into L2 ahead of their phase: results with requests under way, against the CPU oracle. (Which rows
are asked for is looked over in test_weights_ahead.py: a request changes no value.)"""
import pytest

from oracle import fastmtp_oracle as O
from paper_2509_18362_b200 import inputs as I
from tests import test_gpu_extend_layout as layout
from tests.gpu_util import close, copy_kv
from tests.test_gpu_draft import check_draft, run_draft_case
from tests.test_gpu_target import GpuTarget

pytestmark = pytest.mark.gpu


# Rows of 4 KB, so that the ring is full and the producers wait while the consumers attend; a CTA has two or three tiles of 16, the
# third of one row; 38 tiles of 128 and one of 16 rows, which W_o's GEMM (16 row ranges, split along K) asks for.
WIDE = I.Shape(d=2048, n_q_heads=16, n_kv_heads=2, head_dim=128, ffn=4880, vocab=1500, n_layers=1, rms_eps=1e-6,
               rope_theta=1e4, page_size=16)


@pytest.mark.parametrize("batched", [False, True])
@pytest.mark.parametrize("B", [1, 2, 6])       # six rows: the persistent kernel with two sets of accumulators
def test_draft_of_a_wide_layer(B, batched, monkeypatch):
    monkeypatch.setenv("FMTP_BATCHED_MIN", "1" if batched else "99")
    got, ref = run_draft_case(WIDE, 910 + B, B, [130 + 37 * b for b in range(B)], 3, 700)
    check_draft(got, ref, f"B={B} batched={batched}")
    assert (got["launches"] == 1) == (not batched)


@pytest.mark.parametrize("shape,L,n_ext,max_ext", [
    (WIDE, [61], [4], 4),                                                                             # two layouts of shared memory
    (I.Shape(d=3072, n_q_heads=6, n_kv_heads=2, head_dim=64, ffn=4880, vocab=1500, n_layers=1), [63], [4], 4),      # the projection restages
])
def test_extend_rows_of_a_wide_layer(shape, L, n_ext, max_ext):
    layout.test_later_steps_run_in_their_own_layout(shape, L, n_ext, max_ext, 3, 700)


@pytest.mark.parametrize("batched", [False, True])
@pytest.mark.parametrize("M", [1, 4])
def test_target_of_several_wide_layers(M, batched, monkeypatch):
    """Every layer has its own gate/up matrices."""
    monkeypatch.setenv("FMTP_BATCHED_MIN", "1" if batched else "99")
    s = WIDE.with_layers(3)
    kvs = [I.paged_kv(s, [200], M, 921 + l) for l in range(3)]
    Wt = I.target_weights(s, 920)
    gpu = GpuTarget(s, Wt, kvs, 256)
    t = I.token_ids(925, (1, M), s.vocab)
    h, l, _ = gpu.step(t)
    assert (gpu.ctx.launch_count == 1) == (not batched)
    rh, rl = O.target_forward(s, Wt, t, [copy_kv(kv) for kv in kvs])
    close(h.float().cpu().numpy(), rh, "hidden states")
    close(l.float().cpu().numpy(), rl, "logits")
    gpu.close()


@pytest.mark.parametrize("batched", [False, True])
@pytest.mark.parametrize("ffn", [
    2352,      # persistent kernel: at most 16 rows per CTA, one tile
    2384,      # a few CTAs have a second tile of one row
    7168,      # four tiles, the last one of a few rows; batched: 56 tiles of 128, W_o's GEMM has two CTAs and ends before most are asked for
    9520,      # five tiles; batched: the last tile has 48 rows
    19040,     # batched: more tiles of 128 than SMs
])
def test_parity_at_the_edges_of_the_share(ffn, batched, monkeypatch):
    shape = I.Shape(d=256, n_q_heads=4, n_kv_heads=2, head_dim=64, ffn=ffn, vocab=2048, n_layers=1, rms_eps=1e-6,
                    rope_theta=1e4, page_size=16)
    monkeypatch.setenv("FMTP_BATCHED_MIN", "1" if batched else "99")
    got, ref = run_draft_case(shape, 900 + ffn % 97, 2, [5, 130], 2, 512)
    check_draft(got, ref, f"ffn={ffn} batched={batched}")
    assert (got["launches"] == 1) == (not batched)
