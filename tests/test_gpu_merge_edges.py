"""The persistent kernel's merge of chunk partials at the edges of what its threads take at a time, against the CPU oracle."""
import pytest

from paper_2509_18362_b200 import inputs as I
from tests.test_gpu_draft import check_draft, run_draft_case

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("dh,L", [
    # chunks of 64 positions dealt over 8 (head dimension 128) or 16 groups of threads, which take five rounds at a time; a new turn
    # of weights after 32 or 16 rounds: 256 chunks at either head dimension
    (128, [64 * 40 - 2, 64 * 40, 64 * 41, 64 * 79, 64 * 80, 64 * 81]),
    (64, [64 * 80 - 2, 64 * 80, 64 * 81, 64 * 159, 64 * 160, 64 * 161]),
    (128, [64 * 256 - 2, 64 * 256, 64 * 257, 64 * 296 + 5]),
    (64, [64 * 256 - 2, 64 * 256, 64 * 257, 64 * 336 + 5]),
    (128, [64 * 520 + 1]),
])
def test_chunk_counts(dh, L, monkeypatch):
    monkeypatch.setenv("FMTP_BATCHED_MIN", "99")
    shape = I.Shape(d=256, n_q_heads=4, n_kv_heads=2, head_dim=dh, ffn=272, vocab=512, n_layers=1, rms_eps=1e-6,
                    rope_theta=1e4, page_size=16)
    got, ref = run_draft_case(shape, 60 + dh + len(L), len(L), L, 3, 128)
    check_draft(got, ref, f"dh={dh} L={L}")
    assert got["launches"] == 1
