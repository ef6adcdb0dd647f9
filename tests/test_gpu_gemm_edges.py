"""Batched draft calls at the edges of the GEMM's tiles, items and operand widths, against the oracle."""
import pytest

from paper_2509_18362_b200 import inputs as I
from tests.test_gpu_draft import check_draft, run_draft_case

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
