"""Gate/up weights that are asked into L2 ahead of their phase: widths at which a CTA's share ends inside a tile, is one
row past a tile, or is a single tile (nothing is asked for), on both kernel paths, against the CPU oracle."""
import pytest

from paper_2509_18362_b200 import inputs as I
from tests.test_gpu_draft import check_draft, run_draft_case

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("batched", [False, True])
@pytest.mark.parametrize("ffn", [
    2352,      # persistent kernel: at most 16 rows per CTA, one tile
    2384,      # a few CTAs have a second tile of one row
    7168,      # four tiles, the last one of a few rows; batched: 56 tiles of 128
    9520,      # five tiles; batched: the last tile has 48 rows
    19040,     # more tiles of 128 than CTAs: some have two
])
def test_parity_at_the_edges_of_the_share(ffn, batched, monkeypatch):
    shape = I.Shape(d=256, n_q_heads=4, n_kv_heads=2, head_dim=64, ffn=ffn, vocab=2048, n_layers=1, rms_eps=1e-6,
                    rope_theta=1e4, page_size=16)
    monkeypatch.setenv("FMTP_BATCHED_MIN", "1" if batched else "99")
    got, ref = run_draft_case(shape, 900 + ffn % 97, 2, [5, 130], 2, 512)
    check_draft(got, ref, f"ffn={ffn} batched={batched}")
    assert (got["launches"] == 1) == (not batched)
