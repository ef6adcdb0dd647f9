"""Persistent kernel: extend rows whose step 0 leaves few ring stages. The projection's two input vectors then share one place,
and shared memory is laid out anew for the later steps."""
import numpy as np
import pytest

from oracle import fastmtp_oracle as O
from paper_2509_18362_b200 import binding as Bd
from paper_2509_18362_b200 import inputs as I
from tests.gpu_util import close, copy_kv, ids_match
from tests.test_gpu_draft import _extend_case, _run_extend

pytestmark = pytest.mark.gpu

WIDE = I.Shape(d=2048, n_q_heads=6, n_kv_heads=2, head_dim=128, ffn=640, vocab=1500, n_layers=1)
WIDER = I.Shape(d=3072, n_q_heads=6, n_kv_heads=2, head_dim=64, ffn=640, vocab=1500, n_layers=1)


@pytest.mark.parametrize("shape,L,n_ext,max_ext,K,N", [
    (WIDE, [61], [4], 4, 3, 700), (WIDE, [130], [2], 4, 5, None), (WIDE, [0, 64], [2, 1], 2, 3, 700),
    (WIDE, [20], [3], 4, 1, 700),                  # a single step: nothing to switch to
    (WIDER, [63], [4], 4, 3, 700), (WIDER, [9], [2], 3, 2, 700),                    # the projection restages
    (WIDE, [9], [5], 5, 2, 700), (WIDER, [60], [6], 6, 3, 700), (WIDE, [5, 70], [3, 2], 3, 2, None),    # more than four rows: both vectors at once
])
def test_later_steps_run_in_their_own_layout(shape, L, n_ext, max_ext, K, N):
    W, kv, h, tok, ids = _extend_case(shape, 77 + len(L), L, n_ext, max_ext, K, N)
    got = _run_extend(Bd, shape, W, kv, h, tok, ids, n_ext, max_ext, K, max(L) + max_ext + K + 1)
    again = _run_extend(Bd, shape, W, kv, h, tok, ids, n_ext, max_ext, K, max(L) + max_ext + K + 1)
    assert got["status"] == 0 and got["launches"] == 1
    assert np.array_equal(got["h_bits"], again["h_bits"]) and np.array_equal(got["drafts"], again["drafts"])
    okv = copy_kv(kv)
    for b in range(len(L)):
        one = dict(okv)
        one["block_table"], one["seq_lens"] = okv["block_table"][b:b + 1], okv["seq_lens"][b:b + 1]
        ref = O.draft(shape, W, h[b:b + 1, :n_ext[b]], tok[b:b + 1, :n_ext[b]], one, K, ids, forced=got["drafts"][b:b + 1])
        ids_match(got["drafts"][b], ref["drafts"], ref["gap"], f"drafts b={b}")
        close(got["h_out"][b:b + 1], ref["h_out"], f"h_out b={b}")
    close(O.bf16_to_f64(got["k_pages"]), O.bf16_to_f64(okv["k_pages"]), "K cache")
    close(O.bf16_to_f64(got["v_pages"]), O.bf16_to_f64(okv["v_pages"]), "V cache")
