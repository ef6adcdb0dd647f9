"""Persistent kernel: extend rows whose step 0 leaves fewer ring stages than the later steps, so that shared memory is laid out
anew between them."""
import numpy as np
import pytest

from oracle import fastmtp_oracle as O
from paper_2509_18362_b200 import binding as Bd
from paper_2509_18362_b200 import inputs as I
from tests.gpu_util import close, copy_kv, ids_match
from tests.test_gpu_draft import _extend_case, _run_extend

pytestmark = pytest.mark.gpu

WIDE = I.Shape(d=2048, n_q_heads=6, n_kv_heads=2, head_dim=128, ffn=640, vocab=1500, n_layers=1)


@pytest.mark.parametrize("L,n_ext,max_ext,K,N", [
    ([61], [4], 4, 3, 700), ([130], [2], 4, 5, None), ([0, 64], [2, 1], 2, 3, 700),
    ([20], [3], 4, 1, 700),                        # a single step: nothing to switch to
])
def test_later_steps_run_in_their_own_layout(L, n_ext, max_ext, K, N):
    W, kv, h, tok, ids = _extend_case(WIDE, 77 + len(L), L, n_ext, max_ext, K, N)
    got = _run_extend(Bd, WIDE, W, kv, h, tok, ids, n_ext, max_ext, K, max(L) + max_ext + K + 1)
    again = _run_extend(Bd, WIDE, W, kv, h, tok, ids, n_ext, max_ext, K, max(L) + max_ext + K + 1)
    assert got["status"] == 0 and got["launches"] == 1
    assert np.array_equal(got["h_bits"], again["h_bits"]) and np.array_equal(got["drafts"], again["drafts"])
    okv = copy_kv(kv)
    for b in range(len(L)):
        one = dict(okv)
        one["block_table"], one["seq_lens"] = okv["block_table"][b:b + 1], okv["seq_lens"][b:b + 1]
        ref = O.draft(WIDE, W, h[b:b + 1, :n_ext[b]], tok[b:b + 1, :n_ext[b]], one, K, ids, forced=got["drafts"][b:b + 1])
        ids_match(got["drafts"][b], ref["drafts"], ref["gap"], f"drafts b={b}")
        close(got["h_out"][b:b + 1], ref["h_out"], f"h_out b={b}")
    close(O.bf16_to_f64(got["k_pages"]), O.bf16_to_f64(okv["k_pages"]), "K cache")
    close(O.bf16_to_f64(got["v_pages"]), O.bf16_to_f64(okv["v_pages"]), "V cache")
