"""The down projection's last stage of K, at widths that leave it 16, 480 and 496 of 512 columns, against the CPU oracle: a
stage that is full but for its zero-filled end is read like a full one, and its activations have to be there."""
import pytest

from oracle import fastmtp_oracle as O
from paper_2509_18362_b200 import inputs as I
from tests.gpu_util import close, copy_kv
from tests.test_gpu_draft import check_draft, run_draft_case
from tests.test_gpu_target import GpuTarget

pytestmark = pytest.mark.gpu


def _shape(d, ffn, n_layers=1):
    return I.Shape(d=d, n_q_heads=4, n_kv_heads=2, head_dim=64, ffn=ffn, vocab=1024, n_layers=n_layers, rms_eps=1e-6,
                   rope_theta=1e4, page_size=16)


@pytest.mark.parametrize("batched", [False, True])
@pytest.mark.parametrize("B", [1, 2, 4, 6])
@pytest.mark.parametrize("ffn", [496, 528, 992, 1008, 2544])
def test_draft(ffn, B, batched, monkeypatch):
    monkeypatch.setenv("FMTP_BATCHED_MIN", "1" if batched else "99")
    got, ref = run_draft_case(_shape(1024, ffn), 40 + ffn % 31 + B, B, [9 * b + 3 for b in range(B)], 2, 300)
    check_draft(got, ref, f"ffn={ffn} B={B} batched={batched}")
    assert (got["launches"] == 1) == (not batched)
    for b in range(B):
        close(got["logits"][b, 1], O.head_logits(ref["h_out"][b, 1], ref["W"]["lm_head"], ref["ids"]), f"logits b={b}")


@pytest.mark.parametrize("B,M", [(1, 1), (1, 4), (1, 7), (3, 2)])
@pytest.mark.parametrize("ffn", [496, 1008, 2544])
def test_target(ffn, B, M, monkeypatch):
    monkeypatch.setenv("FMTP_BATCHED_MIN", "99")
    s = _shape(2048, ffn, 2)
    kvs = [I.paged_kv(s, [11 * b + 5 for b in range(B)], M, 51 + l) for l in range(2)]
    Wt = I.target_weights(s, 50 + ffn % 31)
    gpu = GpuTarget(s, Wt, kvs, 64)
    t = I.token_ids(53, (B, M), s.vocab)
    h, l, _ = gpu.step(t)
    assert gpu.ctx.launch_count == 1
    rh, rl = O.target_forward(s, Wt, t, [copy_kv(kv) for kv in kvs])
    close(h.float().cpu().numpy(), rh, "hidden states")
    close(l.float().cpu().numpy(), rl, "logits")
    gpu.close()
