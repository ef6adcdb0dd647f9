"""What a context accepts, several contexts in one process, and a context after a timeout."""
import time
from dataclasses import replace

import numpy as np
import pytest
import torch

from paper_2509_18362_b200 import binding as Bd
from paper_2509_18362_b200 import inputs as I
from tests.gpu_util import copy_kv

pytestmark = pytest.mark.gpu


class Drafter:
    """One context with a seeded draft call of B sequences, E pairs each."""

    def __init__(self, shape, B, E=1, seed=500, max_ctx=None, L=None):
        L = [7 * b % 60 for b in range(B)] if L is None else L
        self.B, self.E, self.kv = B, E, I.paged_kv(shape, L, E + 2, seed + 1)
        self.dW = Bd.to_device(I.mtp_weights(shape, seed))
        self.h = Bd.bf16_tensor(I.hidden_bf16(seed + 2, (B, E, shape.d)))
        self.tok = torch.from_numpy(I.token_ids(seed + 3, (B, E), shape.vocab)).cuda()
        self.ctx = Bd.Context(shape, max_rows=max(8, B * E), max_K=2, max_ctx=max_ctx or max(L) + E + 4)
        self.shape = shape

    def call(self):
        """The call's results as one array of bits, and the status word."""
        dkv = Bd.to_device(copy_kv(self.kv))
        out_d = torch.full((self.B, 2), -1, dtype=torch.int32, device="cuda")
        out_h = torch.zeros((self.B, 2, self.shape.d), dtype=torch.bfloat16, device="cuda")
        st = torch.zeros(1, dtype=torch.int32, device="cuda")
        self.ctx.fastmtp_draft(Bd.mtp_w(self.dW), self.h, self.tok, Bd.kv(dkv), self.B, 2, None, out_d, out_h, None, st, max_ext=self.E)
        torch.cuda.synchronize()
        return np.concatenate([Bd.bf16_bits(out_h).ravel(), out_d.cpu().numpy().ravel().astype(np.uint16)]), int(st.item())

    def bits(self):
        got, status = self.call()
        assert status == 0
        return got


WIDE = replace(I.TINY, d=2048, vocab=1500)


@pytest.mark.parametrize("which,shape,B,E", [
    (1, WIDE, 1, 4),                                   # the persistent kernel changes its shared-memory layout between the steps
    (1, replace(I.TINY, d=3072, vocab=1500), 1, 4),    # and its projection restages
    (3, I.TINY, 12, 1), (3, I.TINY, 12, 4),            # batched attention, one and several rows: tile copies
    (3, replace(I.TINY, page_size=5), 12, 1), (3, replace(I.TINY, page_size=5), 12, 4),       # 16-byte copies
])
def test_a_wait_that_runs_out_leaves_the_context_usable(which, shape, B, E):
    """A wait of the next call cannot end and is limited to 20 ms: the call returns soon after with the timeout flag, the next
    one gives the bits of the one before."""
    a = Drafter(shape, B, E)
    want = a.bits()
    a.ctx.fmtp_selftest_inject_wait_timeout(20, which)
    t0 = time.time()
    _, status = a.call()
    assert status & Bd.DEV_TIMEOUT and 0.015 < time.time() - t0 < 2.0
    assert np.array_equal(a.bits(), want)
    a.ctx.close()


@pytest.mark.parametrize("batched,first,second", [
    (True, (I.TINY, 16), (I.TINY, 4)),                 # the operand's widths differ
    (True, (I.TINY, 64), (I.TINY, 20)),
    (False, (WIDE, 1), (I.TINY, 1)),                   # the persistent kernel: one instantiation, two footprints
    (False, (WIDE, 1, 4), (I.TINY, 1, 4)),
    (False, (WIDE, 6), (I.TINY, 8)),
])
def test_contexts_of_different_footprints_take_turns(batched, first, second, monkeypatch):
    """A kernel's shared-memory limit belongs to the device: a context with a small footprint must not take away what another
    one has been given. Same bits in every turn."""
    monkeypatch.setenv("FMTP_BATCHED_MIN", "1" if batched else "99")
    a, b = Drafter(*first), None
    want = a.bits()
    b = Drafter(*second)
    other = b.bits()
    for _ in range(2):
        assert np.array_equal(a.bits(), want)
        assert np.array_equal(b.bits(), other)
    a.ctx.close()
    b.ctx.close()


def test_the_longest_context_is_accepted_and_gives_the_same_bits():
    """The persistent kernel keeps a context's chunk maxima and sums in shared memory, which bounds max_ctx: beside two ring
    stages of 16 KB, 5.5 KB of fixed data and 1280 bytes, eight bytes per 64 positions fit up to this length at this width."""
    most = 24096 * 64
    a, b = Drafter(I.TINY, 1, L=[700]), Drafter(I.TINY, 1, L=[700], max_ctx=most)
    assert np.array_equal(a.bits(), b.bits())
    assert b.ctx.launch_count == 1
    a.ctx.close()
    b.ctx.close()
    with pytest.raises(Bd.FastMTPError):
        Drafter(I.TINY, 1, max_ctx=most + 16 * 64)


# more than 256 MB of weights per layer: the sizes at which the switch points come earlier
LARGE = I.Shape(d=2560, n_q_heads=2, n_kv_heads=1, head_dim=128, ffn=16384, vocab=300, n_layers=1)


def test_the_switch_point_variable_overrides_the_row_rule_of_drafts(monkeypatch):
    """Five pairs of one sequence at a large width: several kernels by default, one launch where FMTP_BATCHED_MIN says so."""
    monkeypatch.delenv("FMTP_BATCHED_MIN", raising=False)
    a = Drafter(LARGE, 1, 5)
    a.bits()
    assert a.ctx.launch_count > 3
    a.ctx.close()
    monkeypatch.setenv("FMTP_BATCHED_MIN", "9")
    b = Drafter(LARGE, 1, 5)
    b.bits()
    assert b.ctx.launch_count == 1
    b.ctx.close()


def test_hidden_states_of_two_sequences_may_start_anywhere():
    """A target call of fewer than three sequences takes out_h at any address; from three on it has to be a multiple of 16."""
    Wt = Bd.to_device(I.target_weights(LARGE, 510))
    w, keep = Bd.target_w(Wt)
    for B in (1, 2, 3):
        dkv = Bd.to_device(I.paged_kv(LARGE, [40, 9, 0][:B], 1, 511))
        tok = torch.from_numpy(I.token_ids(512, (B, 1), LARGE.vocab)).cuda()
        ctx = Bd.Context(LARGE, max_rows=8, max_K=1, max_ctx=64)
        pool = torch.zeros(B * LARGE.d + 8, dtype=torch.bfloat16, device="cuda")
        ctx.fastmtp_target_step(w, tok, [Bd.kv(dkv)], B, 1, pool[:B * LARGE.d])
        want = Bd.bf16_bits(pool[:B * LARGE.d])
        pool.zero_()
        if B < 3:
            ctx.fastmtp_target_step(w, tok, [Bd.kv(dkv)], B, 1, pool[3:])
            got = Bd.bf16_bits(pool)
            assert np.array_equal(got[3:3 + B * LARGE.d], want)
            assert not got[:3].any() and not got[3 + B * LARGE.d:].any()
        else:
            with pytest.raises(Bd.FastMTPError):
                ctx.fastmtp_target_step(w, tok, [Bd.kv(dkv)], B, 1, pool[3:])
        ctx.close()
    del keep


@pytest.mark.parametrize("batched", [False, True])
@pytest.mark.parametrize("E", [1, 3])
def test_a_committed_length_without_bounds_is_flagged(E, batched, monkeypatch):
    """The largest length an int32 holds: no slot for the sequence's positions, the other sequence is not affected."""
    monkeypatch.setenv("FMTP_BATCHED_MIN", "1" if batched else "99")
    a, one = Drafter(I.TINY, 2, E, L=[5, 70]), Drafter(I.TINY, 1, E, L=[5])
    a.kv["seq_lens"][1] = 2 ** 31 - 1
    one.kv["k_pages"], one.kv["v_pages"] = a.kv["k_pages"], a.kv["v_pages"]
    one.kv["block_table"] = a.kv["block_table"][:1]
    one.h, one.tok = a.h[:1].contiguous(), a.tok[:1].contiguous()
    (got, status), want = a.call(), one.bits()
    n = 2 * I.TINY.d
    assert status & Bd.DEV_BAD_POS and not status & Bd.DEV_TIMEOUT
    assert np.array_equal(got[:n], want[:n]) and np.array_equal(got[2 * n:2 * n + 2], want[n:])
    a.ctx.close()
    one.ctx.close()
