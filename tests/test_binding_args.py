"""The arguments that the binding hands to the library (no GPU needed: addresses of host tensors do as well)."""
import torch

from paper_2502_01662_b200.binding import COS_DTYPE_F32, CosVerifier


def _verifier(n=2, gamma=3, vocab=16):
    v = CosVerifier.__new__(CosVerifier)      # without a context
    v._dims, v._dtype = (n, gamma + 1, vocab), COS_DTYPE_F32
    return v


def test_outputs_of_the_caller_may_hold_entries_of_their_own():
    B, P = 2, 4
    logits = torch.zeros(2, B, P, 16)
    drafts, proposer = torch.zeros(B, P - 1, dtype=torch.int32), torch.zeros(B, dtype=torch.int32)
    outs = CosVerifier._alloc_outs(B, P, 16, "cpu", True, True)
    outs["request"] = "abc"                   # the caller's own
    outs["when"] = None
    a = _verifier()._fill_args(logits, drafts, proposer, 1, 2, 0, 0, outs)
    assert a.out_tokens == outs["out_tokens"].data_ptr() and a.accept_count == outs["accept_count"].data_ptr()
    assert a.row_status == outs["row_status"].data_ptr() and a.bonus_prob == outs["bonus_prob"].data_ptr()
    assert a.diag == outs["diag"].data_ptr() and a.dump_r == outs["r"].data_ptr() and a.lse is None
    few = {k: outs[k] for k in ("accept_count", "out_tokens", "row_status")}
    b = _verifier()._fill_args(logits, drafts, proposer, 1, 2, 0, 0, few)
    assert b.bonus_prob is None and b.diag is None and b.dump_r is None
