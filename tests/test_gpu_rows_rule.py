"""Which runs are one launch: rows that start anywhere and positions of few tokens keep a row's cluster longer than whole rows of aligned
vectors do; and the same rows either way."""
import pytest
import torch

import helpers
from paper_2502_01662_b200 import synth

pytestmark = pytest.mark.gpu
ENS, LOGIT = synth.COMBINE_PROB_ENSEMBLE, synth.COMBINE_LOGIT_LINEAR


@pytest.mark.parametrize("combine,n,temperature,batch,gamma,vocab,dtype,mask_model,at_once", [
    (ENS, 2, 1.0, 7, 4, 50001, "bf16", -1, True), (ENS, 2, 1.0, 33, 4, 50001, "bf16", -1, False), (ENS, 2, 1.0, 24, 4, 50001, "f32", -1, False),
    (LOGIT, 2, 1.0, 7, 4, 50001, "f32", 0, True), (LOGIT, 2, 1.0, 24, 4, 50001, "f32", 0, False), (LOGIT, 2, 1.0, 33, 4, 50001, "f32", -1, False),
    (LOGIT, 2, 0.0, 33, 4, 50001, "bf16", 0, None), (ENS, 2, 0.0, 33, 4, 50001, "bf16", -1, None), (LOGIT, 2, 0.0, 2, 2, 252337, "bf16", -1, None),
    (LOGIT, 2, 1.0, 1, 499, 7, "bf16", -1, False), (ENS, 2, 1.0, 1, 499, 7, "bf16", -1, False), (LOGIT, 2, 1.0, 7, 499, 100, "bf16", -1, False),
    (ENS, 2, 1.0, 1, 499, 1000, "bf16", -1, False), (ENS, 4, 1.0, 7, 49, 4000, "bf16", -1, False), (LOGIT, 2, 1.0, 1, 49, 7, "bf16", -1, True)])
def test_runs_of_one_launch(combine, n, temperature, batch, gamma, vocab, dtype, mask_model, at_once):
    weights = (1.0, -0.5) if combine == LOGIT else (1.0 / n,) * n
    w = synth.Workload("rule", n, combine, weights, temperature, batch, gamma, vocab, dtype, "gauss", sigma=2.0, rho=0.85, proposer_rule="cycle",
                       mask_model=mask_model, mask_alpha=0.05 if mask_model >= 0 else 1.0)
    g = torch.Generator(device="cuda").manual_seed(3)
    logits = torch.randn((1, batch, gamma + 1, vocab), generator=g, device="cuda") * 2.0
    logits = (logits + torch.randn((n, batch, gamma + 1, vocab), generator=g, device="cuda")).to(w.torch_dtype)
    drafts = torch.randint(0, vocab, (batch, gamma), generator=g, device="cuda").to(torch.int32)
    drafts[:, 0] = logits[0, :, 0].float().argmax(-1).to(torch.int32)
    proposer = torch.zeros(batch, dtype=torch.int32, device="cuda")
    v, staged = helpers.make_verifier(w), helpers.make_verifier(w, cluster_size=16)
    try:
        v.set_stage_timing(True)
        got = v.run(logits, drafts, proposer, 5, 1)
        assert at_once is None or (len(v.stage_ms()) == 1) == at_once      # (at T = 0 the stages do not tell)
        want = staged.run(logits, drafts, proposer, 5, 1)
        torch.cuda.synchronize()
        for k in ("accept_count", "row_status"):
            assert torch.equal(got[k], want[k]), k
        # (a token where a uniform falls between the sums of the two ways may differ: not in more than one row)
        assert int((got["out_tokens"] != want["out_tokens"]).any(dim=1).sum()) <= 1
    finally:
        v.close()
        staged.close()
