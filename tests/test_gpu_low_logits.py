"""Strongly negative logits among tokens that are ruled out (-inf, or outside the plausibility mask): a lane may meet nothing
but ruled-out tokens for many vectors, and what it then sums must not be measured against an exponent of its own making.  Everything
against the oracle, in every form of a run."""
import numpy as np
import pytest
import torch

import helpers
from paper_2502_01662_b200 import COS_ROW_NONFINITE, COS_RUN_ALL_RESIDUALS, synth

pytestmark = pytest.mark.gpu
ENS, LOGIT = synth.COMBINE_PROB_ENSEMBLE, synth.COMBINE_LOGIT_LINEAR

# combine, weights, temperature, vocab, dtype, mask_model, shift, ruled out: every token but runs of 5 in 200, or from a token on
CASES = [
    (ENS, (0.6, 0.4), 0.1, 20008, "bf16", -1, -14.0, "runs"),
    (ENS, (0.6, 0.4), 1.0, 32000, "f32", -1, -110.0, 29000),      # a padded vocabulary: the last shares hold padding alone
    (ENS, (0.6, 0.4), 1.0, 32001, "bf16", -1, -110.0, 29000),
    (ENS, (0.4, 0.3, 0.2, 0.1), 0.7, 12808, "f16", -1, -90.0, "runs"),
    (ENS, (0.3, 0.25, 0.2, 0.15, 0.1), 1.0, 9001, "bf16", -1, -110.0, "runs"),
    (ENS, (0.6, 0.4), 1.0, 600000, "bf16", -1, -110.0, 300000),   # long shares
    (LOGIT, (1.0, -0.5), 1.0, 32000, "bf16", 0, -230.0, None),
    (LOGIT, (1.0, -0.5), 1.0, 9001, "f16", 1, -230.0, None),
    (LOGIT, (1.0, 0.5, -0.5), 1.0, 32000, "f32", 0, -120.0, None),
    (LOGIT, (1.0, 0.5, -0.5), 1.0, 20008, "bf16", -1, -120.0, None),
]


def _inputs(case):
    combine, weights, temperature, vocab, dtype, mask_model, shift, out = case
    w = synth.Workload("low", len(weights), combine, weights, temperature, 3, 3, vocab, dtype, "gauss", sigma=2.0, rho=0.85,
                       proposer_rule="cycle", mask_model=mask_model, mask_alpha=0.05 if mask_model >= 0 else 1.0)
    logits = synth.make_logits(w, "cuda") + shift
    x = torch.arange(vocab, device="cuda")
    if out == "runs":
        logits[..., x % 200 >= 5] = -float("inf")
    elif out is not None:
        logits[..., out:] = -float("inf")
    proposer = synth.make_proposer(w)
    drafts = synth.make_drafts(w, logits, proposer)
    return w, {"logits": logits, "drafts": torch.as_tensor(drafts, device="cuda"), "proposer": torch.as_tensor(proposer, device="cuda"),
               "seed": w.verify_seed, "offset": 5}


@pytest.mark.parametrize("case", CASES, ids=lambda c: "-".join(str(x) for x in c))
def test_low_logits_match_the_oracle(case):
    w, inputs = _inputs(case)
    ref = helpers.run_oracle(w, inputs)
    gpu = helpers.run_gpu(w, inputs, diag=True, lse=True, flags=COS_RUN_ALL_RESIDUALS)
    assert not np.any(gpu["row_status"] & COS_ROW_NONFINITE)
    assert np.all(np.isfinite(gpu["lse"]))
    helpers.check_parity(w, gpu, ref)
    plain = helpers.run_gpu(w, inputs)
    for k in ("accept_count", "out_tokens", "row_status"):
        assert np.array_equal(plain[k], gpu[k]), k


@pytest.mark.parametrize("form", [1, 2])
@pytest.mark.parametrize("case", [c for c in CASES if c[3] % 8 == 0 and c[5] < 0 and len(c[1]) <= 4], ids=lambda c: "-".join(str(x) for x in c))
def test_low_logits_in_the_one_launch_forms(case, form):
    w, inputs = _inputs(case)
    v = helpers.make_verifier(w)
    try:
        v.set_one_launch(form)
        gpu = helpers.run_gpu(w, inputs, verifier=v, diag=True)
    finally:
        v.close()
    assert not np.any(gpu["row_status"] & COS_ROW_NONFINITE)
    helpers.check_parity(w, gpu, helpers.run_oracle(w, inputs))


# Logits of two heights, 126 to 128 powers of two apart: as far as a 32-bit sum reaches from the reference of its first vector.
FAR = [(combine, n, dtype, where) for combine, n in ((ENS, 1), (ENS, 2), (ENS, 3), (LOGIT, 1), (LOGIT, 2), (LOGIT, 3)) for dtype in ("f32", "bf16")
       for where in ("scattered", "behind", "long")]


@pytest.mark.parametrize("form", [0, 1, 2])
@pytest.mark.parametrize("case", FAR, ids=lambda c: "-".join(str(x) for x in c))
def test_sums_far_above_their_reference(case, form):
    """A warp adds up lanes whose references differ by more than a 32-bit power of two can hold ("scattered": the high tokens lie in
    the first vectors of some lanes only), and lanes whose sums together are more than 32 bits hold ("behind": one high token a
    lane, none in a first vector)."""
    combine, n, dtype, where = case
    weights = {1: (1.0,), 2: (0.5, 0.5), 3: (0.5, 0.25, 0.25)}[n]
    E, V = (4, 8192) if dtype == "f32" else (8, 16384)
    if where == "long":
        V = 800000
    w = synth.Workload("far", n, combine, weights, 1.0, 2, 2, V, dtype, "gauss", proposer_rule="zero")
    g = torch.Generator(device="cuda").manual_seed(7)
    high = torch.zeros(V, dtype=torch.bool, device="cuda")
    if where == "behind":
        high[32 * E:64 * E:E] = True
    else:
        high = torch.rand(V, generator=g, device="cuda") < 0.02
    logits = torch.where(high, 44.25, -44.0).to(w.torch_dtype).expand(n, 2, 3, V).clone()
    drafts = torch.nonzero(high)[:2].flatten().to(torch.int32).repeat(2, 1)
    inputs = {"logits": logits, "drafts": drafts, "proposer": torch.zeros(2, dtype=torch.int32, device="cuda"), "seed": 11, "offset": 3}
    v = helpers.make_verifier(w)
    try:
        v.set_one_launch(form)
        gpu = helpers.run_gpu(w, inputs, verifier=v, diag=True)
    finally:
        v.close()
    assert not np.any(gpu["row_status"] & COS_ROW_NONFINITE)
    helpers.check_parity(w, gpu, helpers.run_oracle(w, inputs, native=True))
