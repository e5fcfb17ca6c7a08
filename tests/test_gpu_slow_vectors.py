"""What the drawing sweep sums beside its fast loop: the vectors that hold a big token, and the ragged ends of a row."""
import numpy as np
import pytest
import torch

import helpers
from paper_2502_01662_b200 import synth

pytestmark = pytest.mark.gpu
ENS, LOGIT = synth.COMBINE_PROB_ENSEMBLE, synth.COMBINE_LOGIT_LINEAR


@pytest.mark.parametrize("cluster_size", [0, 1])
@pytest.mark.parametrize("vocab", [1000, 1001])         # a vector with a big token, and one that is a ragged end as well
@pytest.mark.parametrize("combine,n", [(ENS, 2), (ENS, 3), (ENS, 4), (ENS, 5), (ENS, 8), (LOGIT, 2)])
def test_small_tokens_beside_a_big_one_keep_their_bits(combine, n, vocab, cluster_size):
    """Logits in whole powers of two (log2(e) / T is 1), so that every exponential is exact.  The first vector holds a big token without residual
    mass, one of 2^-8 and six of 2^-33 of it: added up in 32 bits the six are lost, which is 2e-7 of the residual mass.  In 64 bits
    the mass is exact until it is stored."""
    weights = (1.0, 0.0) if combine == LOGIT else tuple(0.5 ** (k + 1) for k in range(n - 1)) + (0.5 ** (n - 1),)
    w = synth.Workload("bits", n, combine, weights, float(np.float32(1.4426950408889634)), 2, 2, vocab, "bf16", "gauss", proposer_rule="zero")
    assert np.float32(1.4426950408889634 / w.temperature) == 1.0
    logits = torch.full((n, 2, 3, vocab), -200.0)
    logits[0, ..., :8] = torch.tensor([0.0, -8.0] + [-33.0] * 6)
    logits[1:, ..., :8] = torch.tensor([0.0, -11.0] + [-40.0] * 6)
    drafts = torch.full((2, 2), vocab, dtype=torch.int32)        # outside the vocabulary: a token is drawn from the residual
    p, q = (2.0 ** logits[k, 0, 0].double().numpy() for k in (0, 1))
    p, q = p / p.sum(), q / q.sum()
    want = (1.0 if combine == LOGIT else 0.5) * np.maximum(0.0, p - q).sum()
    v = helpers.make_verifier(w, cluster_size=cluster_size)
    try:
        got = v.run(logits.to(torch.bfloat16).cuda(), drafts.cuda(), torch.ones(2, dtype=torch.int32, device="cuda"), 3, 1, diag=True)
        S = got["diag"][:, 0, 3].double().cpu().numpy()
    finally:
        v.close()
    # half a unit of the last place for the store, and a tenth of one for the few 64-bit operations and the tokens of 2^-200
    assert np.all(np.abs(S - want) <= 0.6 * np.spacing(np.float32(want))), (S - want) / want
    assert np.all(got["accept_count"].cpu().numpy() == 0) and np.all(got["out_tokens"][:, 0].cpu().numpy() < 8)


@pytest.mark.parametrize("cluster_size", [0, 1])
@pytest.mark.parametrize("n,vocab,dtype,sigma", [(3, 4099, "bf16", 6.0), (4, 23, "f32", 2.0), (5, 3, "bf16", 3.0), (5, 4097, "f32", 8.0), (6, 257, "f16", 1.0),
                                                 (6, 20000, "bf16", 6.0), (7, 23, "f32", 2.0), (8, 9001, "bf16", 8.0), (8, 64, "f16", 0.1), (8, 32768, "f32", 5.0)])
def test_many_channels_with_many_big_tokens(n, vocab, dtype, sigma, cluster_size):
    """Nothing but big tokens, a few among many, ragged ends at both sides of a row, several in a warp's vectors at once."""
    w = synth.Workload("many", n, ENS, tuple([1.0 - 0.125 * (n - 1)] + [0.125] * (n - 1)), 1.0, 6, 3, vocab, dtype, "gauss", sigma=sigma, rho=0.6,
                       proposer_rule="cycle")
    inputs = synth.make_inputs(w, "cuda")
    drafts = inputs["drafts"].clone()
    drafts[0, 0] = vocab
    inputs = dict(inputs, drafts=drafts)
    ref = helpers.run_oracle(w, inputs)
    v = helpers.make_verifier(w, cluster_size=cluster_size)
    try:
        for opts in ({}, {"flags": 1}):     # the token's position alone, and every position's mass
            helpers.check_parity(w, helpers.run_gpu(w, inputs, verifier=v, diag=True, **opts), ref)
    finally:
        v.close()
