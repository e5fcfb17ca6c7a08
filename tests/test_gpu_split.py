"""How a run is split over the device, at the sizes where the split changes: shares of the streaming launch that are padded,
cut across positions, one model's each or long; tiles of 16 positions in the decisions; clusters of one to eight blocks with one
to eight chunks a warp in the drawing launch; ragged rows.  Everything against the oracle, residual masses at every position."""
import pytest
import torch

import helpers
from paper_2502_01662_b200 import synth
from paper_2502_01662_b200.binding import COS_RUN_ALL_RESIDUALS

pytestmark = pytest.mark.gpu

ENS, LOGIT = synth.COMBINE_PROB_ENSEMBLE, synth.COMBINE_LOGIT_LINEAR
WEIGHTS = {1: (1.0,), 2: (0.6, 0.4), 3: (0.5, 0.3, 0.2), 4: (0.4, 0.3, 0.2, 0.1), 5: (0.3, 0.25, 0.2, 0.15, 0.1),
           8: (0.2, 0.2, 0.15, 0.15, 0.1, 0.1, 0.05, 0.05)}
LINEAR = {1: (1.0,), 2: (1.5, -0.5), 3: (1.0, 0.5, -0.5)}

CASES = [
    # combine, n, temperature, batch, gamma, vocab, dtype, mask_model
    (ENS, 2, 1.0, 3, 3, 5, "bf16", -1),              # less than a vector
    (ENS, 2, 1.0, 2, 4, 17, "f16", -1),              # two vectors and a ragged end
    (ENS, 3, 0.7, 2, 4, 2048, "bf16", -1),           # one share of 256 vectors a row
    (ENS, 2, 1.0, 2, 4, 2056, "bf16", -1),           # and one vector more
    (ENS, 4, 1.0, 2, 5, 4111, "f32", -1),            # rows that start anywhere
    (ENS, 1, 1.0, 3, 5, 5000, "bf16", -1),           # decisions in a launch of their own
    (ENS, 5, 0.7, 2, 5, 3001, "bf16", -1),
    (ENS, 8, 1.0, 2, 3, 4096, "f32", -1),
    (ENS, 2, 1.0, 2, 15, 1000, "bf16", -1),          # 16 positions: a tile
    (ENS, 2, 1.0, 2, 16, 1000, "bf16", -1),          # and one more
    (ENS, 8, 0.0, 2, 33, 1003, "f16", -1),
    (ENS, 2, 1.0, 180, 33, 264, "bf16", -1),         # more positions than warps: shares cut across them
    (ENS, 2, 0.0, 180, 33, 264, "f32", -1),
    (ENS, 2, 1.0, 8, 7, 96004, "f32", -1),           # long shares
    (ENS, 3, 1.0, 10, 5, 100003, "f32", -1),
    (ENS, 2, 1.0, 1, 2, 600000, "bf16", -1),         # several chunks a warp
    (ENS, 4, 1.0, 160, 1, 20000, "bf16", -1),        # one block a position
    (LOGIT, 1, 1.0, 2, 4, 4099, "bf16", -1),
    (LOGIT, 2, 1.0, 2, 17, 2049, "f16", 0),
    (LOGIT, 2, 1.0, 40, 8, 9000, "bf16", 1),
    (LOGIT, 3, 0.7, 3, 4, 8192, "f32", 2),
    (LOGIT, 3, 0.0, 3, 17, 4097, "bf16", 0),
]


@pytest.mark.parametrize("case", CASES, ids=lambda c: "-".join(str(x) for x in c))
def test_split_matches_the_oracle(case):
    combine, n, temperature, batch, gamma, vocab, dtype, mask_model = case
    weights = WEIGHTS[n] if combine == ENS else LINEAR[n]
    w = synth.Workload("split", n, combine, weights, temperature, batch, gamma, vocab, dtype, "gauss", sigma=2.5, rho=0.85,
                       proposer_rule="cycle", mask_model=mask_model, mask_alpha=0.05 if mask_model >= 0 else 1.0)
    inputs = synth.make_inputs(w, "cuda")
    # one row agrees with its proposer in everything, so that the bonus position is reached for certain; one holds a NaN
    logits = inputs["logits"].clone()
    logits[:, 0] = logits[int(inputs["proposer"][0]), 0].clone()
    logits[n - 1, batch - 1, gamma, vocab // 2] = float("nan")
    inputs = dict(inputs, logits=logits)
    gpu = helpers.run_gpu(w, inputs, diag=temperature > 0.0, flags=COS_RUN_ALL_RESIDUALS if temperature > 0.0 else 0)
    ref = helpers.run_oracle(w, inputs, native=True)
    helpers.check_parity(w, gpu, ref)
    host = helpers.make_verifier(w, host_staging=True)
    try:
        got = host.run_host(logits.cpu(), inputs["drafts"].cpu(), inputs["proposer"].cpu(), inputs["seed"], inputs["offset"])
    finally:
        host.close()
    for k in ("accept_count", "out_tokens", "row_status"):
        assert torch.equal(got[k], torch.from_numpy(gpu[k])), k
