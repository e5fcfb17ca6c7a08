"""Runs whose rows are all at work at once, each on a cluster of blocks, in one launch: at the sizes where the clusters, the shares of a
row and the rule change, against the oracle; and on settled inputs with an offset that is written just before the call."""
import numpy as np
import pytest
import torch

import helpers
from paper_2502_01662_b200 import synth
from paper_2502_01662_b200.binding import COS_RUN_INPUTS_SETTLED, run_static

pytestmark = pytest.mark.gpu

ENS, LOGIT = synth.COMBINE_PROB_ENSEMBLE, synth.COMBINE_LOGIT_LINEAR
WEIGHTS = {1: (1.0,), 2: (0.6, 0.4), 3: (0.5, 0.3, 0.2), 4: (0.4, 0.3, 0.2, 0.1), 5: (0.3, 0.25, 0.2, 0.15, 0.1)}
LINEAR = {1: (1.0,), 2: (1.5, -0.5), 3: (1.0, 0.5, -0.5)}

CASES = [
    # combine, n, temperature, batch, gamma, vocab, dtype, mask_model
    (ENS, 2, 1.0, 1, 4, 5, "bf16", -1),              # less than a vector, clusters of 16
    (ENS, 2, 1.0, 1, 0, 32000, "f32", -1),           # one position
    (ENS, 2, 0.7, 7, 4, 2057, "bf16", -1),           # rows that start anywhere
    (ENS, 2, 1.0, 8, 17, 4096, "f16", -1),           # two tiles of positions, smaller clusters
    (ENS, 2, 1.0, 40, 5, 9000, "bf16", -1),          # clusters of three or so
    (ENS, 2, 1.0, 74, 3, 2048, "bf16", -1),          # of two
    (ENS, 2, 1.0, 148, 2, 2048, "bf16", -1),         # of one
    (ENS, 3, 0.7, 7, 4, 64008, "bf16", -1),
    (ENS, 4, 1.0, 7, 4, 32000, "f32", -1),
    (ENS, 2, 1.0, 2, 140, 1000, "bf16", -1),         # more positions than warps for each model: shares cut across them
    (ENS, 5, 0.0, 7, 5, 32003, "f16", -1),
    (ENS, 2, 0.0, 33, 6, 32000, "bf16", -1),
    (LOGIT, 1, 1.0, 3, 4, 9001, "bf16", -1),
    (LOGIT, 2, 1.0, 8, 17, 2049, "f16", 1),
    (LOGIT, 2, 0.7, 30, 4, 20000, "bf16", -1),
    (LOGIT, 3, 1.0, 6, 5, 16000, "f32", 2),
    (LOGIT, 2, 0.0, 30, 17, 8003, "bf16", 0),
    (LOGIT, 3, 0.0, 12, 4, 64000, "bf16", -1),
]


def workload(case):
    combine, n, temperature, batch, gamma, vocab, dtype, mask_model = case
    return synth.Workload("rows", n, combine, WEIGHTS[n] if combine == ENS else LINEAR[n], temperature, batch, gamma, vocab, dtype, "gauss",
                          sigma=2.5, rho=0.85, proposer_rule="cycle", mask_model=mask_model, mask_alpha=0.05 if mask_model >= 0 else 1.0)


@pytest.mark.parametrize("case", CASES, ids=lambda c: "-".join(str(x) for x in c))
def test_rows_at_once_match_the_oracle(case):
    combine, n, temperature, batch, gamma, vocab, dtype, mask_model = case
    w = workload(case)
    inputs = synth.make_inputs(w, "cuda")
    # one row agrees with its proposer in everything, so that the bonus position is reached for certain; one holds a NaN
    logits = inputs["logits"].clone()
    logits[:, 0] = logits[int(inputs["proposer"][0]), 0].clone()
    if batch > 1:
        logits[n - 1, batch - 1, gamma, vocab // 2] = float("nan")
    inputs = dict(inputs, logits=logits)
    ref = helpers.run_oracle(w, inputs, native=True)
    v, staged = helpers.make_verifier(w), helpers.make_verifier(w, cluster_size=16)   # (a bound on the streaming launch: never at once)
    try:
        assert v.info()["rows_at_once"] and not staged.info()["rows_at_once"]
        got = helpers.run_gpu(w, inputs, verifier=v, diag=True, lse=True)
        again = helpers.run_gpu(w, inputs, verifier=v)                       # the scratch was left clean
        apart = helpers.run_gpu(w, inputs, verifier=staged, diag=True, lse=True)
    finally:
        v.close()
        staged.close()
    helpers.check_parity(w, got, ref)
    for k in ("accept_count", "out_tokens", "row_status"):
        assert np.array_equal(again[k], got[k]), k
        assert np.array_equal(apart[k], got[k]), k
    # the same sums in another order: an argument up to 64 rounds by 2^-19 and a log-sum-exp is stored to 24 bits
    np.testing.assert_allclose(got["lse"], apart["lse"], rtol=1e-6, atol=2e-6)
    host = helpers.make_verifier(w, host_staging=True)
    try:
        h = host.run_host(logits.cpu(), inputs["drafts"].cpu(), inputs["proposer"].cpu(), inputs["seed"], inputs["offset"])
    finally:
        host.close()
    outs = {"accept_count": torch.empty(batch, dtype=torch.int32, device="cuda"), "row_status": torch.empty(batch, dtype=torch.int32, device="cuda"),
            "out_tokens": torch.empty((batch, gamma + 1), dtype=torch.int32, device="cuda")}
    run_static(n, combine, w.weights, temperature, gamma, vocab, logits, inputs["drafts"], inputs["proposer"], inputs["seed"], inputs["offset"],
               mask_model=mask_model, mask_alpha=w.mask_alpha, outs=outs)
    torch.cuda.synchronize()
    for k in ("accept_count", "out_tokens", "row_status"):
        assert torch.equal(h[k], torch.from_numpy(got[k])) and np.array_equal(outs[k].cpu().numpy(), got[k]), k


@pytest.mark.parametrize("offset_on_device", [False, True])
def test_rows_at_once_on_settled_inputs(offset_on_device):
    w = workload((ENS, 2, 1.0, 40, 4, 20008, "bf16", -1))
    inputs = synth.make_inputs(w, "cuda")
    args = (inputs["logits"], inputs["drafts"], inputs["proposer"], inputs["seed"])
    off = torch.zeros(1, dtype=torch.int64, device="cuda")
    step = torch.ones(1 << 22, dtype=torch.int64, device="cuda")
    v = helpers.make_verifier(w)
    try:
        assert v.info()["rows_at_once"]
        torch.cuda.synchronize()
        queued = []
        for k in range(16):
            if offset_on_device:
                off += step.max()
            queued.append(v.run(*args, k + 1, offset_device=off if offset_on_device else None, flags=COS_RUN_INPUTS_SETTLED))
        torch.cuda.synchronize()
        for k, outs in enumerate(queued):
            want = v.run(*args, k + 1)
            for key in ("accept_count", "out_tokens", "row_status"):
                assert torch.equal(outs[key], want[key]), (k, key)
    finally:
        v.close()
