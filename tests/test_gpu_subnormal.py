"""Drafts whose probability under the proposer is the smallest that 64 bits hold, and nothing under the combined distribution (outside the
plausibility mask): a ratio of 0, which no uniform passes, in every form of a run and as the oracle has it."""
import numpy as np
import pytest
import torch

import helpers
from paper_2502_01662_b200 import synth

pytestmark = pytest.mark.gpu


def _inputs(temperature):
    # the largest logit lies behind a lane's first vector, so that the sums' references stay far below it and the probability itself
    # is what is subnormal: exp(-744.2), 1.27 times the smallest number
    w = synth.Workload("subnormal", 2, synth.COMBINE_LOGIT_LINEAR, (1.0, -0.5), temperature, 16, 4, 256, "f32", "gauss", sigma=1.0,
                       mask_model=0, mask_alpha=0.1)
    logits = torch.zeros((2, w.batch, w.gamma + 1, w.vocab))
    logits[1] = -80.0
    logits[1, ..., 200] = 0.0
    logits[0, ..., 10] = -50.0
    logits[1, ..., 10] = -744.2
    drafts = torch.full((w.batch, w.gamma), 10, dtype=torch.int32)
    return w, {"logits": (logits * temperature).cuda(), "drafts": drafts.cuda(), "proposer": torch.ones(w.batch, dtype=torch.int32, device="cuda"),
               "seed": 5, "offset": 3}


@pytest.mark.parametrize("cluster_size", [0, 1])     # in one launch, and in several
@pytest.mark.parametrize("temperature", [1.0, 0.5])
def test_a_ratio_of_zero_is_never_accepted(temperature, cluster_size):
    w, inputs = _inputs(temperature)
    ref = helpers.run_oracle(w, inputs)
    q = ref["q_d"][:, : w.gamma]
    assert np.all((q > 0.0) & (q < 1e-320)) and np.all(ref["r_d"][:, : w.gamma] == 0.0) and np.any(ref["u_acc"][:, 0] < 0.5)
    v = helpers.make_verifier(w, cluster_size=cluster_size)
    try:
        assert v.info()["rows_at_once"] == (cluster_size == 0)
        for opts in ({}, {"diag": True}):
            got = helpers.run_gpu(w, inputs, verifier=v, **opts)
            assert np.all(got["accept_count"] == 0)
            helpers.check_parity(w, got, ref)
    finally:
        v.close()
