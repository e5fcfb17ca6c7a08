"""T = 0 at logit level: the argmax of the combined logits is the one of the fp64 values, lowest index among equals, whatever
the sweep could rule out in fp32.  Inputs on which that is close: everything equal, few distinct values, values closer than fp32
can tell; at the sizes where batches of vectors and shares end.  Against the oracle, in every entry point."""
import numpy as np
import pytest
import torch

import helpers
from paper_2502_01662_b200 import synth
from paper_2502_01662_b200.binding import CosVerifier, run_static

pytestmark = pytest.mark.gpu
LOGIT = synth.COMBINE_LOGIT_LINEAR
WEIGHTS = {1: (1.0,), 2: (1.5, -0.5), 3: (1.0, 0.5, -0.5), 4: (0.7, 0.6, -0.4, 0.1)}

CASES = [(kind, n, vocab, dtype, mask)
         for kind in ("equal", "steps", "close")
         for n, vocab, dtype, mask in ((1, 4096, "bf16", -1), (2, 7, "f32", -1), (2, 8192, "f32", -1), (2, 8201, "f16", 0), (2, 33000, "bf16", 1),
                                       (3, 8192, "f32", 2), (3, 9001, "bf16", -1), (4, 2056, "f32", 3))]


@pytest.mark.parametrize("case", CASES, ids=lambda c: "-".join(str(x) for x in c))
def test_argmax_is_the_exact_one(case):
    kind, n, vocab, dtype, mask = case
    w = synth.Workload("argmax", n, LOGIT, WEIGHTS[n], 0.0, 5, 4, vocab, dtype, "gauss", sigma=2.5, rho=0.8, proposer_rule="cycle",
                       mask_model=mask, mask_alpha=0.3 if mask >= 0 else 1.0)
    logits = synth.make_logits(w, "cuda").float()
    if kind == "equal":
        logits = torch.full_like(logits, 1.25)
    elif kind == "steps":
        logits = logits.round()                                  # tens of tokens share the maximum
    else:
        # the combined logits lie within a few fp32 roundings of one another (1000 each model; bf16 and f16 keep few of them apart)
        logits = 1000.0 + logits * 2.0 ** -12
        logits[:, 1, :, vocab // 2:] += 2.0 ** -12               # a row whose last tokens win
    logits = logits.to(w.torch_dtype)
    proposer = synth.make_proposer(w)
    drafts = synth.make_drafts(w, logits, proposer)
    drafts[:, 0] = synth.make_drafts(w, logits, np.zeros_like(proposer))[:, 0]
    inputs = {"logits": logits, "drafts": torch.as_tensor(drafts, device="cuda"), "proposer": torch.as_tensor(proposer, device="cuda"),
              "seed": w.verify_seed, "offset": 0}
    ref = helpers.run_oracle(w, inputs)
    gpu = helpers.run_gpu(w, inputs, diag=True)
    helpers.check_parity(w, gpu, ref)
    B, P = w.batch, w.gamma + 1
    outs = CosVerifier._alloc_outs(B, P, vocab, "cuda", False, False)
    run_static(n, LOGIT, WEIGHTS[n], 0.0, w.gamma, vocab, logits, inputs["drafts"], inputs["proposer"], w.verify_seed, 0, mask_model=mask,
               mask_alpha=w.mask_alpha, outs=outs)
    v = helpers.make_verifier(w, host_staging=True)
    try:
        host = v.run_host(logits.cpu(), inputs["drafts"].cpu(), inputs["proposer"].cpu(), w.verify_seed, 0)
    finally:
        v.close()
    for k in ("accept_count", "out_tokens", "row_status"):
        assert np.array_equal(outs[k].cpu().numpy(), gpu[k]), k
        assert np.array_equal(host[k].numpy(), gpu[k]), k
