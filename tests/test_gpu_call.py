"""The native form of CosVerifier.run (plain tensors, outputs of its own) against the long one (a stream of the caller's): the same
outputs, shapes and types, and the same complaints."""
import pytest
import torch

import helpers
from paper_2502_01662_b200 import CosVerifyError, synth

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("name,kw", [("cfg1", dict(batch=2, vocab=4100, gamma=3)), ("cfg2", dict(batch=5, vocab=9001, gamma=4)),
                                     ("cfg5_greedy", dict(batch=3, vocab=8192, gamma=2)), ("cfg3", dict(batch=4, vocab=2048, gamma=0))])
def test_both_ways_of_a_call_agree(name, kw):
    w = synth.CONFIGS[name].scaled(**kw)
    inputs = synth.make_inputs(w, "cuda")
    B, P = w.batch, w.gamma + 1
    table = ((torch.arange(B * P, device="cuda") % w.n).view(B, P)).to(torch.int32)
    off = torch.full((1,), 77, dtype=torch.int64, device="cuda")
    v = helpers.make_verifier(w)
    try:
        for proposer, opts in ((inputs["proposer"], {}), (table, {"bonus_model": w.n - 1}), (table, {"bonus_model": -1, "offset_device": off}),
                               (inputs["proposer"], {"row_base": 1 << 33, "flags": 1 if w.temperature > 0 else 0})):
            args = (inputs["logits"], inputs["drafts"], proposer, inputs["seed"] | 1 << 63, -5)
            short = v.run(*args, **opts)
            long = v.run(*args, stream=torch.cuda.current_stream(), **opts)
            torch.cuda.synchronize()
            assert list(short) == list(long)
            for k in short:
                assert short[k].dtype is long[k].dtype and short[k].shape == long[k].shape and short[k].is_contiguous(), k
                assert torch.equal(torch.nan_to_num(short[k].float(), nan=-7.0), torch.nan_to_num(long[k].float(), nan=-7.0)), k
        good = (inputs["logits"], inputs["drafts"], inputs["proposer"], 1, 0)

        def refused(error, *a, **kw):
            for stream in (None, torch.cuda.current_stream()):
                with pytest.raises(error):
                    v.run(*a, stream=stream, **kw)

        refused(ValueError, good[0].cpu(), *good[1:])
        refused(ValueError, good[0].double(), *good[1:])
        refused(ValueError, good[0].transpose(2, 3).contiguous().transpose(2, 3), *good[1:]) if P > 1 else None
        refused(ValueError, good[0], good[1], good[2].long(), 1, 0)
        refused(ValueError, good[0], good[1], torch.cat([good[2], good[2]]), 1, 0)
        refused(ValueError, *good, offset_device=off.int())
        refused(CosVerifyError, *good, flags=1 << 9)
        refused(CosVerifyError, *good, bonus_model=w.n)
        if w.gamma > 0:
            refused(ValueError, good[0], good[1].float(), *good[2:])
            refused(CosVerifyError, good[0], None, *good[2:])
    finally:
        v.close()
    with pytest.raises(CosVerifyError):        # a context that is closed
        v.run(*good)
