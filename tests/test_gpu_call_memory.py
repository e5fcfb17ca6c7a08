"""No device memory for the outputs of a call: both ways of CosVerifier.run raise what torch raises."""
import pytest
import torch

import helpers
from paper_2502_01662_b200 import synth

pytestmark = pytest.mark.gpu


def test_no_memory_for_the_outputs():
    w = synth.CONFIGS["cfg1"].scaled(batch=2, vocab=4096, gamma=3)
    inputs = synth.make_inputs(w, "cuda")
    args = (inputs["logits"], inputs["drafts"], inputs["proposer"], inputs["seed"], 0)
    v = helpers.make_verifier(w)
    filler = []
    try:
        v.run(*args)
        torch.cuda.synchronize()
        torch.cuda.empty_cache()
        torch.cuda.set_per_process_memory_fraction(0.0)      # (of this process and torch's allocator alone: no new segment)
        with pytest.raises(torch.OutOfMemoryError):
            while len(filler) < 1 << 16:                     # what is left of the segments there are, in the smallest pieces
                filler.append(torch.empty(1, dtype=torch.uint8, device="cuda"))
        for stream in (None, torch.cuda.current_stream()):
            with pytest.raises(torch.OutOfMemoryError):
                v.run(*args, stream=stream)
    finally:
        torch.cuda.set_per_process_memory_fraction(1.0)
        filler.clear()
        v.run(*args)
        torch.cuda.synchronize()
        v.close()
