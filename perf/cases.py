"""The verification calls whose speed matters, as a user's program makes them.

A case is one pass through a public entry point (`CosVerifier.run`, `CosVerifier.run_host` or `run_static`) on
seeded inputs of `paper_2502_01662_b200.synth`: logits of n models for every row and each of gamma + 1 positions,
draft tokens drawn from the proposer's softmax, and the proposer indices.  The fields of a case:

  entry        "run" (device tensors), "host" (pinned host tensors, copies included) or "static" (no context)
  combine      "ensemble" (weighted mixture of softmaxes) or "logit" (linear combination of logits)
  n, batch, gamma, vocab, dtype, temperature (0 = greedy)
  mask_alpha   logit level: plausibility threshold against model 0 (0 = no mask)
  alternate    Algorithm 2: a proposer per draft, the bonus token from a named model, and its probability
  diagnostics  acceptance diagnostics for choosing gamma: ratios, residual masses and log-sum-exps at every position
  generator    "gauss" (flat) or "gumbel_zipf" (peaked, with a common rank bias)
"""
import math

import numpy as np
import torch

from paper_2502_01662_b200 import synth
from paper_2502_01662_b200.binding import COS_RUN_ALL_RESIDUALS, CosVerifier, run_static

ENSEMBLE_WEIGHTS = {1: (1.0,), 2: (0.5, 0.5), 3: (0.5, 0.3, 0.2), 4: (0.4, 0.3, 0.2, 0.1), 5: (0.3, 0.25, 0.2, 0.15, 0.1)}
LOGIT_WEIGHTS = {2: (1.5, -0.5), 3: (1.0, 0.5, -0.5)}
CONTRAST_WEIGHTS = {2: (1.0, -0.5), 3: (1.0, -0.25, -0.25)}
MOST_BYTES = 2 * 256 * 9 * 256000 * 2   # logits of the largest listed case


def _case(name, **kw):
    c = dict(name=name, entry="run", combine="ensemble", n=2, batch=1, gamma=4, vocab=32000, dtype="bf16", temperature=1.0,
             mask_alpha=0.0, alternate=False, diagnostics=False, generator="gauss")
    c.update(kw)
    return c


def listed():
    return [
        # one sequence at a time, small vocabulary: interactive decoding, all latency
        _case("row_32k_f32", dtype="f32"),
        # one sequence at a time at a large vocabulary, the paper's gamma
        _case("row_152k_bf16", gamma=5, vocab=151936, temperature=0.7, generator="gumbel_zipf"),
        # a scheduler that keeps its logits on the host (gpu_verify of the schedulers): copies are part of the call
        _case("host_row_32k_f32", entry="host", gamma=5, dtype="f32", alternate=True),
        # contrastive decoding with the plausibility mask, a small serving batch
        _case("contrast_8x32k", combine="logit", batch=8, gamma=5, mask_alpha=0.1),
        # an engine that has given the whole device to its own pool: the entry point that allocates nothing
        _case("static_32x32k", entry="static", batch=32, gamma=5, temperature=0.7, generator="gumbel_zipf"),
        # three models taking turns as proposers (Algorithm 2), a vocabulary that is no multiple of anything
        _case("alternate3_16x50k_odd", n=3, batch=16, gamma=5, vocab=50001, alternate=True),
        # greedy decoding of an ensemble, half precision
        _case("greedy_16x128k_f16", batch=16, gamma=5, vocab=128256, dtype="f16", temperature=0.0),
        # choosing gamma offline: the residual mass at every draft position
        _case("diagnose_16x128k", batch=16, gamma=8, vocab=128256, diagnostics=True),
        # ordinary serving batches: two and four models
        _case("ensemble2_64x152k", batch=64, gamma=8, vocab=151936, temperature=0.7, generator="gumbel_zipf"),
        _case("ensemble4_32x128k", n=4, batch=32, gamma=6, vocab=128256),
        # the largest batches: logit interpolation of an aligned and a base model, sampled and greedy
        _case("interp_256x256k", combine="logit", batch=256, gamma=8, vocab=256000, generator="gumbel_zipf"),
        _case("interp_greedy_256x256k", combine="logit", batch=256, gamma=8, vocab=256000, temperature=0.0,
              generator="gumbel_zipf"),
    ]


def _between(rng, lo, hi):
    """Uniform over the logarithm."""
    return int(round(math.exp(rng.uniform(math.log(lo), math.log(hi)))))


def draw(rng):
    entry = rng.choice(["run"] * 8 + ["host", "static"])
    combine = rng.choice(["ensemble", "ensemble", "ensemble", "logit", "logit"])
    n = rng.choice([2, 2, 2, 3, 4, 5]) if combine == "ensemble" else rng.choice([2, 2, 2, 3])
    temperature = rng.choice([0.0, 0.7, 1.0, 1.0])
    gamma = rng.randint(2, 8)
    vocab = _between(rng, 32000, 256000)
    if rng.random() < 0.75:
        vocab -= vocab % 64                       # padded, as most are
    else:
        vocab |= 1
    dtype = rng.choice(["bf16", "bf16", "f16", "f32"])
    batch = _between(rng, 1, 4 if entry == "host" else 256)
    room = MOST_BYTES if entry != "host" else MOST_BYTES // 64
    per_row = n * (gamma + 1) * vocab * (4 if dtype == "f32" else 2)
    batch = max(1, min(batch, room // per_row))
    alternate = rng.random() < 0.2
    diagnostics = entry == "run" and temperature > 0.0 and rng.random() < 0.12
    return dict(entry=entry, combine=combine, n=n, batch=batch, gamma=gamma, vocab=vocab, dtype=dtype, temperature=temperature,
                mask_alpha=0.1 if combine == "logit" and rng.random() < 0.5 else 0.0, alternate=alternate,
                diagnostics=diagnostics, generator=rng.choice(["gauss", "gumbel_zipf"]))


def _weights(case):
    if case["combine"] == "ensemble":
        return ENSEMBLE_WEIGHTS[case["n"]]
    return (CONTRAST_WEIGHTS if case["mask_alpha"] > 0.0 else LOGIT_WEIGHTS)[case["n"]]


def prepare(case, seed):
    n, batch, gamma = case["n"], case["batch"], case["gamma"]
    combine = synth.COMBINE_PROB_ENSEMBLE if case["combine"] == "ensemble" else synth.COMBINE_LOGIT_LINEAR
    mask_model = 0 if case["mask_alpha"] > 0.0 else -1
    w = synth.Workload("case", n, combine, _weights(case), case["temperature"], batch, gamma, case["vocab"], case["dtype"],
                       case["generator"], sigma=2.5, rho=0.85, proposer_rule="cycle", mask_model=mask_model,
                       mask_alpha=case["mask_alpha"] or 1.0, seed=20250201 + 101 * seed, verify_seed=0x5EEDC05C05 + seed)
    logits = synth.make_logits(w, "cuda")
    bonus_model = None
    if case["alternate"]:
        rng = np.random.Generator(np.random.Philox(key=w.seed + 29))
        proposer = rng.integers(0, n, size=(batch, gamma + 1), dtype=np.int32)
        of_model = np.stack([synth.make_drafts(w, logits, np.full(batch, i, np.int32)) for i in range(n)])
        drafts = np.take_along_axis(of_model, proposer[None, :, :gamma].astype(np.int64), axis=0)[0]
        bonus_model = int(rng.integers(0, n))
    else:
        proposer = synth.make_proposer(w)
        drafts = synth.make_drafts(w, logits, proposer)
    on_host = case["entry"] == "host"

    def put(a):
        t = torch.from_numpy(np.ascontiguousarray(a))
        return t.pin_memory() if on_host else t.cuda()

    state = {"entry": case["entry"], "drafts": put(drafts), "proposer": put(proposer), "seed": w.verify_seed,
             "offset": 1000 + seed, "bonus_model": bonus_model,
             "flags": COS_RUN_ALL_RESIDUALS if case["diagnostics"] else 0, "diagnostics": bool(case["diagnostics"])}
    if on_host:
        state["logits"] = torch.empty(logits.shape, dtype=logits.dtype, pin_memory=True)
        state["logits"].copy_(logits)
    else:
        state["logits"] = logits
    if case["entry"] == "static":
        state["config"] = dict(n=n, combine=combine, weights=_weights(case), temperature=case["temperature"], gamma=gamma,
                               vocab=case["vocab"], mask_model=mask_model, mask_alpha=w.mask_alpha)
        state["outs"] = {"accept_count": torch.empty(batch, dtype=torch.int32, device="cuda"),
                         "out_tokens": torch.empty((batch, gamma + 1), dtype=torch.int32, device="cuda"),
                         "row_status": torch.empty(batch, dtype=torch.int32, device="cuda"),
                         "bonus_prob": torch.empty(batch, dtype=torch.float32, device="cuda")}
    else:
        state["verifier"] = CosVerifier(n, combine, _weights(case), case["temperature"], gamma, case["vocab"], batch,
                                        w.torch_dtype, mask_model=mask_model, mask_alpha=w.mask_alpha, host_staging=on_host)
    return state


def run(state):
    s = state
    if s["entry"] == "static":
        return run_static(logits=s["logits"], drafts=s["drafts"], proposer=s["proposer"], seed=s["seed"], offset=s["offset"],
                          outs=s["outs"], bonus_model=s["bonus_model"], **s["config"])
    if s["entry"] == "host":
        return s["verifier"].run_host(s["logits"], s["drafts"], s["proposer"], s["seed"], s["offset"],
                                      bonus_model=s["bonus_model"])
    return s["verifier"].run(s["logits"], s["drafts"], s["proposer"], s["seed"], s["offset"], flags=s["flags"],
                             diag=s["diagnostics"], lse=s["diagnostics"], bonus_model=s["bonus_model"])


def work(case):
    """Every logit read once; a scale, an exponential and a sum for each."""
    rows, positions = case["batch"], case["batch"] * (case["gamma"] + 1)
    logits = case["n"] * positions * case["vocab"]
    small = 4 * (2 * positions + 5 * rows) + (4 * positions * (4 + case["n"]) if case["diagnostics"] else 0)
    return {"bytes": logits * (4 if case["dtype"] == "f32" else 2) + small, "flops": 4 * logits}


def tolerance(case):
    """Whole numbers differ only where a uniform falls into the band that separates two correct roundings (about 1e-6
    wide), which costs a row at most; probabilities and masses are sums of 32-bit exponentials, stored as 32-bit numbers
    (against the same in 64 bits they are off by 2e-7 at most)."""
    return {"rel": 1e-6, "max": 5e-6, "differ": 0.005}
