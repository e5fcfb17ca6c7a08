"""GPU parity at the full benchmark sizes (sampled rows) and on the edge cases of the method."""
import numpy as np
import pytest
import torch

import helpers
from paper_2502_01662_b200 import (COS_ROW_BAD_DRAFT, COS_ROW_NONFINITE, COS_ROW_Q_ZERO, COS_ROW_RESIDUAL_EMPTY,
                                   COS_RUN_ALL_RESIDUALS, COS_RUN_INPUTS_SETTLED, CosVerifier, CosVerifyError, synth)
from oracle import cos_oracle as orc

pytestmark = pytest.mark.gpu
C = synth.CONFIGS


@pytest.mark.parametrize("name,nrows", [("cfg1", 1), ("cfg2", 8), ("cfg3", 64), ("cfg4", 32), ("cfg5", 48), ("cfg5_greedy", 48)])
def test_full_size_workloads(name, nrows):
    """The launch configuration bench.py times (default cluster choice, full batch), compared with the
    oracle's C++ twin on every row (workloads 1 to 4) or on a seeded sample of rows (the 2.4 GB workload 5);
    a row's result does not depend on the other rows."""
    w = C[name]
    inputs = synth.make_inputs(w, "cuda")
    rows = sorted(np.random.default_rng(7).choice(w.batch, size=min(nrows, w.batch), replace=False).tolist())
    gpu = helpers.run_gpu(w, inputs, diag=True)
    ref = helpers.run_oracle(w, inputs, rows=rows, native=True)
    stats = helpers.check_parity(w, gpu, ref, rows=rows)
    assert stats["excused_accept"] + stats["excused_sample"] <= 2, stats
    # the rows are not degenerate: some rows reject, and sampling modes do not reject everything at 0
    acc = gpu["accept_count"]
    assert acc.min() >= 0 and acc.max() <= w.gamma
    assert np.all(gpu["out_tokens"][np.arange(w.batch), acc] >= 0)
    # second run with the same arguments is bit-identical (no dependence on scheduling)
    again = helpers.run_gpu(w, inputs, diag=True)
    for k in ("accept_count", "out_tokens", "row_status"):
        assert np.array_equal(gpu[k], again[k]), k
    # four calls queued without a pause on inputs that were complete long before (COS_RUN_INPUTS_SETTLED: a call's
    # streaming launch overlaps the end of the previous call's drawing launch): every one gives the same rows
    v = helpers.make_verifier(w)
    try:
        queued = [v.run(inputs["logits"], inputs["drafts"], inputs["proposer"], inputs["seed"], inputs["offset"],
                        flags=COS_RUN_INPUTS_SETTLED) for _ in range(4)]
        torch.cuda.synchronize()
        for outs in queued:
            for k in ("accept_count", "out_tokens", "row_status"):
                assert np.array_equal(gpu[k], outs[k].cpu().numpy()), k
    finally:
        v.close()
    del inputs
    torch.cuda.empty_cache()


def _small(cfg, **kw):
    return C[cfg].scaled(**kw)


@pytest.mark.parametrize("name,kw", [("cfg3", dict(batch=100, gamma=1)), ("cfg5", dict(batch=80, gamma=1)),
                                     ("cfg3", dict(batch=300, vocab=40000, gamma=1))])
def test_batches_that_do_not_fill_whole_waves(name, kw):
    """Between one and two drawing positions per multiprocessor (and more than two): the one-sweep drawing
    stage then splits a position over more blocks than the device holds at once; every row against the oracle
    on a sample, the residual mass it reports against the oracle's."""
    w = C[name].scaled(name=f"{name}_b{kw['batch']}", **kw)
    inputs = synth.make_inputs(w, "cuda")
    rows = sorted(np.random.default_rng(11).choice(w.batch, size=24, replace=False).tolist())
    gpu = helpers.run_gpu(w, inputs, diag=True)
    ref = helpers.run_oracle(w, inputs, rows=rows)
    stats = helpers.check_parity(w, gpu, ref, rows=rows)
    assert stats["excused_accept"] + stats["excused_sample"] <= 1, stats
    acc = gpu["accept_count"]
    assert np.all(gpu["out_tokens"][np.arange(w.batch), acc] >= 0)
    again = helpers.run_gpu(w, inputs, diag=True)
    for k in ("accept_count", "out_tokens", "row_status"):
        assert np.array_equal(gpu[k], again[k]), k
    del inputs
    torch.cuda.empty_cache()


def test_statistics_of_acceptance_match_eq7():
    """Mean accept flag against mean alpha_j = 1 - sum max(0, r - q) (Eq. 7) from the kernel's own S."""
    w = _small("cfg4", batch=32, vocab=12808, gamma=6, name="stat")
    inputs = synth.make_inputs(w, "cuda")
    gpu = helpers.run_gpu(w, inputs, diag=True, flags=COS_RUN_ALL_RESIDUALS)
    ref = helpers.run_oracle(w, inputs)
    S = gpu["diag"][:, : w.gamma, 3]
    assert np.all(np.isfinite(S))
    np.testing.assert_allclose(S, ref["S"][:, : w.gamma], rtol=1e-5, atol=1e-7)
    alpha = 1.0 - S
    assert np.all(alpha >= np.asarray(w.weights)[inputs["proposer"].cpu().numpy()][:, None] - 1e-6)   # Thm 3.2


@pytest.mark.parametrize("combine,weights,temperature,vocab,dtype", [
    (synth.COMBINE_PROB_ENSEMBLE, (0.16, 0.84), 0.3, 9559, "f32"), (synth.COMBINE_PROB_ENSEMBLE, (0.5, 0.3, 0.2), 0.3, 3920, "bf16"),
    (synth.COMBINE_PROB_ENSEMBLE, (0.3, 0.25, 0.2, 0.15, 0.1), 0.3, 4096, "bf16"), (synth.COMBINE_PROB_ENSEMBLE, (0.54, 0.46), 1.0, 9, "f16"),
    (synth.COMBINE_LOGIT_LINEAR, (1.5,), 0.3, 32, "f32"), (synth.COMBINE_LOGIT_LINEAR, (0.75, 0.75), 0.3, 18664, "f32"),
    (synth.COMBINE_LOGIT_LINEAR, (-0.5, 1.5), 0.3, 28128, "f16")])
def test_residual_masses_next_to_nothing(combine, weights, temperature, vocab, dtype):
    """Distributions of one token or two: r and q agree there to 1e-6 or so, and the residual mass is what is left of
    their difference, a few 1e-7.  To the tolerance of the parity check (1e-7 and 1e-5 of the mass)."""
    w = synth.Workload("nothing", len(weights), combine, weights, temperature, 24, 20, vocab, dtype, "gauss", sigma=6.0, rho=0.9,
                       proposer_rule="cycle")
    inputs = synth.make_inputs(w, "cuda")
    ref = helpers.run_oracle(w, inputs, native=True)
    S = ref["S"][:, : w.gamma]
    assert np.any((S > 2e-7) & (S < 1e-4))
    gpu = helpers.run_gpu(w, inputs, diag=True, flags=COS_RUN_ALL_RESIDUALS)
    got = gpu["diag"][:, : w.gamma, 3]
    assert np.all(np.abs(got - S) <= 1e-5 * np.maximum(S, 1e-3) + 1e-7), np.max(np.abs(got - S))


def test_row_base_and_partial_batches_and_strides():
    w = _small("cfg3", batch=6, vocab=4096, gamma=3, name="layout")
    inputs = synth.make_inputs(w, "cuda")
    full = helpers.run_gpu(w, inputs)
    # rows 2..5 as a shard: same numbers when row_base = 2; context sized for a larger batch
    v = helpers.make_verifier(w, max_batch=16)
    try:
        part = v.run(inputs["logits"][:, 2:], inputs["drafts"][2:].contiguous(), inputs["proposer"][2:].contiguous(),
                     inputs["seed"], inputs["offset"], row_base=2)
        torch.cuda.synchronize()
        for k in ("accept_count", "out_tokens", "row_status"):
            assert np.array_equal(part[k].cpu().numpy(), full[k][2:]), k
        # a padded layout (row pitch larger than V, still 16-byte aligned) and an unaligned one (scalar loads)
        for pad in (8, 3):
            big = torch.zeros((w.n, w.batch, w.gamma + 1, w.vocab + pad), dtype=inputs["logits"].dtype, device="cuda")
            big[..., : w.vocab] = inputs["logits"]
            view = big[..., : w.vocab]
            got = v.run(view, inputs["drafts"], inputs["proposer"], inputs["seed"], inputs["offset"])
            torch.cuda.synchronize()
            for k in ("accept_count", "out_tokens", "row_status"):
                assert np.array_equal(got[k].cpu().numpy(), full[k]), (pad, k)
    finally:
        v.close()


def test_host_pointer_entry_matches_device_entry():
    w = _small("cfg2", batch=5, vocab=8000, gamma=3, name="host")
    dev_in = synth.make_inputs(w, "cuda")
    want = helpers.run_gpu(w, dev_in, diag=True)
    v = helpers.make_verifier(w, host_staging=True)
    try:
        got = v.run_host(dev_in["logits"].cpu().contiguous().pin_memory(), dev_in["drafts"].cpu().pin_memory(),
                         dev_in["proposer"].cpu().pin_memory(), dev_in["seed"], dev_in["offset"], diag=True)
        for k in ("accept_count", "out_tokens", "row_status"):
            assert np.array_equal(got[k].numpy(), want[k]), k
        np.testing.assert_array_equal(got["diag"].numpy()[..., :3], want["diag"][..., :3])
    finally:
        v.close()


@pytest.mark.parametrize("n,form", [(1, 0), (2, 0), (3, 0), (5, 0), (1, 1), (2, 1), (3, 1), (1, 2), (2, 2), (3, 2)])
def test_host_pointer_entry_with_problems_in_the_rows(n, form):
    """Status bits that are added after a row's outputs were written (a residual without mass: identical models and a
    bad draft) reach host memory in every form of a run."""
    weights = {1: (1.0,), 2: (0.5, 0.5), 3: (0.5, 0.25, 0.25), 5: (0.5, 0.5, 0.0, 0.0, 0.0)}[n]   # (r cancels against q exactly)
    w = synth.Workload("host_rows", n, synth.COMBINE_PROB_ENSEMBLE, weights, 1.0, 6, 3, 8192, "bf16", "gauss", sigma=2.0, proposer_rule="zero")
    inputs = synth.make_inputs(w, "cuda")
    logits, drafts = inputs["logits"].clone(), inputs["drafts"].clone()
    logits[:, :4] = logits[0, :4].clone()
    drafts[0, 0] = w.vocab
    drafts[2, 1] = -1
    logits[n - 1, 3, 2, 7] = float("nan")
    v = helpers.make_verifier(w, host_staging=True)
    try:
        v.set_one_launch(form)
        want = {k: t.cpu() for k, t in v.run(logits, drafts, inputs["proposer"], inputs["seed"], 3, diag=True).items()}
        got = v.run_host(logits.cpu(), drafts.cpu(), inputs["proposer"].cpu(), inputs["seed"], 3, diag=True)
    finally:
        v.close()
    assert got["row_status"][0] == COS_ROW_BAD_DRAFT | COS_ROW_RESIDUAL_EMPTY
    assert got["row_status"][2] == COS_ROW_BAD_DRAFT | COS_ROW_RESIDUAL_EMPTY and got["accept_count"][2] == 1
    assert got["row_status"][3] == COS_ROW_NONFINITE and got["accept_count"][3] == 2
    for k in ("accept_count", "out_tokens", "row_status"):
        assert torch.equal(got[k], want[k]), k
    for k in ("diag", "bonus_prob"):
        assert torch.equal(torch.nan_to_num(got[k], nan=-7.0), torch.nan_to_num(want[k], nan=-7.0)), k


def test_data_dependent_problems_are_flagged_not_trapped():
    w = _small("cfg3", batch=6, vocab=2048, gamma=3, name="flags")
    inputs = synth.make_inputs(w, "cuda")
    logits = inputs["logits"].clone()
    drafts = inputs["drafts"].clone()
    logits[1, 0, 0, 77] = float("nan")          # row 0: NaN at position 0
    logits[0, 1, 1, 5] = float("inf")           # row 1: +inf at position 1
    logits[1, 2, 0, 9] = float("-inf")          # row 2: a token one model rules out (legal)
    drafts[3, 0] = w.vocab                      # row 3: draft outside the vocabulary
    drafts[4, 1] = -1                           # row 4: negative draft at position 1
    bad = dict(inputs, logits=logits, drafts=drafts)
    gpu = helpers.run_gpu(w, bad, diag=True)
    ref = helpers.run_oracle(w, bad)
    helpers.check_parity(w, gpu, ref, check_diag=False)
    assert gpu["row_status"][0] & COS_ROW_NONFINITE and gpu["accept_count"][0] == 0 and gpu["out_tokens"][0, 0] == -1
    assert gpu["row_status"][3] & COS_ROW_BAD_DRAFT and gpu["accept_count"][3] == 0
    assert gpu["row_status"][2] == ref["row_status"][2]


def test_identical_models_accept_everything_and_empty_residual_falls_back_to_r():
    w = _small("cfg3", batch=4, vocab=3000, gamma=2, name="same")
    inputs = synth.make_inputs(w, "cuda")
    logits = inputs["logits"].clone()
    logits[1] = logits[0]                        # r == q exactly
    drafts = inputs["drafts"].clone()
    drafts[2, 0] = w.vocab + 5                   # an invalid draft is rejected although the residual is empty
    same = dict(inputs, logits=logits, drafts=drafts)
    gpu = helpers.run_gpu(w, same, diag=True)
    ref = helpers.run_oracle(w, same)
    helpers.check_parity(w, gpu, ref, check_diag=False)
    assert np.all(gpu["accept_count"][[0, 1, 3]] == w.gamma)
    assert gpu["accept_count"][2] == 0
    assert gpu["row_status"][2] == (COS_ROW_BAD_DRAFT | COS_ROW_RESIDUAL_EMPTY)
    assert 0 <= gpu["out_tokens"][2, 0] < w.vocab


def test_greedy_ensemble_atoms_and_q_zero():
    w = synth.Workload("we_greedy", 3, 0, (0.5, 0.3, 0.2), 0.0, 8, 3, 5000, "f32", "gauss", sigma=2.0, rho=0.5,
                       proposer_rule="cycle")
    inputs = synth.make_inputs(w, "cuda")
    drafts = inputs["drafts"].clone()
    drafts[0, 0] = (int(drafts[0, 0]) + 1) % w.vocab     # not the proposer's argmax: q(draft) = 0
    mod = dict(inputs, drafts=drafts)
    gpu = helpers.run_gpu(w, mod, diag=True, dump_r=True)
    ref = helpers.run_oracle(w, mod, return_r=True)
    helpers.check_parity(w, gpu, ref, check_diag=False)
    helpers.check_combined_probabilities(w, gpu["r"], ref["r"])
    assert gpu["row_status"][0] & COS_ROW_Q_ZERO


@pytest.mark.parametrize("name", ["cfg5_greedy", "cfg2_greedy", "we_greedy"])
def test_greedy_with_non_finite_logits(name):
    """T = 0 (Sec. 4.1: one-hot distributions): a NaN or +inf among a position's logits, or a model without a
    finite maximum, leaves the argmax undefined: the position counts as rejected, no token, NONFINITE; -inf
    entries are legal while a finite maximum remains.  Rows against the oracle."""
    if name == "cfg5_greedy":
        w = C["cfg5_greedy"].scaled(batch=8, vocab=16000, gamma=3, name="greedy_nonfinite")
    elif name == "cfg2_greedy":
        w = synth.Workload("cd_greedy", 2, 1, (1.0, -0.5), 0.0, 8, 3, 9001, "bf16", "gauss", sigma=3.0, rho=0.7,
                           proposer_rule="cycle", mask_model=0, mask_alpha=0.1)
    else:
        w = synth.Workload("we_greedy_nf", 3, 0, (0.5, 0.3, 0.2), 0.0, 8, 3, 5000, "f32", "gauss", sigma=2.0, rho=0.5,
                           proposer_rule="cycle")
    inputs = synth.make_inputs(w, "cuda")
    logits = inputs["logits"].clone()
    logits[0, 0, 0, 17] = float("nan")            # row 0 stops at position 0
    logits[1, 1, 1, 3] = float("inf")             # row 1 at position 1 at the latest
    logits[w.n - 1, 2, 2, :] = float("-inf")      # a model with no finite maximum
    worst = int(torch.argmin(logits[0, 3, 0].float()))
    logits[0, 3, :, worst] = float("-inf")        # a ruled-out token that is nobody's argmax: harmless
    mod = dict(inputs, logits=logits)
    gpu = helpers.run_gpu(w, mod, diag=True)
    ref = helpers.run_oracle(w, mod)
    helpers.check_parity(w, gpu, ref, check_diag=False)
    assert gpu["accept_count"][0] == 0 and gpu["out_tokens"][0, 0] == -1 and gpu["row_status"][0] & COS_ROW_NONFINITE
    assert gpu["accept_count"][1] <= 1 and gpu["accept_count"][2] <= 2
    for b in (1, 2):
        if gpu["row_status"][b] & COS_ROW_NONFINITE:
            assert gpu["out_tokens"][b, gpu["accept_count"][b]] == -1
    assert not (gpu["row_status"][3] & COS_ROW_NONFINITE)


@pytest.mark.parametrize("name", ["cfg3", "cfg5", "cfg5_greedy"])
def test_proposer_index_outside_the_models_is_reported_per_row(name):
    """A proposer index outside [0, n) names no distribution q: every position of that row reports NONFINITE
    (so the row stops at position 0 without a token); the other rows are those of the oracle."""
    w = C[name].scaled(batch=6, vocab=8192, gamma=3, name=f"{name}_bad_proposer")
    inputs = synth.make_inputs(w, "cuda")
    prop = inputs["proposer"].clone()
    prop[1] = w.n
    prop[4] = -1
    gpu = helpers.run_gpu(w, dict(inputs, proposer=prop), diag=True)
    ref = helpers.run_oracle(w, inputs)
    good = [0, 2, 3, 5]
    helpers.check_parity(w, gpu, ref, rows=good)
    for b in (1, 4):
        assert gpu["accept_count"][b] == 0 and gpu["row_status"][b] & COS_ROW_NONFINITE
        assert np.all(gpu["out_tokens"][b] == -1)


def test_invalid_arguments_return_errors():
    w = _small("cfg3", batch=2, vocab=1024, gamma=2, name="args")
    inputs = synth.make_inputs(w, "cuda")
    v = helpers.make_verifier(w)
    try:
        with pytest.raises(CosVerifyError):        # batch larger than max_batch
            big = torch.zeros((w.n, 3, w.gamma + 1, w.vocab), dtype=inputs["logits"].dtype, device="cuda")
            v.run(big, torch.zeros((3, w.gamma), dtype=torch.int32, device="cuda"),
                  torch.zeros(3, dtype=torch.int32, device="cuda"), 1, 0)
        with pytest.raises(ValueError):            # wrong vocabulary
            v.run(inputs["logits"][..., :-8], inputs["drafts"], inputs["proposer"], 1, 0)
        with pytest.raises(CosVerifyError):        # host-pointer call without staging
            v.run_host(inputs["logits"].cpu(), inputs["drafts"].cpu(), inputs["proposer"].cpu(), 1, 0)
        with pytest.raises(CosVerifyError):        # bonus model outside [0, n)
            v.run(inputs["logits"], inputs["drafts"], inputs["proposer"], 1, 0, bonus_model=w.n)
        with pytest.raises(CosVerifyError):        # unknown flag bit
            v.run(inputs["logits"], inputs["drafts"], inputs["proposer"], 1, 0, flags=1 << 9)
        with pytest.raises(ValueError):            # a proposer table of the wrong shape
            v.run(inputs["logits"], inputs["drafts"], torch.zeros((2, w.gamma), dtype=torch.int32, device="cuda"), 1, 0)
        with pytest.raises(ValueError):            # the device-resident offset must be an int64 device tensor
            v.run(inputs["logits"], inputs["drafts"], inputs["proposer"], 1, 0,
                  offset_device=torch.zeros(1, dtype=torch.int32, device="cuda"))
        ok = v.run(inputs["logits"], inputs["drafts"], inputs["proposer"], 1, 0)   # the context still works
        torch.cuda.synchronize()
        assert ok["accept_count"].min() >= 0
    finally:
        v.close()


_E, _L = synth.COMBINE_PROB_ENSEMBLE, synth.COMBINE_LOGIT_LINEAR
_early = dict(proposer_rule="cycle", sigma=2.5, rho=0.8)
EARLY = [C["cfg3"],                                                # not taken: every position is read
         C["cfg3"].scaled(batch=256), C["cfg5"], C["cfg5_greedy"],
         synth.Workload("mask", 3, _L, (1.0, -0.25, -0.25), 1.0, 128, 8, 128256, "bf16", "gauss", mask_model=2, mask_alpha=0.1, **_early),
         synth.Workload("mask_greedy", 2, _L, (1.0, -0.5), 0.0, 256, 8, 90001, "f16", "gauss", mask_model=0, mask_alpha=0.1, **_early),
         synth.Workload("one", 1, _E, (1.0,), 1.0, 512, 8, 90001, "bf16", "gauss", **_early),
         synth.Workload("five", 5, _E, (0.3, 0.25, 0.2, 0.15, 0.1), 0.7, 180, 6, 40000, "f32", "gauss", **_early),
         synth.Workload("greedy", 4, _E, (0.4, 0.3, 0.2, 0.1), 0.0, 160, 15, 50001, "bf16", "gauss", **_early)]   # long rows


@pytest.mark.parametrize("w", EARLY, ids=lambda w: f"{w.name}-{w.batch}")
def test_early_exit_hint_gives_the_rows_of_the_full_run(w):
    """COS_RUN_EARLY_EXIT: positions behind a rejection their row has already reported may be left unread
    (Sec. 3.1 discards them).  The rows must be those of the full run; what is reported for positions up to
    and including the first rejection must be there; some later positions are in fact left unread."""
    from paper_2502_01662_b200 import COS_RUN_EARLY_EXIT
    inputs = synth.make_inputs(w, "cuda")
    v = helpers.make_verifier(w)
    try:
        full = helpers.run_gpu(w, inputs, verifier=v, diag=True)
        hint = helpers.run_gpu(w, inputs, verifier=v, diag=True, flags=COS_RUN_EARLY_EXIT)
        once_more = helpers.run_gpu(w, inputs, verifier=v, flags=COS_RUN_EARLY_EXIT)
        again = helpers.run_gpu(w, inputs, verifier=v, diag=True)        # the scratch was left clean
    finally:
        v.close()
    for k in ("accept_count", "out_tokens", "row_status"):
        assert np.array_equal(hint[k], full[k]), k
        assert np.array_equal(again[k], full[k]), k
        assert np.array_equal(once_more[k], full[k]), k
    assert np.array_equal(np.isnan(hint["bonus_prob"]), np.isnan(full["bonus_prob"]))
    # and a sample of the hinted run's rows against the oracle itself
    rows = sorted(np.random.default_rng(13).choice(w.batch, size=24, replace=False).tolist())
    ref = helpers.run_oracle(w, inputs, rows=rows, native=True)
    helpers.check_parity(w, hint, ref, rows=rows, check_diag=False)
    a = full["accept_count"]
    g = w.gamma
    unread = 0
    for b in range(w.batch):
        for j in range(g):
            if j <= a[b]:
                # the same sums in another order: an argument up to 64 rounds by 2^-19, which is 1.4e-6 of its exponential with
                # the exponential's own 2^-22; r and q are quotients of two such terms (3e-6), the ratio one of theirs
                tol = 0.0 if w.temperature == 0.0 else 6e-6
                np.testing.assert_allclose(hint["diag"][b, j, :3], full["diag"][b, j, :3], rtol=tol, atol=0, err_msg=f"{b}, {j}")
            elif np.isnan(hint["diag"][b, j, 1]) and not np.isnan(full["diag"][b, j, 1]):
                unread += 1
    # large runs go through their positions in many waves and leave some unread; in smaller ones nothing can be known in time, and
    # one model rejects nothing
    assert (unread > 0) == (w.batch > 64 and w.n > 1), unread
    del inputs
    torch.cuda.empty_cache()


@pytest.mark.parametrize("name,kw", [("cfg3", dict(batch=40, vocab=20008, gamma=8)), ("cfg5", dict(batch=6, vocab=50000, gamma=3)),
                                     ("cfg2", dict(batch=8, vocab=9001, gamma=5)), ("cfg5_greedy", dict(batch=6, vocab=50000, gamma=3))])
def test_a_run_can_be_captured_in_a_graph_and_replayed(name, kw):
    """The launches of a run depend on its arguments only, and the kernels leave the scratch as they found it:
    a captured run, replayed with the counter offset kept in device memory, gives what an ordinary run with
    that offset gives."""
    w = C[name].scaled(**kw)
    inputs = synth.make_inputs(w, "cuda")
    B, P = w.batch, w.gamma + 1
    v, ref_v = helpers.make_verifier(w), helpers.make_verifier(w)
    try:
        off = torch.zeros(1, dtype=torch.int64, device="cuda")
        outs = v._alloc_outs(B, P, w.vocab, torch.device("cuda"), True, False)
        args = (inputs["logits"], inputs["drafts"], inputs["proposer"], inputs["seed"], 0)
        v.run(*args, outs=outs, offset_device=off)          # an ordinary run first
        torch.cuda.synchronize()
        g = torch.cuda.CUDAGraph()
        with torch.cuda.graph(g):
            v.run(*args, outs=outs, offset_device=off)
        for k in (3, 4, 1 << 40):
            off.fill_(k)
            for t in outs.values():
                t.zero_()
            g.replay()
            torch.cuda.synchronize()
            want = ref_v.run(inputs["logits"], inputs["drafts"], inputs["proposer"], inputs["seed"], k, diag=True)
            torch.cuda.synchronize()
            for key in ("accept_count", "out_tokens", "row_status"):
                assert torch.equal(outs[key], want[key]), (k, key)
            assert torch.equal(torch.nan_to_num(outs["diag"], nan=-7.0), torch.nan_to_num(want["diag"], nan=-7.0))
            assert torch.equal(torch.nan_to_num(outs["bonus_prob"], nan=-7.0), torch.nan_to_num(want["bonus_prob"], nan=-7.0))
        # an ordinary run after the replays still works on the same context
        again = v.run(inputs["logits"], inputs["drafts"], inputs["proposer"], inputs["seed"], 3)
        want = ref_v.run(inputs["logits"], inputs["drafts"], inputs["proposer"], inputs["seed"], 3)
        torch.cuda.synchronize()
        assert torch.equal(again["out_tokens"], want["out_tokens"])
    finally:
        v.close()
        ref_v.close()


@pytest.mark.parametrize("name,kw", [("cfg3", dict(batch=40, vocab=20008, gamma=8)), ("cfg4", dict(batch=30, vocab=12808, gamma=5)),
                                     ("cfg5", dict(batch=36, vocab=16000, gamma=4)), ("cfg5_greedy", dict(batch=36, vocab=16000, gamma=4)),
                                     ("cfg2", dict(batch=8, vocab=9001, gamma=5))])
@pytest.mark.parametrize("settled", [False, True])
def test_calls_queued_back_to_back_give_what_isolated_calls_give(name, kw, settled):
    """Every launch of a run may take its places on the device while the kernel before it in the stream drains,
    and waits for that kernel before it reads or writes anything.  Sixteen calls queued without a pause, on
    logits that a kernel queued just before each call writes, into output buffers of their own, must give what
    the same calls give one by one with a synchronisation in between.  With COS_RUN_INPUTS_SETTLED (inputs that
    were complete long before: no producer kernel) the streaming launch reads them while the previous call's
    drawing launch drains, and the results are the same again."""
    w = C[name].scaled(**kw)
    inputs = synth.make_inputs(w, "cuda")
    B, P = w.batch, w.gamma + 1
    v = helpers.make_verifier(w)
    try:
        variants = [torch.roll(inputs["logits"], shifts=7 * k, dims=-1) for k in range(4)]
        drafts = [((inputs["drafts"] + 7 * k) % w.vocab).to(torch.int32) for k in range(4)]   # rolled with the logits
        live = torch.empty_like(inputs["logits"])
        queued = []
        for k in range(16):
            outs = v._alloc_outs(B, P, w.vocab, torch.device("cuda"), True, False)
            if settled:
                v.run(variants[k % 4], drafts[k % 4], inputs["proposer"], inputs["seed"], 100 + k, outs=outs,
                      flags=COS_RUN_INPUTS_SETTLED)
            else:
                live.copy_(variants[k % 4])                  # a kernel in the same stream produces the logits
                v.run(live, drafts[k % 4], inputs["proposer"], inputs["seed"], 100 + k, outs=outs)
            queued.append(outs)
        torch.cuda.synchronize()
        for k in range(16):
            want = v.run(variants[k % 4], drafts[k % 4], inputs["proposer"], inputs["seed"], 100 + k, diag=True)
            torch.cuda.synchronize()
            for key in ("accept_count", "out_tokens", "row_status"):
                assert torch.equal(queued[k][key], want[key]), (k, key)
            assert torch.equal(torch.nan_to_num(queued[k]["diag"], nan=-7.0), torch.nan_to_num(want["diag"], nan=-7.0)), k
        # and one of them against the oracle
        ref = helpers.run_oracle(w, dict(inputs, logits=variants[1], drafts=drafts[1], offset=101), native=True)
        got = {key: t.cpu().numpy() for key, t in queued[1].items()}
        helpers.check_parity(w, got, ref)
    finally:
        v.close()


@pytest.mark.parametrize("n", [2, 5])       # decisions in the drawing launch, and in a launch of their own
def test_offset_written_just_before_a_call_on_settled_inputs_is_seen(n):
    """COS_RUN_INPUTS_SETTLED promises logits, drafts and proposer, not the offset in device memory: a kernel that
    advances the offset, queued directly before each call, is complete before the call reads it."""
    weights = (0.6, 0.4) if n == 2 else (0.3, 0.25, 0.2, 0.15, 0.1)
    w = synth.Workload("settled_offset", n, synth.COMBINE_PROB_ENSEMBLE, weights, 1.0, 40, 4, 20008, "bf16", "gauss", sigma=2.5, rho=0.8,
                       proposer_rule="cycle")
    inputs = synth.make_inputs(w, "cuda")
    args = (inputs["logits"], inputs["drafts"], inputs["proposer"], inputs["seed"])
    off = torch.zeros(1, dtype=torch.int64, device="cuda")
    step = torch.ones(1 << 22, dtype=torch.int64, device="cuda")
    v = helpers.make_verifier(w)
    try:
        torch.cuda.synchronize()
        queued = []
        for _ in range(24):
            off += step.max()            # two kernels, the first of them longer than the tail of the call before
            queued.append(v.run(*args, 0, offset_device=off, flags=COS_RUN_INPUTS_SETTLED))
        torch.cuda.synchronize()
        for k, outs in enumerate(queued):
            want = v.run(*args, k + 1)
            for key in ("accept_count", "out_tokens", "row_status"):
                assert torch.equal(outs[key], want[key]), (k, key)
    finally:
        v.close()


@pytest.mark.parametrize("combine,weights,mask_model", [(synth.COMBINE_PROB_ENSEMBLE, (0.6, 0.4), -1), (synth.COMBINE_LOGIT_LINEAR, (1.5, -0.5), -1),
                                                        (synth.COMBINE_LOGIT_LINEAR, (1.0, -0.5), 0)])
def test_positions_left_unread_report_no_log_sum_exp(combine, weights, mask_model):
    """COS_RUN_EARLY_EXIT with `lse`: NaN at a position that was left unread, never what an earlier call left behind."""
    from paper_2502_01662_b200 import COS_RUN_EARLY_EXIT
    w = synth.Workload("unread", 2, combine, weights, 1.0, 192, 6, 143360, "bf16", "gauss", sigma=2.5, rho=0.3, proposer_rule="cycle",
                       mask_model=mask_model, mask_alpha=0.1 if mask_model >= 0 else 1.0)     # large: the hint is taken
    inputs = synth.make_inputs(w, "cuda")
    v = helpers.make_verifier(w)
    try:
        full = helpers.run_gpu(w, inputs, verifier=v, diag=True, lse=True)
        other = dict(inputs, logits=inputs["logits"] * 0.5)
        helpers.run_gpu(w, other, verifier=v, diag=True, lse=True)          # leaves other statistics behind
        hint = helpers.run_gpu(w, inputs, verifier=v, diag=True, lse=True, flags=COS_RUN_EARLY_EXIT)
    finally:
        v.close()
    for k in ("accept_count", "out_tokens", "row_status"):
        assert np.array_equal(hint[k], full[k]), k
    drafts = w.gamma
    unread = np.isnan(hint["diag"][:, :drafts, 1]) & ~np.isnan(full["diag"][:, :drafts, 1])
    assert unread.any()
    assert np.all(np.isnan(hint["lse"][:, :drafts][unread]))
    assert np.allclose(hint["lse"][:, :drafts][~unread], full["lse"][:, :drafts][~unread], rtol=1e-6, atol=0)
    del inputs, other
    torch.cuda.empty_cache()


@pytest.mark.parametrize("n,combine,weights", [(4, synth.COMBINE_PROB_ENSEMBLE, (0.41, 0.435, 0.042, 0.113)), (2, synth.COMBINE_LOGIT_LINEAR, (1.5, -0.25)),
                                               (2, synth.COMBINE_PROB_ENSEMBLE, (0.6, 0.4))])
def test_tokens_from_residuals_next_to_nothing(n, combine, weights):
    """A token that has to be drawn (bad drafts) from a residual of a few 1e-7, with and without the masses of all positions."""
    w = synth.Workload("scraps", n, combine, weights, 0.3, 64, 3, 3000, "f16", "gauss", sigma=6.0, rho=0.9, proposer_rule="cycle")
    inputs = synth.make_inputs(w, "cuda")
    drafts = inputs["drafts"].clone()
    drafts[:, 0] = w.vocab
    inputs = dict(inputs, drafts=drafts)
    ref = helpers.run_oracle(w, inputs, native=True)
    assert np.any((ref["S"][:, 0] > 1e-7) & (ref["S"][:, 0] < 1e-3))
    for flags in (0, COS_RUN_ALL_RESIDUALS):
        helpers.check_parity(w, helpers.run_gpu(w, inputs, diag=True, flags=flags), ref)
