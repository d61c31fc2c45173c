"""GPU parity of the fused target LM head + acceptance (sf_verify_lm_head_accept)
against the fp64 oracle.

The hidden states and LM-head weights are small integers (weights scaled by a
power of two): every fp32 partial sum is exact, so the GPU's logits must equal
the oracle's LM-head logits bit for bit, and the accepted lengths and tokens
are then compared exactly with the oracle's rule on those logits (excluding
decisions within 1e-6 of a threshold or CDF boundary, as for sf_accept).
The draft distribution q is the softmax of the target logits plus noise.
"""
import numpy as np
import pytest
import torch
from scipy.special import softmax

from paper_2505_12728_gb300 import specflash_verify as sfv
from paper_2505_12728_gb300.workloads import (AcceptInputs, HIDDEN_SIZES, WORKLOADS, f32_to_bf16_bits,
                                              make_draft_tail_case, temperatures)
from tests.gpu_helpers import bf16_tensor, compare_accept, oracle_accept, require_gpu, run_accept

pytestmark = pytest.mark.gpu


@pytest.fixture(scope="module", autouse=True)
def _gpu():
    require_gpu()


def make_case(oracle_mod, B, k, V, d, seed, mode="sampling", sharpness=1.0):
    # exact small-integer hidden states [B*(k+1)][d] and weights [V][d]
    dt = make_draft_tail_case(B * (k + 1), d, V, seed=seed, exact=True)
    logits = oracle_mod.lm_head_logits(dt.hidden, dt.weight).reshape(B, k + 1, V)
    rng = np.random.default_rng([7, *np.atleast_1d(seed)])
    q = softmax(sharpness * logits[:, :k] + rng.standard_normal((B, k, V)), axis=-1).astype(np.float32)
    temp = temperatures(mode, B)
    tokens = np.empty((B, k), np.int32)
    for b in range(B):
        for i in range(k):
            if temp[b] > 0:
                c = np.cumsum(q[b, i].astype(np.float64))
                tokens[b, i] = min(int(np.searchsorted(c, rng.random() * c[-1], side="right")), V - 1)
            else:
                tokens[b, i] = int(np.argmax(q[b, i]))
    u = rng.random((B, k + 1), dtype=np.float32)
    inp = AcceptInputs(target_logits=logits.astype(np.float32), draft_probs=q, draft_tokens=tokens,
                       uniforms=u, temperature=temp)
    return dt.hidden.reshape(B, k + 1, d), dt.weight, inp, logits


def run_fused(hidden, weight, inp):
    B, k1, d = hidden.shape
    ws = sfv.new_workspace(sfv.verify_lm_head_accept_workspace_size(B, k1 - 1, weight.shape[0]))
    logits, n, toks, ratio = sfv.verify_lm_head_accept(
        bf16_tensor(hidden), bf16_tensor(weight), torch.from_numpy(inp.draft_probs).cuda(),
        torch.from_numpy(inp.draft_tokens).cuda(), torch.from_numpy(inp.uniforms).cuda(),
        torch.from_numpy(inp.temperature).cuda(), workspace=ws)
    torch.cuda.synchronize()
    assert sfv.read_device_status(ws) == 0
    return logits.cpu().numpy(), n.cpu().numpy(), toks.cpu().numpy(), ratio.cpu().numpy()


@pytest.mark.parametrize("B,k,V,d,mode", [
    (1, 5, 32000, 4096, "sampling"),    # image7b acceptance with LLaVA's LM head
    (1, 5, 32000, 4096, "greedy"),
    (8, 6, 6000, 512, "alternate"),
    (4, 8, 3001, 256, "sampling"),      # ragged vocabulary
    (16, 8, 2000, 128, "alternate"),    # 144 rows
    (2, 1, 50, 64, "sampling"),
])
def test_fused_acceptance_matches_oracle(oracle_mod, B, k, V, d, mode):
    hidden, weight, inp, ref_logits = make_case(oracle_mod, B, k, V, d, seed=[B, k, V], mode=mode)
    logits, n, toks, ratio = run_fused(hidden, weight, inp)
    assert np.array_equal(logits.astype(np.float64), ref_logits)
    excluded = compare_accept(oracle_accept(oracle_mod, inp), n, toks, ratio)
    assert excluded <= max(1, B // 10)


def test_fused_agrees_with_unfused_acceptance(oracle_mod):
    hidden, weight, inp, _ = make_case(oracle_mod, 8, 4, 5000, 256, seed=11, mode="alternate",
                                       sharpness=1.5)
    _, n, toks, _ = run_fused(hidden, weight, inp)
    n2, toks2, _ = run_accept(inp)
    assert np.array_equal(n, n2) and np.array_equal(toks, toks2)


def test_fused_qwen_vocabulary(oracle_mod):
    # QwenVL-sized head (152064 x 3584) for 4 sequences with k = 8
    V, d = 152064, HIDDEN_SIZES[152064]
    hidden, weight, inp, ref_logits = make_case(oracle_mod, 4, 8, V, d, seed=5, mode="sampling",
                                                sharpness=1.5)
    logits, n, toks, ratio = run_fused(hidden, weight, inp)
    assert np.array_equal(logits.astype(np.float64), ref_logits)
    compare_accept(oracle_accept(oracle_mod, inp), n, toks, ratio)


def test_fused_invalid_arguments():
    lib = sfv.load_library()
    assert lib.sf_verify_lm_head_accept_workspace_size(32, 8, 1000) == 0  # 288 rows
    assert lib.sf_verify_lm_head_accept_workspace_size(1, 0, 1000) == 0
    assert lib.sf_verify_lm_head_accept_workspace_size(1, 5, 32000) > 0


@pytest.mark.parametrize("B,k,V", [
    (1, 1, 128),       # two rows, one record each
    (3, 15, 4000),     # 16 rows, 32 records: one per lane
    (2, 16, 4200),     # 17 rows, the most; 33 records
    (15, 16, 20000),   # 255 rows, a record of every SM
])
def test_decisions_with_a_warp_for_each_row(oracle_mod, B, k, V):
    hidden, weight, inp, ref_logits = make_case(oracle_mod, B, k, V, 64, seed=[B, k, V], mode="alternate")
    logits, n, toks, ratio = run_fused(hidden, weight, inp)
    assert np.array_equal(logits.astype(np.float64), ref_logits)
    assert compare_accept(oracle_accept(oracle_mod, inp), n, toks, ratio) == 0


@pytest.mark.parametrize("B,k,V", [
    (13, 5, 32000),    # draft rows of 8.32 MB: one cluster launch after the projection
    (14, 5, 32000),    # 8.96 MB: statistics, decisions and draw
    (1, 8, 32768),     # more than five drafts of few sequences: the same
    (1, 5, 32768),     # the longest rows of a cluster
    (1, 5, 32772),     # one step beyond
    (1, 8, 32772),
    (1, 5, 12288),     # five drafts of one sequence: statistics up to here
    (1, 5, 12292),     # and a cluster launch from here
    (2, 5, 12292),
    (2, 3, 5000),      # few rows: cluster
    (3, 3, 5000),      # statistics
    (4, 2, 8192),      # cluster
    (4, 2, 8196),      # statistics
    (11, 6, 8000),     # statistics
    (12, 6, 8000),     # many sequences: cluster
    (12, 9, 8000),     # statistics: nine drafts
    (17, 2, 16384),    # cluster
    (17, 1, 16388),    # statistics
    (8, 8, 32000),     # statistics
    (12, 8, 21840),    # draft rows of just under 8 MiB
    (2, 16, 32000),    # rows and draft rows don't fit shared memory together
    (3, 4, 5001),      # not 16-byte aligned
    (5, 1, 16),
])
def test_routes_behind_the_projection_agree(oracle_mod, B, k, V):
    mode = "alternate" if B > 1 else "sampling"  # (alternating starts with a greedy sequence)
    hidden, weight, inp, ref_logits = make_case(oracle_mod, B, k, V, 64, seed=[B, k, V, 1], mode=mode)
    ref = oracle_accept(oracle_mod, inp)
    for _ in range(2):
        logits, n, toks, ratio = run_fused(hidden, weight, inp)
        assert np.array_equal(logits.astype(np.float64), ref_logits)
        assert compare_accept(ref, n, toks, ratio) == 0  # no sequence is excused by its margin


@pytest.mark.parametrize("V,d", [(152064, 3584), (32000, 4096)])
def test_lm_head_then_accept_on_one_stream(oracle_mod, V, d):
    # The target logits written by sf_lm_head are read by sf_accept launched
    # right after it on the same stream, with no synchronisation between:
    # the projection lets its successor start early, so the acceptance must
    # wait for it before reading any input.  The logits buffer is filled with
    # NaN before each projection, so an early read would show.
    hidden, weight, inp, ref_logits = make_case(oracle_mod, 4, 8, V, d, seed=[21, V], mode="alternate",
                                                sharpness=1.5)
    B, k1, _ = hidden.shape
    h = bf16_tensor(hidden.reshape(B * k1, d))
    w = bf16_tensor(weight)
    dev = {key: torch.from_numpy(getattr(inp, key)).cuda()
           for key in ("draft_probs", "draft_tokens", "uniforms", "temperature")}
    logits = torch.empty((B * k1, V), dtype=torch.float32, device="cuda")
    ws_lm = sfv.new_workspace(sfv.draft_tail_workspace_size(B * k1, V))
    ws_acc = sfv.new_workspace(sfv.accept_workspace_size(B, k1 - 1, V))
    ref = oracle_accept(oracle_mod, inp)
    for _ in range(3):
        logits.fill_(float("nan"))
        sfv.lm_head(h, w, logits=logits, workspace=ws_lm)
        n, toks, ratio = sfv.accept(logits.view(B, k1, V), dev["draft_probs"], dev["draft_tokens"],
                                    dev["uniforms"], dev["temperature"], workspace=ws_acc)
        torch.cuda.synchronize()
        assert np.array_equal(logits.cpu().numpy().reshape(B, k1, V).astype(np.float64), ref_logits)
        assert sfv.read_device_status(ws_acc) == 0
        compare_accept(ref, n.cpu().numpy(), toks.cpu().numpy(), ratio.cpu().numpy())


def test_greedy_calls_back_to_back_on_one_workspace(oracle_mod):
    # the next call's projection overwrites the logits and statistics that the
    # decisions of this one read
    B, k, V, d = 2, 3, 40000, 64
    cases = [make_case(oracle_mod, B, k, V, d, seed=[V, i], mode="greedy") for i in range(6)]
    devs = [(bf16_tensor(h), bf16_tensor(w), *(torch.from_numpy(a).cuda() for a in (
        inp.draft_probs, inp.draft_tokens, inp.uniforms, inp.temperature))) for h, w, inp, _ in cases]
    ws = sfv.new_workspace(sfv.verify_lm_head_accept_workspace_size(B, k, V))
    logits = torch.empty((B, k + 1, V), device="cuda")  # shared, as the workspace
    for _ in range(20):
        outs = [sfv.verify_lm_head_accept(*dev, logits=logits, workspace=ws)[1:] for dev in devs]
    torch.cuda.synchronize()
    assert sfv.read_device_status(ws) == 0
    for (_, _, inp, _), out in zip(cases, outs):
        assert compare_accept(oracle_accept(oracle_mod, inp), *(t.cpu().numpy() for t in out)) == 0


@pytest.mark.parametrize("V", [8000, 32000, 40000])
def test_row_sums_carry_the_scaled_difference_in_float_float(V):
    """A token at logit 0 in every 2000 (the slice of a CTA of the cluster) and
    the others at -a, with a / tau a little above 8 and its fp32 rounding error as
    large as it gets, of one sign in a row: the row sum must not show it.

    The bound: p(0) = 1 / S (and q = 1), of which the share s comes from the terms
    at -a, shows s times the error of one term, expf's (one unit in the last
    place at most, 2^-23) and the product's with 1 + lo (2^-24), and the quotient's
    rounding (2^-24): 1.25e-7 at s = 0.36.  An fp32 a / tau is off by 2^-21, which
    alone is 1.7e-7 of S."""
    rng = np.random.default_rng(V)
    B, k, d = 16, 1, 8
    hidden, weight = np.zeros((B, k + 1, d), np.float32), np.zeros((V, d), np.float32)
    weight[:, 0] = -1.0
    weight[::2000, 0] = 0.0
    a, tau = np.empty(B), np.empty(B, np.float32)
    for b in range(B):  # a: eight bits (exact in bf16); tau: the worst of many for it
        a[b] = hidden[b, :, 0] = rng.integers(128, 256) / 16.0
        t = (a[b] / (8.02 + 0.2 * rng.random(200000))).astype(np.float32)
        off = (np.float32(a[b]) / t).astype(np.float64) - a[b] / t.astype(np.float64)
        tau[b] = t[np.argmax(off) if b % 2 else np.argmin(off)]
        assert abs(off).max() > 0.9 * 2.0 ** -21
    inp = AcceptInputs(target_logits=None, draft_probs=np.ones((B, k, V), np.float32),
                       draft_tokens=np.zeros((B, k), np.int32), uniforms=np.full((B, k + 1), 0.5, np.float32),
                       temperature=tau)
    logits, _, _, ratio = run_fused(f32_to_bf16_bits(hidden), f32_to_bf16_bits(weight), inp)
    np.testing.assert_array_equal(logits[:, 0, 1], -a.astype(np.float32))
    ones = V // 2000
    rest = (V - ones) * np.exp(-a / tau.astype(np.float64))
    want = 1.0 / (ones + rest)
    err = np.abs(ratio[:, 0].astype(np.float64) - want) / want
    assert (err <= rest * want * (2.0 ** -23 + 2.0 ** -24) + 2.0 ** -24).all(), err
