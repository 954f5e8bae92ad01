"""The production row kernel's second pass runs only for rows whose decision
needs it; every outcome of that choice against the oracle.

A row that passes its acceptance test at D = 0, or fails it at the gate's
largest D, is decided by its normalisers alone; the others need the divergence,
and rejected rows the residual masses.
"""
import numpy as np
import pytest

from paper_2608_26004_gb300 import asymspec as A
from paper_2608_26004_gb300 import synth
from tests._parity import check_decisions, device_inputs, run_gpu, run_oracle

pytestmark = pytest.mark.gpu

GREEDY, STOCH = A.MODE_GREEDY, A.MODE_STOCHASTIC


@pytest.fixture(scope="module")
def torch():
    import torch as _torch
    assert _torch.cuda.is_available(), "the gpu tests need a CUDA device"
    from paper_2608_26004_gb300 import build
    build.build_cuda()
    return _torch


def batch_over_the_threshold(B, K, V, dtype, seed, torch, mode=STOCH, gamma=0.5, beta=1.0):
    """Inputs whose acceptance ratios spread from a quarter of gamma to four
    times gamma: below gamma / 2 rejected at every D, above gamma accepted at
    every D, between them decided by D (drafts' probabilities set from the
    oracle's q(d); greedy: the verifier's logit of the draft token moved)."""
    rc = synth.Recipe(sigma_c=4.0, frac_lo=0.2, frac_hi=0.4)
    b = synth.generate(rc, seed, B, K, V, dtype)
    rng = np.random.default_rng(seed)
    want = gamma * 2.0 ** rng.uniform(-2, 2, (B, K))
    x = device_inputs(b, torch, device="cpu")
    a, c, t = (x[n].double() for n in "abt")
    d = x["tokens"].long()[..., None]
    if mode == STOCH:
        s = t + beta * (a - c)
        q = (s[:, :K].gather(-1, d) - s[:, :K].logsumexp(-1, keepdim=True)).exp()[..., 0].numpy()
        u = np.maximum(b.uniforms[:, :K], 0.05)
        # q / (p u) = want, with p in (0, 1]
        p = np.clip(q / (want * u), 1e-30, 1.0)
        b.draft_probs[:] = p.astype(np.float32)
        b.uniforms[:, :K] = u
        ratio = q / (b.draft_probs.astype(np.float64) * u)
    else:
        lb = (c[:, :K].gather(-1, d) - c[:, :K].logsumexp(-1, keepdim=True))[..., 0].numpy()
        tk, e = t[:, :K].numpy(), np.exp
        ratio = np.empty((B, K))
        for i in range(B):
            for k in range(K):
                row, di = tk[i, k], int(d[i, k, 0])
                rest = np.log(np.sum(e(np.delete(row, di))))
                pt = min(want[i, k] * e(lb[i, k]), 0.9)  # softmax(t)[d] wanted
                val = rest + np.log(pt / (1 - pt))
                f = np.float32(val)
                if dtype == synth.BF16:
                    w = (f.view(np.uint32) + np.uint32(0x8000)) >> np.uint32(16)
                    b.logits_ver[i, k, di] = np.uint16(w)
                    f = np.uint32(w << np.uint32(16)).view(np.float32)
                else:
                    b.logits_ver[i, k, di] = f
                lt = float(f) - np.logaddexp(rest, float(f))
                ratio[i, k] = e(lt - lb[i, k])
    return b, ratio / gamma


def accept_and_next(batch, torch, mode, **kw):
    g = run_gpu(batch, torch, mode=mode, full="row", **kw)
    return g["accept_len"], g["next_token"], int(g["error_word"][0])


SHAPES = [(6, 3, 4104, synth.BF16), (5, 4, 40000, synth.BF16), (4, 3, 12288, synth.FP32),
          (40, 3, 2048, synth.FP32), (3, 2, 16, synth.BF16)]


@pytest.mark.parametrize("div", [A.DIV_JSD, A.DIV_KL, A.DIV_NONE, A.DIV_LAMBDA])
@pytest.mark.parametrize("B,K,V,dtype", SHAPES)
@pytest.mark.parametrize("mode", [GREEDY, STOCH])
def test_every_path_agrees_with_the_oracle(torch, B, K, V, dtype, mode, div):
    batch, r = batch_over_the_threshold(B, K, V, dtype, 500 + V + div, torch, mode)
    if B * K >= 12:
        assert (r < 0.5).any() and (r > 1.0).any() and ((r > 0.5) & (r < 1.0)).any()
    L, N, err = accept_and_next(batch, torch, mode, divergence=div)
    o = run_oracle(batch, mode=mode, divergence=div, logprobs=False)
    assert err == 0 and not o.error.any()
    check_decisions(batch, np.arange(B), L, N, o, mode)


@pytest.mark.parametrize("where", ["a", "b", "t"])
@pytest.mark.parametrize("mode", [GREEDY, STOCH])
def test_non_finite_logits_void_the_element_on_every_path(torch, mode, where):
    # whether or not the row's decision needs D
    batch, r = batch_over_the_threshold(9, 3, 12288, synth.FP32, 77, torch, mode)
    arr = {"a": batch.logits_full, "b": batch.logits_comp, "t": batch.logits_ver}[where]
    hit = np.zeros(9, bool)
    for i, k, v in ((1, 0, np.nan), (3, 1, np.inf), (5, 2, np.nan), (7, 0, np.inf)):
        arr[i, k, 17 + 400 * i] = v
        hit[i] = True
    L, N, err = accept_and_next(batch, torch, mode)
    assert np.array_equal(L < 0, hit) and np.array_equal(N < 0, hit)
    assert err & A.DATA_NONFINITE


@pytest.mark.parametrize("gap", [60.0, 95.0, 200.0])
def test_contexts_far_apart_on_a_token(torch, gap):
    # finite logits with b - a beyond the range of q/p = e^gap in fp32
    batch, _ = batch_over_the_threshold(8, 3, 4096, synth.FP32, 31, torch, STOCH)
    batch.logits_full[::2, :, 100:104] -= np.float32(gap)
    batch.logits_comp[1::2, :, 200] += np.float32(gap)
    for mode in (GREEDY, STOCH):
        L, N, err = accept_and_next(batch, torch, mode)
        o = run_oracle(batch, mode=mode, logprobs=False)
        assert err == 0 and not o.error.any()
        check_decisions(batch, np.arange(8), L, N, o, mode)


def test_more_rows_than_the_decision_kernel_keeps_on_chip(torch):
    # K + 1 above 64: the stop row's group is selected again after the scan
    for K in (63, 64, 80):
        batch, _ = batch_over_the_threshold(3, K, 1024, synth.BF16, 900 + K, torch, STOCH, gamma=0.01)
        batch.draft_probs[:2, :50] *= np.float32(1e-3)  # accepted for at least 50 rows
        for gamma in (0.01, 1e-6):
            L, N, err = accept_and_next(batch, torch, STOCH, gamma=gamma)
            o = run_oracle(batch, mode=STOCH, gamma=gamma, logprobs=False)
            assert err == 0
            check_decisions(batch, np.arange(3), L, N, o, STOCH)
