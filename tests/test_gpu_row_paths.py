"""The streaming row kernel: its second pass runs only for rows whose decision
needs it, and rows may start off the 16-byte boundaries; every outcome of both
against the oracle.

A row that passes its acceptance test at D = 0, or fails it at the gate's
largest D, is decided by its normalisers alone; the others need the divergence,
and rejected rows the residual masses.
"""
import numpy as np
import pytest

from paper_2608_26004_gb300 import asymspec as A
from paper_2608_26004_gb300 import synth
from tests._parity import D_TOL, check_decisions, compare, device_inputs, run_gpu, run_oracle

pytestmark = pytest.mark.gpu

GREEDY, STOCH = A.MODE_GREEDY, A.MODE_STOCHASTIC


@pytest.fixture(scope="module", name="torch")
def torch_():
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


# ---------------------------------------------------------------- rows off the 16-byte boundaries

def shifted(x, offset, torch):
    """The logits in buffers that start `offset` elements after a 16-byte boundary."""
    out = dict(x)
    for key in "abt":
        buf = torch.full((x[key].numel() + offset + 16,), float("nan"), dtype=x[key].dtype,
                         device="cuda")
        assert buf.data_ptr() % 16 == 0
        view = buf[offset:offset + x[key].numel()]
        view.copy_(x[key].reshape(-1))
        out[key] = view.view(x[key].shape)
    return out


@pytest.mark.parametrize("mode", [GREEDY, STOCH])
@pytest.mark.parametrize("dtype", [synth.BF16, synth.FP32])
@pytest.mark.parametrize("V", [16384, 16385, 16387, 16391, 33333])
def test_rows_at_odd_addresses(torch, V, dtype, mode):
    # every offset of a row inside its first vector: odd V moves it from row to
    # row, an offset base moves all rows; the buffers around the rows hold NaN
    batch, _ = batch_over_the_threshold(4, 3, V, dtype, 40 + V, torch, mode)
    o = run_oracle(batch, mode=mode, logprobs=False)
    x = device_inputs(batch, torch)
    for offset in (0, 1, 2, 3, 5) if dtype == synth.BF16 else (0, 1, 3):
        g = run_gpu(batch, torch, mode=mode, full="row", inputs=shifted(x, offset, torch))
        assert int(g["error_word"][0]) == 0
        check_decisions(batch, np.arange(4), g["accept_len"], g["next_token"], o, mode)


@pytest.mark.parametrize("mode", [GREEDY, STOCH])
@pytest.mark.parametrize("dtype", [synth.BF16, synth.FP32])
def test_edges_hold_the_answer(torch, dtype, mode):
    # the emitted token, the draft token and the spike of every row among the
    # first or last elements of the row, which no whole vector holds
    B, K, V = 6, 2, 16391
    for at in (0, 1, 2, V - 3, V - 2, V - 1):
        batch, _ = batch_over_the_threshold(B, K, V, dtype, 7000 + at, torch, mode)
        bits = np.float32(30.0)
        big = (bits.view(np.uint32) >> 16).astype(np.uint16) if dtype == synth.BF16 else bits
        batch.logits_ver[..., at] = big
        batch.draft_tokens[::2] = at
        for cluster in (0, 5, 16):
            g = run_gpu(batch, torch, mode=mode, full="row", cluster_size=cluster)
            o = run_oracle(batch, mode=mode, logprobs=False)
            assert int(g["error_word"][0]) == 0
            check_decisions(batch, np.arange(B), g["accept_len"], g["next_token"], o, mode)
        batch.logits_full[1, 0, at] = np.float32("nan").view(np.uint32) >> 16 \
            if dtype == synth.BF16 else np.nan
        g = run_gpu(batch, torch, mode=mode, full="row")
        assert g["accept_len"][1] == -1 and (np.delete(g["accept_len"], 1) >= 0).all()


def test_an_overflowing_sum_beside_an_edge(torch):
    batch, _ = batch_over_the_threshold(3, 2, 16391, synth.FP32, 8, torch, STOCH)
    for arr in (batch.logits_full, batch.logits_comp, batch.logits_ver):
        arr[0, 1, 0] = 150.0
        arr[1, 0, 16390] = 150.0
        arr[2, 2, 9000] = 150.0
    for mode in (GREEDY, STOCH):
        L, N, err = accept_and_next(batch, torch, mode)
        o = run_oracle(batch, mode=mode, logprobs=False)
        assert err == 0
        check_decisions(batch, np.arange(3), L, N, o, mode)


def test_rows_at_different_offsets_take_the_generic_kernel(torch):
    batch, _ = batch_over_the_threshold(2, 2, 16385, synth.BF16, 12, torch, STOCH)
    x = device_inputs(batch, torch)
    y = shifted(x, 3, torch)
    x["b"] = y["b"]
    g = run_gpu(batch, torch, mode=STOCH, full="row", inputs=x)
    o = run_oracle(batch, mode=STOCH, logprobs=False)
    check_decisions(batch, np.arange(2), g["accept_len"], g["next_token"], o, STOCH)


# ---------------------------------------------------------------- every row recorded

@pytest.mark.parametrize("mode", [GREEDY, STOCH])
@pytest.mark.parametrize("B,K,V,dtype,offset,cluster", [
    (3, 2, 40000, synth.BF16, 0, 0), (2, 2, 12288, synth.FP32, 0, 1), (2, 3, 8200, synth.BF16, 0, 16),
    (3, 2, 16391, synth.BF16, 0, 0), (2, 2, 16391, synth.BF16, 3, 5), (2, 2, 16385, synth.FP32, 1, 0),
    (2, 1, 16, synth.BF16, 0, 0), (1, 70, 1024, synth.FP32, 0, 0)])
def test_recorded_rows(torch, B, K, V, dtype, offset, cluster, mode):
    # statistics, tokens and log-probabilities of every row, on and off the
    # 16-byte boundaries (16-byte and single stores of the log-probabilities)
    batch, _ = batch_over_the_threshold(B, K, V, dtype, 60 + V, torch, mode)
    x = shifted(device_inputs(batch, torch), offset, torch)
    for div in (A.DIV_JSD, A.DIV_KL, A.DIV_LAMBDA):
        g = run_gpu(batch, torch, mode=mode, divergence=div, inputs=x, cluster_size=cluster)
        o = run_oracle(batch, mode=mode, divergence=div)
        assert int(g["error_word"][0]) == 0
        # KL is not bounded by ln 2: its error grows with it, each p carrying the
        # rounding of its exponent (2^-23 |log2 p|, up to about 30 of them: 2.5e-6
        # of the sum in relative terms)
        compare(batch, g, o, mode=mode, check_stats=div != A.DIV_KL)
        err = np.abs(g["row_stats"][..., 4] - o.D)
        assert np.all(err <= D_TOL * np.maximum(1.0, np.abs(o.D)))


# ---------------------------------------------------------------- the order of the rows

@pytest.mark.parametrize("B,K", [(40, 3), (300, 1), (61, 5), (127, 4)])
@pytest.mark.parametrize("mode", [GREEDY, STOCH])
def test_every_row_is_taken_in_batches_of_several_waves(torch, B, K, mode):
    # more clusters than the chip holds: the bonus rows of the last elements
    # come last (all of them, or some), recorded rows likewise
    batch, _ = batch_over_the_threshold(B, K, 2048, synth.BF16, 2000 + B, torch, mode)
    o = run_oracle(batch, mode=mode)
    for cluster in (0, 4, 16):
        g = run_gpu(batch, torch, mode=mode, full="row", cluster_size=cluster)
        check_decisions(batch, np.arange(B), g["accept_len"], g["next_token"], o, mode)
    compare(batch, run_gpu(batch, torch, mode=mode, cluster_size=16), o, mode=mode)


@pytest.mark.parametrize("first,second", [
    # (B, V, recorded) of two calls on one workspace: every element of the
    # second is decided, whatever the first left where its counters lie
    ((4, 16392, False), (64, 16392, True)),
    ((4, 16391, False), (64, 1001, False)),   # then the generic kernel
    ((64, 16392, True), (4, 1001, False)),
    ((64, 16392, True), (4, 16392, True)),
])
@pytest.mark.parametrize("mode", [GREEDY, STOCH])
def test_batches_of_several_sizes_share_a_workspace(torch, mode, first, second):
    K = 7
    fv = A.FuseVerify(64, K, V_max=16392)
    for B, V, recorded in (first, second):
        batch = synth.generate(synth.Recipe(), 7, B, K, V, synth.BF16)
        x = device_inputs(batch, torch)
        out = {"accept_len": torch.full((B,), -7, dtype=torch.int32, device="cuda"),
               "next_token": torch.full((B,), -7, dtype=torch.int32, device="cuda"),
               "error_word": torch.zeros(1, dtype=torch.int32, device="cuda")}
        res = fv(x["a"], x["b"], x["t"], x["tokens"], x["probs"], x["unif"], mode=mode,
                 row_stats=recorded, row_tokens=recorded, out=out)
        torch.cuda.synchronize()
        want = run_gpu(batch, torch, mode=mode, full=recorded, tokens=recorded, logprobs=False)
        for name in ("accept_len", "next_token"):
            np.testing.assert_array_equal(res[name].cpu().numpy(), want[name])


@pytest.mark.parametrize("dtype", [synth.BF16, synth.FP32])
def test_a_token_that_holds_the_row_beside_a_low_reference(torch, dtype):
    # One entry M near 0 anywhere in a row of -14: the warp's first step mostly
    # sees the -14s.  What may round after M's term has entered the sum, each time
    # relative to the whole sum: 3 steps of its block, 2 additions in its vector
    # and 1 in its pair, 5 of the warp, 7 of the cluster's records, then the
    # logarithm and the addition of M: 20 roundings, uniform within 2^-24, 3.4e-8
    # RMS each and 1.6e-7 together.  (Not a bound on the largest error, for which
    # the 20 may add up to 1.2e-6; M's exponent against a reference of -14, 20 log2
    # units, rounds by 2.8e-7 RMS on its own.)
    B, K, V = 24, 3, 33333
    gen = torch.Generator().manual_seed(5)
    dt = torch.float32 if dtype == synth.FP32 else torch.bfloat16
    x = torch.full((3, B, K + 1, V), -14.0)
    at = torch.randint(V, (3, B, K + 1, 1), generator=gen)
    x.scatter_(-1, at, torch.rand(at.shape, generator=gen) * 1.4 - 0.7)
    a, b, t = x.to(dt).cuda()
    tokens = torch.zeros(B, K, dtype=torch.int32, device="cuda")
    res = A.FuseVerify(B, K)(a, b, t, tokens, row_stats=True)
    stats = res["row_stats"].double()
    err = torch.stack([stats[..., q] - z.double().logsumexp(-1) for q, z in enumerate((a, b, t))])
    assert err.square().mean().sqrt().item() <= 1.6e-7


@pytest.mark.parametrize("mode", [GREEDY, STOCH])
@pytest.mark.parametrize("V,cluster", [
    # vectors a CTA and where its slice starts in a line: one line and less,
    (8 * 8, 1), (8 * 9, 1), (8 * 67, 2),
    # slices that start off the lines,
    (8 * 1001, 3), (8 * 4001, 6),
    # and blocks of the last size cut on lines (504 vectors), one more, the largest
    (8 * 4032, 1), (8 * 4033, 1), (8 * 4096, 1),
])
def test_recorded_rows_in_blocks_cut_on_lines(torch, V, cluster, mode):
    batch = synth.generate(synth.Recipe(), 11, 3, 2, V, synth.BF16)
    g = run_gpu(batch, torch, mode=mode, cluster_size=cluster)
    compare(batch, g, run_oracle(batch, mode=mode), mode=mode)


@pytest.mark.parametrize("first,second", [
    # (B, V, arguments) of two calls on one workspace, the one's records and
    # results over the other's tickets:
    ((64, 1001, {}), (4, 1001, {})),                                  # generic, both
    ((4, 1001, {}), (64, 1001, {})),
    ((8, 16392, dict(delta_source=A.DELTA_A)), (64, 1001, {})),       # staged, then generic
    ((8, 16392, dict(row_tokens=True)), (64, 1001, {})),
    ((64, 16392, {}), (4, 1001, {})),                                 # streaming, then generic
    ((64, 1001, {}), (4, 16392, dict(row_stats=True))),
    (None, (64, 1001, {})), (None, (4, 16392, dict(row_stats=True))), (None, (4, 16392, {})),
    (None, (4, 16391, {})), (None, (4, 16392, dict(row_tokens=True))),
])
@pytest.mark.parametrize("own_size", [False, True])  # workspace_bytes of each call's own batch
@pytest.mark.parametrize("mode", [GREEDY, STOCH])
def test_whatever_lies_in_a_workspace(torch, mode, own_size, first, second):
    K = 7
    fv = A.FuseVerify(64, K, V_max=16392)
    fv.workspace.fill_(255)  # (no call needs it zeroed)
    whole = fv.nbytes
    for B, V, args in (c for c in (first, second) if c):
        batch = synth.generate(synth.Recipe(), 7, B, K, V, synth.BF16)
        x = device_inputs(batch, torch)
        out = {"accept_len": torch.full((B,), -7, dtype=torch.int32, device="cuda"),
               "next_token": torch.full((B,), -7, dtype=torch.int32, device="cuda"),
               "error_word": torch.zeros(1, dtype=torch.int32, device="cuda")}
        fv.nbytes = A.workspace_bytes(B, K, V) if own_size else whole
        fv(x["a"], x["b"], x["t"], x["tokens"], x["probs"], x["unif"], mode=mode, out=out, **args)
    torch.cuda.synchronize()
    o = run_oracle(batch, mode=mode, logprobs=False, delta_source=args.get("delta_source", A.DELTA_AB))
    assert int(out["error_word"].item()) == 0
    check_decisions(batch, np.arange(B), out["accept_len"].cpu().numpy(),
                    out["next_token"].cpu().numpy(), o, mode)


@pytest.mark.parametrize("top", [0.0, -0.2])
@pytest.mark.parametrize("full", ["row", True])
@pytest.mark.parametrize("V", [16384, 16387])
def test_a_draw_at_zero_beside_flushed_masses(torch, V, full, top):
    # bonus rows drawn at u = 0, their first entries around the smallest mass of
    # fp32: a token of positive mass is drawn, not an error
    bits = np.concatenate([np.arange(-128.0, -99.0, 0.125), np.arange(-126.6, -125.8, 0.01)])
    B = bits.size
    t = np.full((B, 2, V), -20.0, np.float32)
    t[..., 9000] = top
    t[:, 1, :4096] = (bits * np.log(2.0))[:, None]
    x = {n: torch.zeros(B, 2, V, device="cuda") for n in "ab"}
    tokens = torch.full((B, 1), 9000, dtype=torch.int32, device="cuda")
    r = A.FuseVerify(B, 1)(x["a"], x["b"], torch.from_numpy(t).cuda(), tokens,
                           torch.full((B, 1), 1e-3, device="cuda"), torch.zeros(B, 2, device="cuda"),
                           mode=STOCH, row_stats=full is True)
    L, N = r["accept_len"].cpu().numpy(), r["next_token"].cpu().numpy()
    assert int(r["error_word"].item()) == 0 and np.all(L == 1)
    assert np.all((N == 0) | (N >= 2048) & (N <= 4096))


@pytest.mark.parametrize("mode,div", [(STOCH, A.DIV_JSD), (STOCH, A.DIV_KL), (STOCH, A.DIV_NONE),
                                      (GREEDY, A.DIV_JSD)])
def test_more_elements_than_the_streaming_grid_holds(torch, mode, div):
    # above 65535 elements the staged kernel's production programs run: the same
    # decisions as on the streaming kernel (in halves), and as the oracle's on a few
    B, K, V = 65540, 1, 64
    gen = torch.Generator(device="cuda").manual_seed(3)
    a, b, t = (2 * torch.randn(B, K + 1, V, generator=gen, device="cuda") for _ in range(3))
    b = a + 0.5 * b
    a, b, t = (v.bfloat16() for v in (a, b, t))
    tokens = a[:, :K].float().argmax(-1).int()
    probs = a[:, :K].float().softmax(-1).max(-1).values
    unif = torch.rand(B, K + 1, generator=gen, device="cuda")
    assert A.plan(B, K, V, A.BF16, A.gate_params(mode=mode, divergence=div)).kernel == A.KERNEL_TMA

    def step(s):
        r = A.FuseVerify(s.stop - s.start, K)(a[s], b[s], t[s], tokens[s], probs[s], unif[s], mode=mode,
                                              divergence=div)
        assert int(r["error_word"].item()) == 0
        return np.stack([r["accept_len"].cpu().numpy(), r["next_token"].cpu().numpy()])

    whole = step(slice(0, B))
    halves = np.concatenate([step(slice(0, B // 2)), step(slice(B // 2, B))], 1)
    assert np.mean((whole != halves).any(0)) < 1e-3  # (near ties)
    sel = np.r_[0:40, B - 40:B]
    bits = [v[sel].contiguous().view(torch.int16).cpu().numpy().view(np.uint16) for v in (a, b, t)]
    few = synth.generate(synth.Recipe(), 1, sel.size, K, V, synth.BF16)
    few.logits_full[:], few.logits_comp[:], few.logits_ver[:] = bits
    few.draft_tokens[:], few.draft_probs[:] = tokens[sel].cpu().numpy(), probs[sel].cpu().numpy()
    few.uniforms[:] = unif[sel].cpu().numpy()
    o = run_oracle(few, mode=mode, divergence=div, logprobs=False)
    check_decisions(few, np.arange(sel.size), whole[0, sel], whole[1, sel], o, mode)
