"""The one-kernel cross-family step (fuse_verify_xrow) against the oracle:
increasing maps (rows read in token order, with long unpaired runs) and maps in
any order, rows on and off the 16-byte boundaries, one CTA and several a row.

Unpaired logits hold NaN, so reading one would void its element.
"""
import numpy as np
import pytest

from paper_2608_26004_gb300 import asymspec as A
from paper_2608_26004_gb300 import synth
from tests.test_gpu_xvocab import compare, oracle, run, torch  # noqa: F401  (the fixture too)

pytestmark = pytest.mark.gpu

GREEDY, STOCH = A.MODE_GREEDY, A.MODE_STOCHASTIC


def batch(B, K, S, V_d, V_v, dtype, kind, seed):
    x = synth.make_xvocab(synth.CONFIGS[3].recipe, seed, B, K, S, V_d, V_v, dtype)
    rng = np.random.default_rng(seed)
    nan = np.float32("nan") if dtype == synth.FP32 else np.uint16(0x7FC0)
    if kind == "any":      # the drafter's tokens renumbered at random
        to, V = rng.permutation(V_d), V_d
    elif kind == "gaps":   # runs of 4096 unpaired tokens in front, inside and behind
        to, V = np.arange(V_d) + 4096 * (1 + (np.arange(V_d) >= V_d // 2)), V_d + 3 * 4096
    else:
        to, V = np.arange(V_d), V_d

    def move(rows, idx, new_idx, V_new):
        out = np.full(rows.shape[:2] + (V_new,), nan, rows.dtype)
        out[..., new_idx] = rows[..., idx]
        return out

    md = to[x.map_d].astype(np.int32)
    return synth.XBatch(move(x.logits_full, x.map_d, md, V), move(x.logits_comp, x.map_d, md, V),
                        move(x.logits_ver, x.map_v, x.map_v, V_v), md, x.map_v, x.draft_tokens,
                        x.draft_probs, x.uniforms, B, K, S, V, V_v, dtype)


@pytest.mark.parametrize("kind", ["increasing", "gaps", "any"])
@pytest.mark.parametrize("B,K,S,V_d,V_v,dtype", [
    (40, 3, 600, 800, 704, synth.BF16),          # one CTA a row (every SM has a row)
    (3, 2, 40000, 52000, 48000, synth.BF16),     # a few CTAs a row
    (3, 2, 39999, 52008, 48001, synth.BF16),     # odd S, rows of t off the boundaries
    (2, 2, 20011, 26005, 24000, synth.FP32),     # rows of a and b off the boundaries
    (2, 3, 30000, 40004, 36004, synth.FP32),     # a unit of eight tokens past the row's end
    (5, 1, 2, 9, 5, synth.FP32),                 # the smallest shared set
])
def test_agrees_with_the_oracle(torch, B, K, S, V_d, V_v, dtype, kind):  # noqa: F811
    x = batch(B, K, S, V_d, V_v, dtype, kind, 300 + S)
    for mode in (GREEDY, STOCH):
        got = run(torch, x, mode)
        compared, flagged = compare(x, got, oracle(x, mode))
        assert compared + flagged == B and compared and got[3] == 0


def test_scores_of_unpaired_tokens_are_never_taken(torch):  # noqa: F811
    # every paired score far below what stands in for an unpaired one
    x = batch(4, 2, 600, 800, 704, synth.FP32, "increasing", 9)
    x.logits_ver[..., x.map_v] -= np.float32(2e30)
    for arr in (x.logits_full, x.logits_comp):
        arr[..., x.map_d] = np.round(arr[..., x.map_d])
    L, N, I, err = run(torch, x, GREEDY, beta=0.0)
    assert np.all((I >= 0) & (I < x.S)) and np.all(N == x.map_v[I]) and np.all(L >= 0)


def test_an_entry_far_above_its_warp(torch):  # noqa: F811
    for kind in ("increasing", "any"):
        x = batch(3, 2, 20000, 26000, 24000, synth.FP32, kind, 4)
        for i, j in ((0, 13000), (1, 3), (2, 19999)):
            x.logits_full[i, i, x.map_d[j]] = 150.0
            x.logits_comp[i, i, x.map_d[j]] = 150.0
            x.logits_ver[i, i, x.map_v[j]] = 150.0
        for mode in (GREEDY, STOCH):
            got = run(torch, x, mode)
            compare(x, got, oracle(x, mode))
            assert got[3] == 0


def test_another_map_on_the_same_workspace(torch):  # noqa: F811
    # calls queued one behind another, each with a map of its own: what a call
    # reads is the inverse map that its own check wrote
    B, K, S, V = 2, 2, 30000, 40000
    xs = [batch(B, K, S, V, V, synth.BF16, "any", 70 + i) for i in range(4)]
    want = [run(torch, x, GREEDY) for x in xs]
    keep = []
    ws = torch.zeros(A.xvocab_workspace_bytes(B, K, S, V, V, A.BF16), dtype=torch.uint8, device="cuda")
    for x in xs:
        logits = [torch.from_numpy(v.view(np.int16)).view(torch.bfloat16).cuda()
                  for v in (x.logits_full, x.logits_comp, x.logits_ver)]
        ints = [torch.from_numpy(np.ascontiguousarray(v, np.int32)).cuda()
                for v in (x.map_d, x.map_v, x.draft_tokens)]
        keep.append((logits, ints, torch.full((2, B), -7, dtype=torch.int32, device="cuda")))
    torch.cuda.synchronize()
    for (a, b, t), (md, mv, d), out in keep:
        st = A.fuse_verify_xvocab(a.data_ptr(), b.data_ptr(), V, t.data_ptr(), V, md.data_ptr(),
                                  mv.data_ptr(), S, d.data_ptr(), 0, 0, B, K, A.BF16,
                                  A.gate_params(mode=GREEDY), out[0].data_ptr(), out[1].data_ptr(),
                                  0, ws.data_ptr(), ws.numel(), 0,
                                  torch.cuda.current_stream().cuda_stream)
        assert st == A.OK
    torch.cuda.synchronize()
    for (_, _, out), (L, N, _, _) in zip(keep, want):
        assert np.array_equal(out.cpu().numpy(), np.stack([L, N]))
