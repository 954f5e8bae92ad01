"""A CTA that gives up waiting for its cluster's pass-1 records voids its row,
whichever rank it has: the streaming kernels in a build whose rank-1 CTAs give
up at once (the records still land, and the CTA still waits for them before it
exits), without any fault.
"""
import numpy as np
import pytest

from paper_2608_26004_gb300 import asymspec as A
from paper_2608_26004_gb300 import build, synth
from tests._parity import device_inputs, run_gpu
from tests.test_gpu_xvocab import run as run_xvocab

pytestmark = pytest.mark.gpu

GREEDY, STOCH = A.MODE_GREEDY, A.MODE_STOCHASTIC


@pytest.fixture(scope="module")
def torch(tmp_path_factory):
    import torch as _torch
    assert _torch.cuda.is_available(), "the gpu tests need a CUDA device"
    path = str(tmp_path_factory.mktemp("late") / "libasymspec_late.so")
    build.build_cuda(force=True, target=path, defines=("ASYMSPEC_TEST_LATE_RANK=1",))
    keep = A._lib, A.LIB_PATH
    A._lib, A.LIB_PATH = None, path
    yield _torch
    A._lib, A.LIB_PATH = keep


def all_void(L, N, err):
    return np.all(L == -1) and np.all(N == -1) and err & A.DATA_TIMEOUT


@pytest.mark.parametrize("full", ["row", True])
@pytest.mark.parametrize("V", [32000, 32001])  # on and off the 16-byte boundaries
@pytest.mark.parametrize("mode", [GREEDY, STOCH])
@pytest.mark.parametrize("div", [A.DIV_JSD, A.DIV_KL, A.DIV_NONE])
def test_a_late_rank_voids_every_row_of_the_step(torch, div, mode, V, full):
    batch = synth.generate(synth.Recipe(), 17, 3, 2, V, synth.BF16)
    g = run_gpu(batch, torch, mode=mode, divergence=div, full=full)
    assert all_void(g["accept_len"], g["next_token"], int(g["error_word"][0]))
    # clusters of one CTA have no rank 1, and find no mark of the call before
    x = device_inputs(batch, torch)
    fv = A.FuseVerify(3, 2)
    for C in (0, 1):
        r = fv(x["a"], x["b"], x["t"], x["tokens"], x["probs"], x["unif"], mode=mode,
               divergence=div, row_stats=full is True, cluster_size=C)
        L, N, err = (r[n].cpu().numpy() for n in ("accept_len", "next_token", "error_word"))
        assert all_void(L, N, int(err[0])) if C == 0 else (np.all(L >= 0) and err[0] == 0)


@pytest.mark.parametrize("mode", [GREEDY, STOCH])
def test_a_late_rank_voids_every_row_of_the_cross_family_step(torch, mode):
    x = synth.make_xvocab(synth.CONFIGS[1].recipe, 5, 2, 2, 40000, 52000, 48000, synth.BF16)
    L, N, I, err = run_xvocab(torch, x, mode)
    assert all_void(L, N, err) and np.all(I == -1)
