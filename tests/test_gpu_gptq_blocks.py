"""GPTQ packing where its blocks of 512 columns have edges: a narrow first block, alone or before others, one to 28 blocks, and rows so long that
U's diagonal blocks lie in the errors' slots.  Rows do not interact, so the oracle's fp64 sweep takes some of them: those of the first and the last
CTA and a few between.  Bit for bit."""
import numpy as np
import pytest

import synth
from oracle import gptq
from tests import plans
from tests.gpu_util import dev, host

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("N,K,r,R,fp16", [
    (24, 96, 32, 1, True),        # a block of three groups: rounding warps without one
    (592, 512, 64, 4, False),     # one whole block
    (16, 544, 32, 1, False),      # a first block of one group
    (304, 1056, 64, 3, True),     # the same before two whole ones
    (904, 992, 96, 7, False),     # a first block of 15 groups
    (600, 768, 256, 5, False),    # of eight: a group per rounding warp
    (664, 800, 0, 5, False),      # of nine
    (1184, 1536, 64, 8, True),    # whole blocks only
    (1040, 3584, 448, 8, False),  # no room behind the errors
    (152, 14336, 1792, 2, False),  # the same with two rows
])
def test_pack_weights_gptq_blocks(N, K, r, R, fp16):
    import paper_2412_14363_b200 as resq

    assert plans.gptq_rows(N, K) == R
    rng = np.random.default_rng(N + K)
    Wp = synth.projected_weights_direct(N, K, seed=40 + N)
    U = np.zeros((K, K), np.float32)
    if K < 8000:  # random feedback of the size that a correlated Hessian gives
        U[:] = np.triu(rng.standard_normal((K, K), dtype=np.float32) * np.float32(1.2 / np.sqrt(K)), 1)
    else:
        j = rng.integers(0, K - 1, 4096)
        U[j, j + 1 + (rng.random(4096) * (K - 1 - j)).astype(int)] = 0.3
    U[np.arange(K), np.arange(K)] = rng.uniform(0.4, 2.0, K)
    desc = resq.layer_desc(K, N, r, resq.SCALE_FP16 if fp16 else resq.SCALE_FP32)
    W = resq.resq_pack_weights_gptq(desc, dev(Wp), dev(U))
    assert resq.resq_device_status() == resq.OK
    rows = np.unique(np.r_[0:R, N - 1 - (N - 1) % R:N, rng.integers(0, N, 5)])
    pw = gptq.pack_weights_gptq(Wp[rows], r, U, scale_fp16=fp16)
    assert (host(W.w8)[rows] == pw.q8).all()
    assert (host(W.w4_i8)[rows] == pw.q4).all()
    assert (host(W.w4)[rows] == pw.w4_packed).all()
    assert (host(W.s_w8.float())[rows].view(np.uint32) == pw.s8.view(np.uint32)).all()
    assert (host(W.s_w4.float())[rows].view(np.uint32) == pw.s4.view(np.uint32)).all()


def test_a_short_wait_limit_leaves_a_sweep_alone():
    """Warps wait for whole blocks of columns (0.2 ms here), longer than a limit that serves the waits of other kernels."""
    import torch

    import paper_2412_14363_b200 as resq

    K, N = 8192, 296
    g = torch.Generator(device="cuda").manual_seed(K)
    Wp = torch.randn(N, K, device="cuda", generator=g) / K ** 0.5
    U = torch.triu(torch.randn(K, K, device="cuda", generator=g) / K ** 0.5)
    U.diagonal().copy_(torch.rand(K, device="cuda", generator=g) + 0.5)
    desc = resq.layer_desc(K, N, 1024)
    want = resq.resq_pack_weights_gptq(desc, Wp, U)
    resq.resq_set_option(resq.OPT_WAIT_LIMIT_US, 100)
    try:
        got = resq.resq_pack_weights_gptq(desc, Wp, U)
        assert resq.resq_device_status() == resq.OK
    finally:
        resq.resq_set_option(resq.OPT_WAIT_LIMIT_US, 2_000_000)
    assert torch.equal(got.w8, want.w8) and torch.equal(got.w4_i8, want.w4_i8)
