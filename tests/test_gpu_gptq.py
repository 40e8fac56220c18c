"""GPU parity of GPTQ rounding at pack time (Section 5.1) through the C ABI: codes, packed bytes and scales bit for
bit against the oracle's fp64 sweep given the same inverse-Hessian factor, and the layer run on those weights."""
import numpy as np
import pytest
import torch

import oracle
import synth
from oracle import gptq
from tests import plans
from tests.gpu_util import bf16_bits_from_dev, bf16_to_dev, dev, host
from tests.test_gpu_parity import check_output

pytestmark = pytest.mark.gpu


@pytest.fixture(scope="module")
def resq():
    import paper_2412_14363_b200 as m
    return m


def _calibration(K, n, seed, dead_col=None):
    """Correlated calibration inputs with outlier channels: the Hessian is far from diagonal."""
    rng = np.random.default_rng(seed)
    X = synth.activations(n, K, "t4", seed=seed).astype(np.float64)
    X = X + 0.5 * np.roll(X, 1, axis=1) + 0.25 * (X @ (rng.standard_normal((K, 8)) / np.sqrt(K))) @ rng.standard_normal((8, K))
    if dead_col is not None:
        X[:, dead_col] = 0.0
    return X.astype(np.float32)


@pytest.mark.parametrize("N,K,r,fp16,dead_col", [(264, 512, 64, False, None), (72, 1024, 128, True, 17),
                                                 (40, 2048, 256, False, None), (16, 512, 0, False, 3)])
def test_pack_weights_gptq_bit_exact(resq, N, K, r, fp16, dead_col):
    Wp = synth.projected_weights_direct(N, K, seed=500 + N)
    H, dead = gptq.hessian(_calibration(K, 2 * K, 600 + N, dead_col))
    U = np.ascontiguousarray(gptq.inverse_factor(H).astype(np.float32))
    pw = gptq.pack_weights_gptq(Wp, r, U, dead, scale_fp16=fp16)
    desc = resq.layer_desc(K, N, r, resq.SCALE_FP16 if fp16 else resq.SCALE_FP32)
    W = resq.resq_pack_weights_gptq(desc, dev(Wp), dev(U), dev(dead.astype(np.uint8)) if dead.any() else None)
    assert resq.resq_device_status() == resq.OK
    assert (host(W.w8) == pw.q8).all()
    assert (host(W.w4_i8) == pw.q4).all()
    assert (host(W.w4) == pw.w4_packed).all()
    assert (host(W.s_w8.float()).view(np.uint32) == pw.s8.view(np.uint32)).all()
    assert (host(W.s_w4.float()).view(np.uint32) == pw.s4.view(np.uint32)).all()
    # the rounding differs from round-to-nearest and lowers the layer-output error on the calibration statistics
    rtn = oracle.pack_weights(Wp if not dead.any() else np.where(dead[None, :], 0, Wp).astype(np.float32), r, scale_fp16=fp16)
    assert (pw.q4 != rtn.q4).mean() > 0.05
    assert gptq.objective(Wp, pw, H).sum() < 0.9 * gptq.objective(Wp, rtn, H).sum()
    if dead_col is not None:
        assert not host(W.w4_i8 if dead_col >= r else W.w8)[:, dead_col - r if dead_col >= r else dead_col].any()


@pytest.mark.parametrize("N,K,r,kind,R", [
    (1200, 288, 32, "dense", 5),    # a last block of one 32-column group
    (600, 544, 512, "dense", 5),    # segment boundary on a block boundary
    (8, 32, 0, "dense", 1),         # one group
    (2400, 256, 64, "dense", 6),    # two rounds of CTAs
    (304, 288, 64, "dense", 3),     # a last CTA with one row of three
    (592, 256, 32, "dense", 4),
    (608, 320, 0, "dense", 5),      # three of five
    (752, 256, 32, "dense", 6),     # two of six
    (904, 544, 64, "dense", 7),     # one of seven
    (1184, 512, 64, "dense", 8),    # as many rows as a CTA takes
    (8, 14336, 1792, "sparse", 1),  # long rows
    (16, 512, 64, "ties", 1),       # quotients on half-integers, no feedback
    (16, 512, 64, "tiny", 1),       # diagonal below the normal float range, zero rows
])
def test_pack_weights_gptq_edges(resq, N, K, r, kind, R):
    """Bit for bit against the fp64 sweep where the kernel's tiling (R rows per CTA) and its two division routes have edges."""
    assert plans.gptq_rows(N, K) == R
    rng = np.random.default_rng(N + K)
    Wp = synth.projected_weights_direct(N, K, seed=900 + N)
    U = np.diag(rng.uniform(0.3, 3.0, K))
    if kind == "dense":
        U += np.triu(rng.standard_normal((K, K)) * 0.2, 1)
    elif kind == "sparse":
        j = rng.integers(0, K - 1, 256)
        U[j, j + 1 + (rng.random(256) * (K - 1 - j)).astype(int)] = 0.3
    elif kind == "ties":
        Wp = (rng.integers(-14, 15, (N, K)) * 0.5 / 64).astype(np.float32)
        Wp[:, :r] = rng.integers(-254, 255, (N, r)) * 0.5 / 64
        Wp[:, 0], Wp[:, r] = 127 / 64, 7 / 64  # scales exactly 1/64
    else:
        U *= 1e-39
        U[:, 5] += 1e-41 * (np.arange(K) < 5)
        Wp[3] = 0.0
        Wp[4, 1:] = 0.0
    U = np.ascontiguousarray(U.astype(np.float32))
    pw = gptq.pack_weights_gptq(Wp, r, U)
    W = resq.resq_pack_weights_gptq(resq.layer_desc(K, N, r), dev(Wp), dev(U))
    assert (host(W.w8) == pw.q8).all()
    assert (host(W.w4_i8) == pw.q4).all()
    assert (host(W.w4) == pw.w4_packed).all()
    assert (host(W.s_w8).view(np.uint32) == pw.s8.view(np.uint32)).all()
    assert (host(W.s_w4).view(np.uint32) == pw.s4.view(np.uint32)).all()


def test_layer_on_gptq_weights(resq):
    """resq_linear consumes the GPTQ-rounded weights like any packed weights: output exact against the oracle's layer."""
    T, K, N, r = 48, 1024, 264, 128
    C_bits = synth.f32_to_bf16_bits(synth.activations(T, K, "t4", seed=701))
    Wp = synth.projected_weights_direct(N, K, seed=702)
    H, dead = gptq.hessian(_calibration(K, 2 * K, 703))
    U = np.ascontiguousarray(gptq.inverse_factor(H).astype(np.float32))
    pw = gptq.pack_weights_gptq(Wp, r, U)
    res = oracle.linear(C_bits, None, pw)
    desc = resq.layer_desc(K, N, r)
    W = resq.resq_pack_weights_gptq(desc, dev(Wp), dev(U))
    ws = resq.alloc_workspace(desc, T, False, True)
    y32 = torch.empty((T, N), dtype=torch.float32, device="cuda")
    resq.resq_linear(W, bf16_to_dev(C_bits), None, y32, ws)
    ybf = torch.empty((T, N), dtype=torch.bfloat16, device="cuda")
    resq.resq_linear(W, bf16_to_dev(C_bits), None, ybf, ws)
    assert resq.resq_device_status() == resq.OK
    check_output(res, pw, host(y32), bf16_bits_from_dev(ybf))


def test_gptq_rejects_rows_too_wide_for_shared_memory(resq):
    K = 28672
    desc = resq.layer_desc(K, 8, K // 8)
    z = torch.zeros(16, dtype=torch.float32, device="cuda")
    st = resq.lib.resq_pack_weights_gptq(__import__("ctypes").byref(desc), z.data_ptr(), z.data_ptr(), None, z.data_ptr(), z.data_ptr(),
                                         z.data_ptr(), z.data_ptr(), None, None)
    assert st == resq.ERR_SHAPE
