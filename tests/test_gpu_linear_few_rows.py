"""resq_linear and resq_linear_asym of up to eight tokens, whose rows the product quantizes itself: the bits of the row quantizer and the
product in two calls, at the edges of the rule, with rows that are zero, constant, half-way between codes, infinite or NaN."""
import pytest
import torch

from tests import plans


def test_rule_for_quantizing_rows():
    for T, widest in ((1, 16384), (2, 8192), (3, 2048), (4, 2048), (5, 1024), (8, 1024)):
        assert plans.quantizes_rows(T, widest) and not plans.quantizes_rows(T, widest + 32), T
    assert not plans.quantizes_rows(9, 64)


def test_ranges_that_meet():
    base = 0x7F0000000000
    for a, an, b, bn in ((0, 64, 64, 16), (64, 16, 0, 64), (0, 4096, 8192, 16), (0, 16, 16, 1 << 40)):
        assert not plans.ranges_meet(base + a, an, base + b, bn)
    for a, an, b, bn in ((0, 64, 0, 64), (0, 64, 48, 64), (48, 64, 0, 64), (0, 1 << 40, 1 << 39, 16), (16, 16, 0, 1 << 40), (0, 65, 64, 16)):
        assert plans.ranges_meet(base + a, an, base + b, bn)


def _rows(T, K, g):
    x = torch.randn(T, K, device="cuda", generator=g) * torch.exp2(torch.randint(-6, 7, (T, 1), device="cuda", generator=g))
    x[:, :: 97] *= 20
    return x.to(torch.bfloat16)


@pytest.mark.gpu
@pytest.mark.parametrize("asym", [False, True])
@pytest.mark.parametrize("T,K,r,N", [
    (1, 2048, 256, 3072), (1, 64, 32, 8), (1, 16384, 2048, 1024), (1, 16416, 2048, 64),  # the last: a quantizer of its own
    (2, 8192, 1024, 264), (2, 4096, 0, 40), (2, 8224, 32, 8), (3, 2048, 256, 2000), (4, 2048, 2016, 1184), (4, 2080, 32, 64), (5, 1024, 128, 2048),
    (6, 1056, 32, 136), (6, 992, 32, 136), (7, 800, 224, 3072), (8, 1024, 256, 6144), (8, 512, 0, 8), (9, 1024, 256, 512)])
def test_linear_of_few_rows(T, K, r, N, asym):
    import paper_2412_14363_b200 as resq

    g = torch.Generator(device="cuda").manual_seed(T * K + r)
    desc = resq.layer_desc(K, N, r, resq.SCALE_FP16 if T % 2 else resq.SCALE_FP32)
    W = resq.resq_pack_weights(desc, torch.randn(N, K, device="cuda", generator=g), with_w4_i8=asym)
    wsum = resq.resq_weight_row_sums(W) if asym else None
    ws = (resq.alloc_workspace_asym if asym else resq.alloc_workspace)(desc, T, False, asym)
    X = _rows(T, K, g)
    forms = [X, X.clone(), X.clone()]
    forms[1][0] = 0
    forms[1][-1, r:] = 3.0                                       # a constant segment
    forms[1][T // 2] = (torch.arange(K, device="cuda") % 15 - 7) * 0.5  # quotients on half-integers
    forms[1][T // 2, 0] = 7
    forms[2][0, K // 2] = float("inf")
    forms[2][-1, K - 1] = float("nan")
    z = lambda n, dt=torch.float32: torch.zeros(n, dtype=dt, device="cuda")
    for X in forms:
        for dt in (torch.bfloat16, torch.float32):
            Y, want = (torch.full((T, N), 5.0, dtype=dt, device="cuda") for _ in range(2))
            s = [z(T) for _ in range(4)]
            x4 = z((T, (K - r) // 2), torch.uint8)
            if asym:
                resq.resq_linear_asym(W, *wsum, X, None, Y, ws)
                u8 = z((T, max(r, 1)), torch.uint8) if r else None
                resq.resq_project_quantize_asym(X, None, r, u8, x4, *s)
                resq.resq_mixed_gemm_asym(W, *wsum, u8, x4, *s, want, ws)
            else:
                resq.resq_linear(W, X, None, Y, ws)
                x8 = z((T, r), torch.int8) if r else None
                resq.resq_project_quantize(X, None, r, x8, x4, s[0], s[1])
                resq.resq_mixed_gemm(W, x8, x4, s[0], s[1], want, ws)
            assert resq.resq_device_status() == resq.OK
            same = (Y == want) | (Y.isnan() & want.isnan())
            assert same.all(), (X is forms[2], dt, (~same).sum().item())


@pytest.mark.gpu
@pytest.mark.parametrize("asym", [False, True])
@pytest.mark.parametrize("T,K,r,N", [(1, 4096, 512, 6144), (4, 2048, 256, 2048), (8, 1024, 128, 4096)])
def test_weights_packed_just_before(T, K, r, N, asym):
    """The call may directly follow the packing of its layer, also with the option that lets products of few tokens stream weights early."""
    import ctypes

    import paper_2412_14363_b200 as resq

    g = torch.Generator(device="cuda").manual_seed(K)
    desc = resq.layer_desc(K, N, r)
    raw = [torch.randn(N, K, device="cuda", generator=g) for _ in range(2)]
    W = resq.resq_pack_weights(desc, raw[0])
    ws = (resq.alloc_workspace_asym if asym else resq.alloc_workspace)(desc, T, False, True)
    X, Y = _rows(T, K, g), torch.empty((T, N), device="cuda")

    def pack(i):
        assert resq.lib.resq_pack_weights(ctypes.byref(desc), raw[i].data_ptr(), *(t.data_ptr() for t in (W.w8, W.w4, W.s_w8, W.s_w4, W.w4_i8)),
                                          torch.cuda.current_stream().cuda_stream) == resq.OK

    def linear(sums):
        if asym:
            resq.resq_linear_asym(W, *sums, X, None, Y, ws)
        else:
            resq.resq_linear(W, X, None, Y, ws)

    sums, want = [], []
    for i in range(2):
        pack(i)
        sums.append(resq.resq_weight_row_sums(W))
        torch.cuda.synchronize()
        linear(sums[i])
        want.append(Y.clone())
    resq.resq_set_option(resq.OPT_DECODE_EARLY_WEIGHTS, 1)
    try:
        for k in range(40):
            torch.cuda._sleep(200000)  # the calls below are enqueued before the first of them runs
            pack(k & 1)
            linear(sums[k & 1])
            assert torch.equal(Y, want[k & 1]), k
    finally:
        resq.resq_set_option(resq.OPT_DECODE_EARLY_WEIGHTS, 0)
    assert resq.resq_device_status() == resq.OK


@pytest.mark.gpu
@pytest.mark.parametrize("asym", [False, True])
@pytest.mark.parametrize("T,K,N,dt,at", [
    (1, 2048, 2048, torch.bfloat16, 0), (4, 2048, 2048, torch.bfloat16, 0), (8, 1024, 1024, torch.bfloat16, 0), (9, 1024, 1024, torch.bfloat16, 0),
    (17, 1024, 1024, torch.bfloat16, 0), (2, 4096, 2048, torch.float32, 0), (8, 1024, 512, torch.float32, 32), (3, 1024, 4096, torch.bfloat16, 4096),
    (1, 16384, 16384, torch.bfloat16, 32752)])
def test_y_over_x(T, K, N, dt, at, asym):
    """Y on X, or on a part of it from byte `at` on: the bits of a call with buffers apart, many times over; right behind X it is one launch."""
    import paper_2412_14363_b200 as resq

    g = torch.Generator(device="cuda").manual_seed(K + T)
    r = K // 8
    desc = resq.layer_desc(K, N, r)
    W = resq.resq_pack_weights(desc, torch.randn(N, K, device="cuda", generator=g))
    sums = resq.resq_weight_row_sums(W) if asym else None
    ws = (resq.alloc_workspace_asym if asym else resq.alloc_workspace)(desc, T, False, True)
    x_bytes, y_bytes = T * K * 2, T * N * dt.itemsize
    buf = torch.zeros(x_bytes + y_bytes, dtype=torch.uint8, device="cuda")
    view = lambda start, n, t, cols: buf[start:start + n].view(t).view(T, cols)
    X0 = _rows(T, K, g)

    def linear(Y):
        X = view(0, x_bytes, torch.bfloat16, K)
        X.copy_(X0)
        before = resq.resq_launch_count()
        if asym:
            resq.resq_linear_asym(W, *sums, X, None, Y, ws)
        else:
            resq.resq_linear(W, X, None, Y, ws)
        return resq.resq_launch_count() - before

    want = torch.empty((T, N), dtype=dt, device="cuda")
    apart = linear(want)
    assert linear(view(x_bytes, y_bytes, dt, N)) == apart == (1 if plans.quantizes_rows(T, K) else 2)
    assert torch.equal(view(x_bytes, y_bytes, dt, N), want)
    Y = view(at, y_bytes, dt, N)
    for _ in range(25):
        assert linear(Y) == 2
        assert torch.equal(Y, want)
    assert resq.resq_device_status() == resq.OK
