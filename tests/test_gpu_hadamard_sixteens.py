"""Rows of a power of two (from 1024 on groups of sixteen coefficients, then passes over pairs): codes and scales of the butterflies taken one
index bit after another, lowest first, each sum rounded to fp32: bit for bit."""
import pytest
import torch


def _butterflies(X, K):
    c = X.float()
    for bit in range(K.bit_length() - 1):
        v = c.view(X.shape[0], K >> (bit + 1), 2, 1 << bit)
        c = torch.stack([v[:, :, 0] + v[:, :, 1], v[:, :, 0] - v[:, :, 1]], 2).reshape(X.shape[0], K)
    return c * torch.tensor(1.0 / K ** 0.5, dtype=torch.float64).to(torch.float32).cuda()


@pytest.mark.gpu
@pytest.mark.parametrize("K", [32, 256, 512, 1024, 2048, 4096, 8192, 16384, 32768])
@pytest.mark.parametrize("T,part", [(1, 0), (148, 32), (300, 0), (200, 1)])
def test_power_of_two_rows(K, T, part):
    import paper_2412_14363_b200 as resq

    r = 0 if K == 32 else K // 8 if part == 1 else part
    g = torch.Generator(device="cuda").manual_seed(K + T)
    X = (torch.randn(T, K, device="cuda", generator=g) * torch.exp2(torch.randint(-6, 7, (T, 1), device="cuda", generator=g))).to(torch.bfloat16)
    if T > 2:
        X[1] = 0
        X[2] = 1.0
    z = lambda shape, dt: torch.full(shape, 77, dtype=dt, device="cuda")
    q8, q4, q4e = z((T, r), torch.int8) if r else None, z((T, (K - r) // 2), torch.uint8), z((T, K - r), torch.int8)
    s8, s4 = z((T,), torch.float32), z((T,), torch.float32)
    resq.resq_hadamard_quantize(X, r, q8, q4, s8, s4, q4e)
    assert resq.resq_device_status() == resq.OK
    C = _butterflies(X, K)
    for seg, q, s, top in ((C[:, :r], q8, s8, 127.0), (C[:, r:], q4e, s4, 7.0)):
        if seg.shape[1] == 0:
            assert (s == 0).all()
            continue
        want = seg.abs().amax(1) / torch.full((T,), top, device="cuda")
        assert torch.equal(s, want)
        codes = torch.where(want[:, None] > 0, torch.round(seg / want[:, None]), torch.zeros_like(seg))
        assert torch.equal(q.float(), codes)
    n = q4e.to(torch.int16) & 15
    assert torch.equal(q4.to(torch.int16), n[:, ::2] | n[:, 1::2] << 4)
