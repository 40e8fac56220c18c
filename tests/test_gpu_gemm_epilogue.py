"""The mixed products, exact sums first, then the scaled values, with and without the sums written out: beyond 16 tokens every split of the
reduction at the edges of the token groups and channel tiles; from 9 to 16 tokens both forms of staged activations."""
import pytest
import torch

from tests import plans


def _unpack(w4, K4):
    lo = (w4 & 15).to(torch.int16)
    hi = (w4 >> 4).to(torch.int16)
    q = torch.stack([lo, hi], -1).reshape(w4.shape[0], K4)
    return torch.where(q > 7, q - 16, q)


@pytest.mark.gpu
@pytest.mark.parametrize("asym", [False, True])
@pytest.mark.parametrize("T,K,r,N,splits", [
    (17, 512, 64, 200, 1), (33, 256, 32, 264, 1), (300, 1024, 96, 520, 1), (40, 256, 224, 8, 1), (1537, 14336, 0, 4096, 1),
    (17, 8192, 1024, 8192, 2), (250, 14336, 0, 2184, 2), (23, 6144, 6112, 256, 3), (61, 14336, 1792, 1032, 3), (257, 14336, 32, 2048, 3),
    (1700, 256, 32, 3000, 0), (2049, 512, 480, 2056, 0), (1793, 384, 0, 4104, 0), (2100, 256, 128, 2064, 0),
    (9, 256, 32, 1024, None), (16, 2560, 320, 136, None), (16, 2592, 320, 136, None), (9, 4096, 512, 1192, None), (9, 4096, 512, 1176, None),
    (12, 3136, 0, 2000, None), (13, 2944, 2912, 2400, None), (15, 2048, 256, 3072, None)])  # None: weights streamed; 0: 256 x 256 tiles
def test_sums_and_scales(T, K, r, N, splits, asym):
    import paper_2412_14363_b200 as resq

    if splits is not None:
        pl = plans.mid(T, K, N, r)
        assert (pl.splits if pl.use else 0) == splits
    g = torch.Generator(device="cuda").manual_seed(T + K)
    K4 = K - r
    desc = resq.layer_desc(K, N, r, resq.SCALE_FP16 if T % 2 else resq.SCALE_FP32)
    W = resq.resq_pack_weights(desc, torch.randn(N, K, device="cuda", generator=g))
    codes = lambda lo, hi, n: torch.randint(lo, hi + 1, (T, n), device="cuda", generator=g)
    q8, q4 = (codes(0, 255, r), codes(0, 15, K4)) if asym else (codes(-128, 127, r), codes(-8, 7, K4))
    x8 = q8.to(torch.uint8 if asym else torch.int8) if r else None
    x4 = ((q4[:, ::2] & 15) | (q4[:, 1::2] & 15) << 4).to(torch.uint8)
    s8, s4, z8, z4 = (torch.rand(T, device="cuda", generator=g) + 0.01 for _ in range(4))
    ws = (resq.alloc_workspace_asym if asym else resq.alloc_workspace)(desc, T, False, True)
    w8, w4 = W.w8.double(), _unpack(W.w4, K4).double()
    a8, a4 = q8.double() @ w8.T, q4.double() @ w4.T  # whole numbers below 2^53: exact
    t8 = a8 * (s8.double()[:, None] * W.s_w8.double()) if r else torch.zeros_like(a8)
    t4 = a4 * (s4.double()[:, None] * W.s_w4.double())
    want, size = t8 + t4, t8.abs() + t4.abs()
    if asym:
        wsum = resq.resq_weight_row_sums(W)
        for z, sw, s in ((z8, W.s_w8, w8.sum(1)), (z4, W.s_w4, w4.sum(1))):
            if s.numel() and (r or sw is W.s_w4):
                term = z.double()[:, None] * (sw.double() * s)
                want, size = want + term, size + term.abs()
    for dt in (torch.float32, torch.bfloat16):
        outs = []
        for dbg in (False, True):
            skip = 16 // dt.itemsize if dbg else 0  # once on 32 bytes, once 16 behind
            Y = torch.full((skip + (T + 1) * N,), 9.0, dtype=dt, device="cuda")[skip:].view(T + 1, N)
            d = [torch.full((T, N), 77, dtype=torch.int32, device="cuda") if dbg else None for _ in range(2)]
            if asym:
                resq.resq_mixed_gemm_asym(W, *wsum, x8, x4, s8, s4, z8, z4, Y[:T], ws, *d)
            else:
                resq.resq_mixed_gemm(W, x8, x4, s8, s4, Y[:T], ws, *d)
            assert resq.resq_device_status() == resq.OK
            assert (Y[T] == 9).all()  # nothing behind the last token
            outs.append(Y[:T])
            if dbg:
                assert (d[0].double() == a8).all() and (d[1].double() == a4).all()
        assert torch.equal(outs[0], outs[1])
        # a rounding each: the sum to fp32, its scale and their product; the column factor and its product; up to three additions
        bound = 6 * 2.0 ** -24 * size
        if dt is torch.bfloat16:
            bound = bound + 2.0 ** -8 * want.abs()
        assert ((outs[0].double() - want).abs() <= bound).all()
