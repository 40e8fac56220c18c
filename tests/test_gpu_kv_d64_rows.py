"""Attention of single rows at d_head = 64, whose keys and values are read from the cache's bytes in the products' own order: every group size,
lengths around a tile and a step, scores that grow along the cache (the reference is raised again and again) or fall; against softmax
in 64 bits over the cache's own codes.  2e-5 of the largest value: the bound of test_gpu_kv_d64.py."""
import math

import pytest
import torch

pytestmark = pytest.mark.gpu


def _dequantize(cache, b, n):
    """Keys and values of sequence b in 64 bits, [n][Hkv][64]."""
    blk = cache.data.view(cache.c.n_seqs, cache.c.n_kv_heads, -1, 3328)[b].transpose(0, 1)  # [blocks][Hkv][bytes]
    lead, out = blk.shape[:2], []
    for at in (0, 1664):
        c8 = blk[..., at:at + 256].reshape(*lead, 32, 8).double()
        c4 = blk[..., at + 256:at + 1152].reshape(*lead, 32, 28)
        c4 = torch.stack((c4 & 15, c4 >> 4), dim=-1).reshape(*lead, 32, 56).double()
        m = blk[..., at + 1152:at + 1664].contiguous().view(torch.float32).reshape(*lead, 32, 4).double()
        x = torch.cat((c8 * m[..., :1] + m[..., 1:2], c4 * m[..., 2:3] + m[..., 3:]), dim=-1)
        out.append(x.transpose(1, 2).reshape(-1, lead[1], 64)[:n])
    return out


@pytest.mark.parametrize("slope", [0.0, 0.05, -0.05])
@pytest.mark.parametrize("Hkv,group", [(3, 1), (2, 2), (1, 3), (2, 4), (1, 5), (1, 6), (2, 7), (1, 8)])
def test_attention_of_single_rows(Hkv, group, slope):
    import paper_2412_14363_b200 as resq
    from paper_2412_14363_b200 import kv

    d, Hq = 64, Hkv * group
    lens = [1, 2, 15, 16, 17, 31, 32, 33, 47, 64, 65, 96, 383, 385, 800, 0]
    g = torch.Generator(device="cuda").manual_seed(group)
    cache = kv.KvCache(len(lens), Hkv, 800, d)
    cache.data.fill_(0xFF)
    wq, su = kv.resq_uc_quantize(torch.linalg.qr(torch.randn(d, d, device="cuda", generator=g))[0].contiguous())
    common = torch.randn(Hkv, d, device="cuda", generator=g)
    for b, n in enumerate(lens):
        if n:
            k, v = (torch.randn(n, Hkv, d, device="cuda", generator=g) for _ in range(2))
            k = k + slope * torch.arange(n, device="cuda")[:, None, None] * common  # along the queries' common direction
            kv.resq_kv_append(cache, k.to(torch.bfloat16), v.to(torch.bfloat16), torch.full((n,), b, dtype=torch.int32, device="cuda"),
                              torch.arange(n, dtype=torch.int32, device="cuda"), wq, su)
    q = torch.randn(len(lens), Hq, d, device="cuda", generator=g) + common.repeat_interleave(group, 0) * (slope != 0)
    q16 = torch.empty(q.shape, dtype=torch.float16, device="cuda")
    kv.resq_query_project(q.to(torch.bfloat16), wq, su, q16)
    out = torch.full((len(lens), Hq, d), float("nan"), device="cuda")
    kv.resq_attention_decode(cache, q16, torch.tensor(lens, dtype=torch.int32, device="cuda"), out, kv.attention_workspace(cache, Hq))
    assert resq.resq_device_status() == resq.OK
    for b, n in enumerate(lens):
        if n == 0:
            assert (out[b] == 0).all()
            continue
        K, V = _dequantize(cache, b, n)
        for h in range(Hkv):
            rows = slice(h * group, (h + 1) * group)
            want = torch.softmax(q16[b, rows].double() @ K[:, h].T / math.sqrt(d), dim=1) @ V[:, h]
            assert (out[b, rows].double() - want).abs().amax() <= 2e-5 * V[:, h].abs().amax(), (n, h)
