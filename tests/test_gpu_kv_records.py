"""Attention of single rows at d_head = 128 where its block list and its merge have edges: more sequences than a warp scans at once,
runs of no block, records of one (sequence, head) in more than one chunk of sixteen and in all four groups of threads, in chunks of eight, and
many of one sequence beside few of the others (edges of the sixteen that four warps share); against softmax in 64 bits over the dequantized cache."""
import math

import pytest
import torch

from tests.kv_util import OFF

pytestmark = pytest.mark.gpu


def _dequantize(cache, b, n, which):
    """Keys or values of sequence b in 64 bits, [n][Hkv][128]."""
    o8, o4, om = OFF[which]
    blk = cache.data.view(cache.c.n_seqs, cache.c.n_kv_heads, -1, 5632)[b].transpose(0, 1)  # [blocks][Hkv][bytes]
    lead = blk.shape[:2]
    c8 = blk[..., o8:o8 + 512].reshape(*lead, 32, 16).double()
    c4 = blk[..., o4:o4 + 1792].reshape(*lead, 32, 56)
    c4 = torch.stack((c4 & 15, c4 >> 4), dim=-1).reshape(*lead, 32, 112).double()
    s8, z8, s4, z4 = blk[..., om:om + 512].contiguous().view(torch.float32).reshape(*lead, 32, 4).double().unbind(-1)
    x = torch.cat((c8 * s8[..., None] + z8[..., None], c4 * s4[..., None] + z4[..., None]), dim=-1)
    return x.transpose(1, 2).reshape(-1, lead[1], 128)[:n]


@pytest.mark.parametrize("Hkv,group,lens", [
    (1, 8, [1]),                                      # one block, 1775 runs of none
    (2, 1, [1700, 3]),                                # runs of no block, records of single blocks
    (1, 3, [40000]),                                  # 1250 records of one head: many chunks, four groups
    (1, 5, [9000, 0, 31, 32, 33]),
    (3, 2, [17 + 29 * i for i in range(33)]),         # a second scan of one sequence
    (8, 4, [(37 * i) % 600 for i in range(100)]),     # four scans, lengths of 0 among them
    (8, 7, [6000 - 371 * i for i in range(16)]),      # records in one chunk of sixteen
    (2, 3, [100 + 31 * i for i in range(150)]),       # in one chunk of eight
    (8, 4, [512, 513, 545, 1056, 1088] + [20] * 75),  # 16, 17, 18, 33 and 34 records of single blocks, some runs of none
    (4, 7, [9000, 3000] + [50 + i for i in range(160)]),  # about 200 and 65 records
])
def test_attention_records(Hkv, group, lens):
    import paper_2412_14363_b200 as resq
    from paper_2412_14363_b200 import kv

    d, Hq, B = 128, Hkv * group, len(lens)
    g = torch.Generator(device="cuda").manual_seed(sum(lens) + group)
    cap = (max(lens) + 31) // 32 * 32
    cache = kv.KvCache(B, Hkv, cap, d)
    cache.data.zero_()
    wq, su = kv.resq_uc_quantize(torch.linalg.qr(torch.randn(d, d, device="cuda", generator=g))[0].contiguous())
    for b, n in enumerate(lens):
        if n:
            k, v = (torch.randn(n, Hkv, d, device="cuda", generator=g).to(torch.bfloat16) for _ in range(2))
            kv.resq_kv_append(cache, k, v, torch.full((n,), b, dtype=torch.int32, device="cuda"),
                              torch.arange(n, dtype=torch.int32, device="cuda"), wq, su)
    q = (2 * torch.randn(B, Hq, d, device="cuda", generator=g)).half()
    out = torch.full((B, Hq, d), float("nan"), device="cuda")
    ws = torch.full_like(kv.attention_workspace(cache, Hq), 0xFF)  # scratch holds anything
    kv.resq_attention_decode(cache, q, torch.tensor(lens, dtype=torch.int32, device="cuda"), out, ws)
    assert resq.resq_device_status() == resq.OK
    for b, n in enumerate(lens):
        if n == 0:
            assert (out[b] == 0).all()
            continue
        K, V = (_dequantize(cache, b, n, which) for which in "kv")
        for h in range(Hkv):
            rows = q[b, h * group:(h + 1) * group].double()
            want = torch.softmax(rows @ K[:, h].T / math.sqrt(d), dim=1) @ V[:, h]
            err = (out[b, h * group:(h + 1) * group].double() - want).abs().amax() / V[:, h].abs().amax()
            assert err < 1e-3, (b, h, float(err))  # the weights times the value scales are halves (2^-11), see test_gpu_kv.py
