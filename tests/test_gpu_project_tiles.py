"""Query projection and key / value append beyond 9216 (d_head = 128) or 4096 (64) head vectors, where a warp takes 16 tokens of one head (or 16 query rows): the
same bytes as calls of a few tokens, which take one warp per vector and are checked against the CPU oracle in test_gpu_kv.py and
test_gpu_kv_d64.py.  Both forms round the same IEEE quotients and sum the same integers, so nothing may differ."""
import numpy as np
import pytest
import torch

import synth
from tests import plans
from tests.gpu_util import bf16_to_dev, dev, host

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("d", [128, 64])
@pytest.mark.parametrize("T, Hq, Hkv, part", [
    (433, 24, 3, "qkv"),      # a last tile of one token, an odd number of KV heads
    (1039, 12, 1, "qkv"),     # fifteen tokens, one KV head
    (1024, 4, 5, "qkv"),      # whole tiles, more key and value tiles than query tiles
    (1237, 11, 0, "q"),       # queries alone, rows not a multiple of 16
    (1231, 0, 5, "kv"),       # keys and values alone
    (9217, 1, 0, "q"),        # one vector more than the other form takes at 128
    (4097, 1, 0, "q"),        # and at 64
    (2400, 16, 16, "qkv"),    # a CTA's warps go through tiles together: three rounds and a few
    (2007, 13, 19, "qkv"),    # two and most of a third, of queries and the last values
    (2200, 0, 18, "kv"),      # two and a few of the last values
])
def test_tiles_write_what_single_vectors_write(d, T, Hq, Hkv, part):
    import paper_2412_14363_b200 as resq
    from paper_2412_14363_b200 import kv
    assert plans.append_together(d, T, Hq, Hkv) == (T >= 2000 and Hkv > 1)
    wq, s_u = kv.resq_uc_quantize(dev(np.ascontiguousarray(synth.haar_orthogonal(d).T.astype(np.float32))))
    seq_ids, positions = dev((np.arange(T) % 3).astype(np.int32)), dev((np.arange(T) // 3).astype(np.int32))
    heads = {}
    for i, n in enumerate(part):
        x = synth.head_vectors(T, Hq if n == "q" else Hkv, d, stream=900 + i, lead=4.0, scale=0.7)
        x[T - 1, -1] = 0.0
        x[17, 0, 3] = np.inf                 # a key: every projected value is NaN
        x[18, 0, d - 1] = np.nan
        x[21, 0, d // 8:] = np.inf           # a value: the whole 4-bit segment, the 8-bit one below
        x[22, 0, :d // 8] = -np.inf
        x[23, 0] = np.nan
        x[24, 0, ::2] = np.inf
        x[24, 0, 1::2] = -np.inf
        x[19, 0] *= 1e-36
        x[20, 0] *= 1e36
        heads[n] = bf16_to_dev(synth.f32_to_bf16_bits(x))
    out = []
    for step in (T, 100):
        cache = kv.KvCache(3, max(Hkv, 1), (T // 3 + 32) // 32 * 32, d)
        cache.data.fill_(7)
        q_out = torch.zeros((T, max(Hq, 1), d), dtype=torch.float16, device="cuda")
        for t in range(0, T, step):
            s = slice(t, min(T, t + step))
            if "q" in part:
                kv.resq_query_project(heads["q"][s], wq, s_u, q_out[s]) if part == "q" else kv.resq_qkv_project_append(
                    cache, heads["q"][s], q_out[s], heads["k"][s], heads["v"][s], seq_ids[s].clone(), positions[s].clone(), wq, s_u)
            else:
                kv.resq_kv_append(cache, heads["k"][s], heads["v"][s], seq_ids[s].clone(), positions[s].clone(), wq, s_u)
        assert resq.resq_device_status() == resq.OK
        out.append((host(q_out).view(np.uint16), host(cache.data)))
    assert (out[0][0] == out[1][0]).all()
    assert (out[0][1] == out[1][1]).all()
