"""A causal run's rows do not depend on the tokens after them, whatever those hold: the last token's key and value are NaN or
infinite (what a padded batch can leave behind a prompt), and every earlier row equals, bit for bit, the run whose last
token is zero."""
import numpy as np
import pytest
import torch

import synth
from tests.gpu_util import bf16_to_dev, dev, host

pytestmark = pytest.mark.gpu


def _run(resq, kv, d, prefix, T, Hq, Hkv, last):
    S = prefix + T
    wq, s_u = kv.resq_uc_quantize(dev(np.ascontiguousarray(synth.haar_orthogonal(d).T.astype(np.float32))))
    cache = kv.KvCache(1, Hkv, (S + 31) // 32 * 32, d_head=d)
    cache.data.fill_(0xFF)
    k = bf16_to_dev(synth.f32_to_bf16_bits(synth.head_vectors(S, Hkv, d, stream=1500, lead=1.0, scale=1.5)))
    v = bf16_to_dev(synth.f32_to_bf16_bits(synth.head_vectors(S, Hkv, d, stream=1501, lead=4.0, shift=0.3)))
    k[-1] = v[-1] = 0.0
    if last == "nan":
        k[-1] = v[-1] = float("nan")
    elif last == "inf":
        k[-1, :, 3] = v[-1, :, 1] = float("inf")  # one coefficient of the 8-bit segment
        v[-1, :, d - 2] = -float("inf")           # and one of the 4-bit segment
    kv.resq_kv_append(cache, k, v, dev(np.zeros(S, np.int32)), dev(np.arange(S, dtype=np.int32)), wq, s_u)
    q16 = torch.empty((T, Hq, d), dtype=torch.float16, device="cuda")
    kv.resq_query_project(bf16_to_dev(synth.f32_to_bf16_bits(synth.head_vectors(T, Hq, d, stream=1502, lead=1.0, scale=1.5))),
                          wq, s_u, q16)
    out = torch.zeros((T, Hq, d), dtype=torch.float32, device="cuda")
    kv.resq_attention_prefill(cache, q16, 0, prefix, out)
    assert resq.resq_device_status() == resq.OK
    return host(out)


@pytest.mark.parametrize("last", ["nan", "inf"])
@pytest.mark.parametrize("d,prefix,T,Hq,Hkv", [
    (128, 0, 37, 8, 2),      # one tile of rows per CTA
    (128, 1, 600, 32, 8),    # two
    (128, 2000, 40, 8, 2),   # the steps split over a cluster
    (64, 0, 37, 8, 2),
    (64, 100, 300, 12, 2),   # rows of a token on both sides of a tile edge
    (64, 2000, 40, 8, 2),    # the steps split over a cluster
])
def test_rows_do_not_see_a_later_token(d, prefix, T, Hq, Hkv, last):
    import paper_2412_14363_b200 as resq
    from paper_2412_14363_b200 import kv
    ref = _run(resq, kv, d, prefix, T, Hq, Hkv, "zero")
    got = _run(resq, kv, d, prefix, T, Hq, Hkv, last)
    assert np.isfinite(ref).all()
    assert (got[:-1].view(np.uint32) == ref[:-1].view(np.uint32)).all()
    assert not np.isfinite(got[-1]).any()  # the row that does see it
