"""Causal attention where there are more tiles of 128 rows than SMs (csrc/kv_prefill.cu): a CTA takes a long and a short tile in
turn, the middle one of an odd number alone; two neighbours together, the last one without its second; one tile each at
d_head = 64.  Against the oracle's fp64 definition on its own codes, on rows drawn over the run, the first and the last among
them.  Tolerances as in test_gpu_kv_prefill.py (1e-3 of the largest value) and test_gpu_kv_d64.py (1e-4)."""
import numpy as np
import pytest
import torch

import synth
from oracle import kv as okv
from tests.gpu_util import bf16_to_dev, dev, host

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("D,prefix,T,Hq,Hkv,tiles", [
    (128, 0, 1660, 12, 4, 39 * 4),    # in turn: groups of three, an odd number of tiles
    (64, 37, 1660, 12, 4, 39 * 4),
    (64, 0, 1000, 32, 8, 32 * 8),     # in turn: every CTA two tiles
    (128, 5, 1200, 32, 32, 10 * 32),  # together, groups of one
    (128, 70, 1000, 35, 7, 40 * 7),   # in turn: groups of five behind a prefix
    (128, 0, 780, 56, 8, 43 * 8),     # together: groups of seven, the last pair's second tile empty
    (64, 0, 1200, 32, 32, 10 * 32),   # one each, more than two rounds
])
def test_runs_of_many_tiles_against_the_oracle(D, prefix, T, Hq, Hkv, tiles):
    import paper_2412_14363_b200 as resq
    from paper_2412_14363_b200 import kv
    g, S = Hq // Hkv, prefix + T
    assert -(-T * g // 128) * Hkv == tiles and tiles > 148
    W_C = np.ascontiguousarray(synth.haar_orthogonal(D).T.astype(np.float32))
    wq, s_u = kv.resq_uc_quantize(dev(W_C))
    cache = kv.KvCache(1, Hkv, (S + 31) // 32 * 32, d_head=D)
    cache.data.fill_(0xFF)  # unwritten positions hold NaN patterns
    k = synth.head_vectors(S, Hkv, D, stream=970, lead=1.0, scale=1.5)
    v = synth.head_vectors(S, Hkv, D, stream=971, lead=4.0, shift=0.3)
    kv.resq_kv_append(cache, bf16_to_dev(synth.f32_to_bf16_bits(k)), bf16_to_dev(synth.f32_to_bf16_bits(v)),
                      dev(np.zeros(S, np.int32)), dev(np.arange(S, dtype=np.int32)), wq, s_u)
    q = synth.head_vectors(T, Hq, D, stream=972, lead=1.0, scale=1.5)
    q16 = torch.empty((T, Hq, D), dtype=torch.float16, device="cuda")
    kv.resq_query_project(bf16_to_dev(synth.f32_to_bf16_bits(q)), wq, s_u, q16)
    out = torch.full((T, Hq, D), float("nan"), dtype=torch.float32, device="cuda")
    kv.resq_attention_prefill(cache, q16, 0, prefix, out)
    assert resq.resq_device_status() == resq.OK
    got = host(out)
    assert np.isfinite(got).all()
    Yk, _, _ = okv.project_int8(k.reshape(-1, D), *okv.quantize_uc(W_C))
    dk = okv.kv_dequantize(okv.kv_quantize(Yk)).reshape(S, Hkv, D)
    dv = okv.kv_dequantize(okv.kv_quantize(v.reshape(-1, D))).reshape(S, Hkv, D)
    rows = np.unique(np.concatenate([[0, 1, T - 2, T - 1], np.random.default_rng(T).integers(0, T, 60)]))
    ref = okv.attention_queries(host(q16)[rows], [[dk[:, h] for h in range(Hkv)]], [[dv[:, h] for h in range(Hkv)]],
                                np.zeros(len(rows), np.int32), (prefix + rows + 1).astype(np.int32), Hq, Hkv)
    for h in range(Hq):
        err = np.abs(got[rows, h] - ref[:, h]).max()
        assert err <= (1e-3 if D == 128 else 1e-4) * np.abs(dv[:, h // g]).max(), (h, err)
