"""Causal attention where there are more tiles of 128 rows than SMs (csrc/kv_prefill.cu): a CTA takes a long and a short tile in
turn, the middle one of an odd number alone; two neighbours together, the last one without its second; one tile each at
d_head = 64.  Then, in every form, scores that grow with the position, so that a row's reference is raised again and again.
Against the oracle's fp64 definition on its own codes, on rows drawn over the run, the first and the last among them.
Tolerances as in test_gpu_kv_prefill.py (1e-3 of the largest value) and test_gpu_kv_d64.py (1e-4)."""
import numpy as np
import pytest
import torch

import synth
from oracle import kv as okv
from tests import plans
from tests.gpu_util import bf16_to_dev, dev, host

pytestmark = pytest.mark.gpu


TURN, TOGETHER, ONE = (2, 0), (2, 1), (1, 0)  # tiles of a CTA, whether they walk together


def _form(D, prefix, T, Hq, Hkv):
    form = plans.prefill(prefix, T, Hq, Hkv, D)
    return form.tiles_per_cta, form.pair


def _check(D, prefix, T, Hq, Hkv, growing):
    """The run's outputs on drawn rows, the first and the last among them, against the oracle."""
    import paper_2412_14363_b200 as resq
    from paper_2412_14363_b200 import kv
    g, S = Hq // Hkv, prefix + T
    W_C = np.ascontiguousarray(synth.haar_orthogonal(D).T.astype(np.float32))
    wq, s_u = kv.resq_uc_quantize(dev(W_C))
    cache = kv.KvCache(1, Hkv, (S + 31) // 32 * 32, d_head=D)
    cache.data.fill_(0xFF)  # unwritten positions hold NaN patterns
    k = synth.head_vectors(S, Hkv, D, stream=970, lead=1.0, scale=1.0 if growing else 1.5)
    if growing:
        k = synth.to_bf16_values(k * (0.2 + 6.0 * np.arange(S) / S)[:, None, None].astype(np.float32))
    v = synth.head_vectors(S, Hkv, D, stream=971, lead=4.0, shift=0.3)
    kv.resq_kv_append(cache, bf16_to_dev(synth.f32_to_bf16_bits(k)), bf16_to_dev(synth.f32_to_bf16_bits(v)),
                      dev(np.zeros(S, np.int32)), dev(np.arange(S, dtype=np.int32)), wq, s_u)
    q = synth.head_vectors(T, Hq, D, stream=972, lead=1.0, scale=2.0 if growing else 1.5)
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


@pytest.mark.parametrize("D,prefix,T,Hq,Hkv,tiles,form", [
    (128, 0, 1660, 12, 4, 39 * 4, TURN),        # groups of three, an odd number of tiles
    (64, 37, 1660, 12, 4, 39 * 4, TURN),
    (64, 0, 1000, 32, 8, 32 * 8, TURN),         # every CTA two tiles
    (128, 5, 1200, 32, 32, 10 * 32, TOGETHER),  # groups of one
    (128, 70, 1000, 35, 7, 40 * 7, TURN),       # groups of five behind a prefix
    (128, 1400, 700, 28, 7, 22 * 7, TOGETHER),  # the same behind a longer one
    (128, 0, 780, 56, 8, 43 * 8, TOGETHER),     # groups of seven, the last pair's second tile empty
    (64, 0, 1200, 32, 32, 10 * 32, ONE),        # one each, more than two rounds
])
def test_runs_of_many_tiles_against_the_oracle(D, prefix, T, Hq, Hkv, tiles, form):
    assert -(-T * Hq // Hkv // 128) * Hkv == tiles and tiles > 148
    assert _form(D, prefix, T, Hq, Hkv) == form
    _check(D, prefix, T, Hq, Hkv, growing=False)


@pytest.mark.parametrize("D,prefix,T,Hq,Hkv,form,splits", [
    (128, 3, 1200, 32, 32, TOGETHER, 1), (128, 1400, 700, 28, 7, TOGETHER, 1), (128, 0, 1660, 12, 4, TURN, 1),
    (64, 0, 400, 8, 2, ONE, 1), (64, 900, 60, 4, 4, ONE, 2), (64, 200, 1900, 1, 1, ONE, 8), (64, 0, 1000, 32, 8, TURN, 1),
    (64, 150, 1660, 12, 4, TURN, 1), (64, 0, 1200, 32, 32, ONE, 1),
])
def test_scores_that_keep_growing(D, prefix, T, Hq, Hkv, form, splits):
    assert _form(D, prefix, T, Hq, Hkv) == form
    assert plans.prefill(prefix, T, Hq, Hkv, D).splits == splits
    _check(D, prefix, T, Hq, Hkv, growing=True)
