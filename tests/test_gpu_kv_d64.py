"""GPU parity of the attention-block path at d_head = 64 (the Llama-3.2-1B head width: 8 coefficients in 8 bits, 56
in 4; Section 4.3, Eq. 8; Section 5.1) through the C ABI against the CPU oracle: U_C codes, the projected
half-precision query and every cache byte bit for bit; attention (single-query, many-query and the causal run of new
tokens) within 1e-4 of the largest dequantized value magnitude -- at this width every step after the integer product
is fp32, so only summation order and the exponential's last bits separate the two sides."""
import numpy as np
import pytest
import torch

import synth
from oracle import kv as okv
from tests import plans
from tests.gpu_util import bf16_to_dev, dev, host

pytestmark = pytest.mark.gpu
D, R8, B4 = 64, 8, 28
HALF, BLOCK_BYTES = 32 * (R8 + B4 + 16), 2 * 32 * (R8 + B4 + 16)


@pytest.fixture(scope="module")
def resq():
    import paper_2412_14363_b200 as m
    return m


@pytest.fixture(scope="module")
def kv():
    from paper_2412_14363_b200 import kv as m
    return m


@pytest.fixture(scope="module")
def uc(kv):
    W_C = np.ascontiguousarray(synth.haar_orthogonal(D).T.astype(np.float32))
    wq, s_u = kv.resq_uc_quantize(dev(W_C))
    return W_C, wq, s_u


def _record(image, which, b, h, pos):
    """(c8 [8], c4 [28], meta fp32 [4]) of one head vector from a cache image [n_seqs][H][blocks][BLOCK_BYTES]."""
    blk, p = image[b, h, pos // 32], pos % 32
    o = 0 if which == "k" else HALF
    return (blk[o + R8 * p: o + R8 * p + R8], blk[o + 32 * R8 + B4 * p: o + 32 * R8 + B4 * p + B4],
            blk[o + 32 * (R8 + B4) + 16 * p: o + 32 * (R8 + B4) + 16 * p + 16].copy().view(np.float32))


def _oracle_records(k, v, W_C):
    Yk, _, _ = okv.project_int8(k.reshape(-1, D), *okv.quantize_uc(W_C))
    return okv.kv_quantize(Yk), okv.kv_quantize(v.reshape(-1, D))


def test_uc_quantize_and_query_project_bit_exact(resq, kv, uc):
    W_C, wq, s_u = uc
    owq, os_u = okv.quantize_uc(W_C)
    assert (host(wq) == owq).all() and (host(s_u).view(np.uint32) == os_u.view(np.uint32)).all()
    T, H = 37, 32
    q = synth.head_vectors(T, H, D, stream=910, lead=1.0, scale=3.0)
    q[0, 0, :] = 0.0
    q_out = torch.empty((T, H, D), dtype=torch.float16, device="cuda")
    kv.resq_query_project(bf16_to_dev(synth.f32_to_bf16_bits(q)), wq, s_u, q_out)
    assert resq.resq_device_status() == resq.OK
    Y, _, _ = okv.project_int8(q.reshape(-1, D), owq, os_u)
    assert (host(q_out).view(np.uint16) == okv.query_fp16(Y).reshape(T, H, D).view(np.uint16)).all()


@pytest.mark.parametrize("T,H", [(70, 8), (5, 2)])
def test_kv_append_bit_exact(resq, kv, uc, T, H):
    W_C, wq, s_u = uc
    k = synth.head_vectors(T, H, D, stream=920 + T, lead=1.0, scale=2.0)
    v = synth.head_vectors(T, H, D, stream=940 + T, lead=4.0, shift=0.5)
    v[1, 0, :R8] = v[1, 0, 0]                  # a constant 8-bit segment: s = 0, codes 0
    cache = kv.KvCache(2, H, 128, d_head=D)
    assert cache.nbytes == 2 * H * 4 * BLOCK_BYTES
    cache.data.fill_(0xEE)
    seq_ids = np.ones(T, np.int32)
    positions = np.arange(3, 3 + T, dtype=np.int32)
    seq_ids[-1], positions[-1] = 5, 0          # out of range: skipped and reported
    kv.resq_kv_append(cache, bf16_to_dev(synth.f32_to_bf16_bits(k)), bf16_to_dev(synth.f32_to_bf16_bits(v)),
                      dev(seq_ids), dev(positions), wq, s_u)
    assert resq.resq_device_status() == kv.ERR_INDEX
    image = host(cache.data).reshape(2, H, 4, BLOCK_BYTES)
    hk, hv = _oracle_records(k, v, W_C)
    for t in range(T - 1):
        for h in range(H):
            row = t * H + h
            for which, rec in (("k", hk), ("v", hv)):
                c8, c4, meta = _record(image, which, 1, h, positions[t])
                assert (c8 == rec.c8[row]).all() and (c4 == rec.c4[row]).all(), (which, t, h)
                assert (meta.view(np.uint32) == rec.meta[row].view(np.uint32)).all(), (which, t, h)
    assert (image[0] == 0xEE).all()


def test_attention_three_forms_against_the_oracle(resq, kv, uc):
    """Llama-3.2-1B head geometry (32 query / 8 KV heads x 64): single-query over two sequences, many-query with
    scattered prefixes, and the causal run of new tokens, each against the oracle's fp64 definition; the fused
    project-and-append call fills one of the sequences."""
    W_C, wq, s_u = uc
    Hq, Hkv, S0, S1 = 32, 8, 150, 41
    cache = kv.KvCache(2, Hkv, 160, d_head=D)
    cache.data.fill_(0xFF)
    K_hat, V_hat = [None, None], [None, None]
    for b, n in ((0, S0), (1, S1)):
        k = synth.head_vectors(n, Hkv, D, stream=950 + b, lead=1.0, scale=1.5)
        v = synth.head_vectors(n, Hkv, D, stream=960 + b, lead=4.0, shift=0.3)
        args = (bf16_to_dev(synth.f32_to_bf16_bits(k)), bf16_to_dev(synth.f32_to_bf16_bits(v)), dev(np.full(n, b, np.int32)),
                dev(np.arange(n, dtype=np.int32)), wq, s_u)
        if b == 0:
            kv.resq_kv_append(cache, *args)
        else:
            qd = synth.head_vectors(n, Hq, D, stream=969, lead=1.0)
            qo = torch.empty((n, Hq, D), dtype=torch.float16, device="cuda")
            kv.resq_qkv_project_append(cache, bf16_to_dev(synth.f32_to_bf16_bits(qd)), qo, *args)
        hk, hv = _oracle_records(k, v, W_C)
        dk, dv = okv.kv_dequantize(hk).reshape(n, Hkv, D), okv.kv_dequantize(hv).reshape(n, Hkv, D)
        K_hat[b], V_hat[b] = [dk[:, h] for h in range(Hkv)], [dv[:, h] for h in range(Hkv)]
    vmax = max(np.abs(v).max() for b in range(2) for v in V_hat[b])
    T = 60
    q = synth.head_vectors(T, Hq, D, stream=970, lead=1.0, scale=1.5)
    q16 = torch.empty((T, Hq, D), dtype=torch.float16, device="cuda")
    kv.resq_query_project(bf16_to_dev(synth.f32_to_bf16_bits(q)), wq, s_u, q16)
    hq16 = host(q16)
    # causal run: the last T tokens of sequence 0
    out = torch.full((T, Hq, D), float("nan"), dtype=torch.float32, device="cuda")
    kv.resq_attention_prefill(cache, q16, 0, S0 - T, out)
    ref = okv.attention_queries(hq16, K_hat, V_hat, np.zeros(T, np.int32), np.arange(S0 - T + 1, S0 + 1), Hq, Hkv)
    assert np.abs(host(out) - ref).max() <= 1e-4 * vmax
    # many-query: scattered (sequence, prefix) pairs, one empty
    q_seq = (np.arange(T) % 2).astype(np.int32)
    q_len = np.where(q_seq == 0, (np.arange(T) * 7) % (S0 + 1), (np.arange(T) * 5) % (S1 + 1)).astype(np.int32)
    q_len[3] = 0
    kv.resq_attention_queries(cache, q16, dev(q_seq), dev(q_len), out)
    ref = okv.attention_queries(hq16, K_hat, V_hat, q_seq, q_len, Hq, Hkv)
    got = host(out)
    assert np.abs(got - ref).max() <= 1e-4 * vmax and (got[3] == 0).all()
    # single-query: one row per sequence
    one = torch.empty((2, Hq, D), dtype=torch.float32, device="cuda")
    kv.resq_attention_decode(cache, q16[:2].contiguous(), dev(np.array([S0, S1], np.int32)), one,
                             kv.attention_workspace(cache, Hq))
    ref = okv.attention_decode(hq16[:2], K_hat, V_hat, [S0, S1], Hq, Hkv)
    assert np.abs(host(one) - ref).max() <= 1e-4 * vmax
    assert resq.resq_device_status() == resq.OK


@pytest.mark.parametrize("Hq,Hkv,lens,T", [
    (8, 8, [1, 33, 1029, 2050], 1),     # one head per group; few CTAs: the positions are split over a cluster
    (16, 2, [705, 64, 31], 43),         # eight heads per group, a tile of 64 rows ends inside a token's group
    (12, 4, [130], 130),                # three heads per group: rows of a token on both sides of a tile edge
    (64, 8, [385] * 5, 9),              # no split: 40 (sequence, head) pairs
])
def test_attention_tile_edges(resq, kv, uc, Hq, Hkv, lens, T):
    """Single-query over all sequences, the causal run of the last T positions of the first, and the same rows as many
    queries, on caches whose unwritten bytes are 0xFF.  |out - oracle| <= 2e-5 max|v|: everything is fp32, a score of at most 40 in log2 units carries 2^-22 of itself."""
    W_C, wq, s_u = uc
    B, cap = len(lens), (max(lens) + 31) // 32 * 32 + 32
    cache = kv.KvCache(B, Hkv, cap, d_head=D)
    cache.data.fill_(0xFF)
    K_hat, V_hat = [], []
    for b, n in enumerate(lens):
        k = synth.head_vectors(n, Hkv, D, stream=1100 + b, lead=1.0, scale=1.5)
        v = synth.head_vectors(n, Hkv, D, stream=1200 + b, lead=4.0, shift=0.3, scale=10.0 ** (2 * b - 2))
        kv.resq_kv_append(cache, bf16_to_dev(synth.f32_to_bf16_bits(k)), bf16_to_dev(synth.f32_to_bf16_bits(v)),
                          dev(np.full(n, b, np.int32)), dev(np.arange(n, dtype=np.int32)), wq, s_u)
        hk, hv = _oracle_records(k, v, W_C)
        dk, dv = okv.kv_dequantize(hk).reshape(n, Hkv, D), okv.kv_dequantize(hv).reshape(n, Hkv, D)
        K_hat.append([dk[:, h] for h in range(Hkv)])
        V_hat.append([dv[:, h] for h in range(Hkv)])
    vmax = [max(np.abs(x).max() for x in V) for V in V_hat]
    n_q = max(T, B)
    q16 = torch.empty((n_q, Hq, D), dtype=torch.float16, device="cuda")
    kv.resq_query_project(bf16_to_dev(synth.f32_to_bf16_bits(synth.head_vectors(n_q, Hq, D, stream=1300, lead=1.0, scale=1.5))),
                          wq, s_u, q16)
    hq16 = host(q16)
    one = torch.full((B, Hq, D), float("nan"), dtype=torch.float32, device="cuda")
    kv.resq_attention_decode(cache, q16[:B].contiguous(), dev(np.array(lens, np.int32)), one, kv.attention_workspace(cache, Hq))
    ref = okv.attention_decode(hq16[:B], K_hat, V_hat, lens, Hq, Hkv)
    for b in range(B):
        assert np.abs(host(one)[b] - ref[b]).max() <= 2e-5 * vmax[b], b
    pos0 = lens[0] - T
    q = q16[:T].contiguous()
    ref = okv.attention_queries(hq16[:T], K_hat, V_hat, np.zeros(T, np.int32), np.arange(pos0 + 1, pos0 + T + 1), Hq, Hkv)
    run = torch.full((T, Hq, D), float("nan"), dtype=torch.float32, device="cuda")
    kv.resq_attention_prefill(cache, q, 0, pos0, run)
    assert np.abs(host(run) - ref).max() <= 2e-5 * vmax[0]
    many = torch.full((T, Hq, D), float("nan"), dtype=torch.float32, device="cuda")
    kv.resq_attention_queries(cache, q, dev(np.zeros(T, np.int32)), dev(np.arange(pos0 + 1, pos0 + T + 1, dtype=np.int32)), many)
    assert np.abs(host(many) - ref).max() <= 2e-5 * vmax[0]
    assert resq.resq_device_status() == resq.OK


@pytest.mark.parametrize("outlier", [5, -1])
@pytest.mark.parametrize("k", [20, 28])
def test_attention_beside_a_far_larger_value_scale(resq, kv, uc, outlier, k):
    """One position's values are 2^k times the others' and its key is so far from every query that its weight is below 2^-100
    (outlier = 5), or it is the run's last token, which only the last row attends: the outputs keep the accuracy of a cache
    without it, 2e-5 of the largest other value (the bound of test_attention_tile_edges)."""
    W_C, wq, s_u = uc
    Hq, Hkv, S, T = 8, 2, 140, 40
    K = synth.head_vectors(S, Hkv, D, stream=1400, lead=1.0, scale=1.5)
    v = synth.head_vectors(S, Hkv, D, stream=1401, lead=4.0, shift=0.3)
    q = synth.head_vectors(T, Hq, D, stream=1402, lead=1.0, scale=0.5)
    common = np.where(np.arange(D) % 2, 4.0, -4.0).astype(np.float32)
    q = synth.to_bf16_values(q + common)
    K[outlier] = synth.to_bf16_values(-2.0 * common)      # score about -2 * 16 * 64 / 8 = -256
    v[outlier] = v[outlier] * np.float32(2.0 ** k)
    cache = kv.KvCache(1, Hkv, 160, d_head=D)
    cache.data.fill_(0xFF)
    kv.resq_kv_append(cache, bf16_to_dev(synth.f32_to_bf16_bits(K)), bf16_to_dev(synth.f32_to_bf16_bits(v)),
                      dev(np.zeros(S, np.int32)), dev(np.arange(S, dtype=np.int32)), wq, s_u)
    hk, hv = _oracle_records(K, v, W_C)
    dk, dv = okv.kv_dequantize(hk).reshape(S, Hkv, D), okv.kv_dequantize(hv).reshape(S, Hkv, D)
    K_hat, V_hat = [dk[:, h] for h in range(Hkv)], [dv[:, h] for h in range(Hkv)]
    others = np.arange(S) != outlier % S
    vmax = max(np.abs(x[others]).max() for x in V_hat)
    q16 = torch.empty((T, Hq, D), dtype=torch.float16, device="cuda")
    kv.resq_query_project(bf16_to_dev(synth.f32_to_bf16_bits(q)), wq, s_u, q16)
    lens = np.arange(S - T + 1, S + 1)
    ref = okv.attention_queries(host(q16), [K_hat], [V_hat], np.zeros(T, np.int32), lens, Hq, Hkv)
    run = torch.full((T, Hq, D), float("nan"), dtype=torch.float32, device="cuda")
    kv.resq_attention_prefill(cache, q16, 0, S - T, run)
    assert np.abs(host(run) - ref).max() <= 2e-5 * vmax
    many = torch.full((T, Hq, D), float("nan"), dtype=torch.float32, device="cuda")
    kv.resq_attention_queries(cache, q16, dev(np.zeros(T, np.int32)), dev(lens.astype(np.int32)), many)
    assert np.abs(host(many) - ref).max() <= 2e-5 * vmax
    assert resq.resq_device_status() == resq.OK


@pytest.mark.parametrize("rows,Hq,Hkv,longest,warps,pack", [
    (148, 4, 1, 100, 12, 0),    # an item for every SM
    (83, 16, 2, 130, 12, 1),    # 166 items: a CTA of twelve warps takes one, or twelve short ones; the last block has ten
    (149, 15, 5, 100, 12, 1),   # 745: short is up to two steps; blocks span three rows
    (445, 4, 2, 300, 4, 1),     # 890 items: one CTA of four warps each, or four short ones together
    (891, 8, 1, 150, 4, 1),     # blocks of four rows, the last of three, lengths on both sides of short
    (300, 24, 3, 40, 4, 1),     # all short, a row's heads in two blocks
    (889, 8, 8, 60, 4, 2),      # 7112 items: four to a CTA whatever the lengths
])
def test_attention_of_many_short_rows(resq, kv, uc, rows, Hq, Hkv, longest, warps, pack):
    """The many-query form where it hands a CTA several items, or one, by their lengths; empty prefixes, a length and a sequence
    out of range among them.  The bound of test_attention_tile_edges."""
    form = plans.rows64(rows, Hkv, (longest + 31) // 32 * 32)
    assert (form.warps, form.pack) == (warps, pack)
    W_C, wq, s_u = uc
    S = (longest + 31) // 32 * 32
    cache = kv.KvCache(2, Hkv, S, d_head=D)
    cache.data.fill_(0xFF)
    K_hat, V_hat = [], []
    for b in range(2):
        k = synth.head_vectors(S, Hkv, D, stream=1420 + b, lead=1.0, scale=1.5)
        v = synth.head_vectors(S, Hkv, D, stream=1430 + b, lead=4.0, shift=0.3)
        kv.resq_kv_append(cache, bf16_to_dev(synth.f32_to_bf16_bits(k)), bf16_to_dev(synth.f32_to_bf16_bits(v)),
                          dev(np.full(S, b, np.int32)), dev(np.arange(S, dtype=np.int32)), wq, s_u)
        hk, hv = _oracle_records(k, v, W_C)
        dk, dv = okv.kv_dequantize(hk).reshape(S, Hkv, D), okv.kv_dequantize(hv).reshape(S, Hkv, D)
        K_hat.append([dk[:, h] for h in range(Hkv)])
        V_hat.append([dv[:, h] for h in range(Hkv)])
    vmax = max(np.abs(x).max() for V in V_hat for x in V)
    q16 = torch.empty((rows, Hq, D), dtype=torch.float16, device="cuda")
    kv.resq_query_project(bf16_to_dev(synth.f32_to_bf16_bits(synth.head_vectors(rows, Hq, D, stream=1440, lead=1.0, scale=1.5))),
                          wq, s_u, q16)
    rng = np.random.default_rng(rows)
    q_seq = rng.integers(0, 2, rows).astype(np.int32)
    q_len = np.where(rng.random(rows) < 0.1, longest, rng.integers(0, 34, rows)).astype(np.int32)
    out = torch.full((rows, Hq, D), float("nan"), dtype=torch.float32, device="cuda")
    kv.resq_attention_queries(cache, q16, dev(q_seq), dev(q_len), out)
    assert resq.resq_device_status() == resq.OK
    ref = okv.attention_queries(host(q16), K_hat, V_hat, q_seq, q_len, Hq, Hkv)
    assert np.abs(host(out) - ref).max() <= 2e-5 * vmax
    q_len[7], q_seq[8] = S + 5, 9        # clamped to the capacity, unspecified; both reported
    again = torch.full((rows, Hq, D), float("nan"), dtype=torch.float32, device="cuda")
    kv.resq_attention_queries(cache, q16, dev(q_seq), dev(q_len), again)
    assert resq.resq_device_status() == kv.ERR_INDEX
    ref[7] = okv.attention_queries(host(q16[7:8]), K_hat, V_hat, q_seq[7:8], np.array([S]), Hq, Hkv)[0]
    same = np.arange(rows) != 8
    assert np.abs(host(again)[same] - ref[same]).max() <= 2e-5 * vmax
