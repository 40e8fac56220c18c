"""How far causal attention at d_head = 64 is from 64 bits on the cache's own codes: its softmax weights and sums are to keep fp32's
precision (csrc/kv_prefill.cu).  u = 2^-24 is fp32's unit roundoff."""
import pytest
import torch

pytestmark = pytest.mark.gpu
D = 64


def _cached(cache, S, Hkv):
    """Keys and values of sequence 0 in fp64, from the bytes of the cache (resq_kv.h)."""
    half = 32 * 8 + 32 * 28 + 512
    raw = cache.data.view(Hkv, cache.capacity // 32, 2, half)
    out = []
    for h in range(2):
        x = raw[:, :, h]
        c8 = x[..., :256].reshape(Hkv, -1, 8).double()
        w = x[..., 256:1152].reshape(Hkv, -1, 28)
        c4 = torch.stack([w & 15, w >> 4], -1).reshape(Hkv, -1, 56).double()
        m = x[..., 1152:].contiguous().view(torch.float32).reshape(Hkv, -1, 4).double()
        out.append(torch.cat([c8 * m[..., 0:1] + m[..., 1:2], c4 * m[..., 2:3] + m[..., 3:4]], -1)[:, :S])
    return out


@pytest.mark.parametrize("Hq,Hkv,T,prefix", [(8, 2, 300, 0), (8, 2, 200, 4000), (32, 8, 1000, 0)])
@pytest.mark.parametrize("mean", [0.0, 1.0, 100.0])
def test_error_against_64_bits(Hq, Hkv, T, prefix, mean):
    """Values with and without a common mean.  With one, the outputs are about as large as the values: the error is below 2 u, and no
    bias of u / 2 or more shows (a sum that truncates has one).  Without, the outputs are a few times smaller than what is summed: 5 u."""
    import paper_2412_14363_b200 as resq
    from paper_2412_14363_b200 import kv
    S, g = prefix + T, Hq // Hkv
    gen = torch.Generator().manual_seed(11 + T)
    normal = lambda *shape: torch.randn(*shape, generator=gen).cuda()
    wq, s_u = kv.resq_uc_quantize(torch.linalg.qr(normal(D, D))[0].contiguous())
    cache = kv.KvCache(1, Hkv, (S + 31) // 32 * 32, D)
    cache.data.zero_()
    kv.resq_kv_append(cache, normal(S, Hkv, D).bfloat16(), (normal(S, Hkv, D) + mean).bfloat16(), torch.zeros(S, dtype=torch.int32, device="cuda"),
                      torch.arange(S, dtype=torch.int32, device="cuda"), wq, s_u)
    q16 = (1.5 * normal(T, Hq, D)).half()
    out = torch.empty((T, Hq, D), dtype=torch.float32, device="cuda")
    kv.resq_attention_prefill(cache, q16, 0, prefix, out)
    assert resq.resq_device_status() == resq.OK
    K, V = _cached(cache, S, Hkv)
    hidden = torch.arange(S, device="cuda")[None] > torch.arange(prefix, S, device="cuda")[:, None]
    ref = torch.empty((T, Hq, D), dtype=torch.float64, device="cuda")
    for h in range(Hq):
        scores = (q16[:, h].double() @ K[h // g].T / D ** 0.5).masked_fill(hidden, float("-inf"))
        ref[:, h] = torch.softmax(scores, -1) @ V[h // g]
    diff, u = out.double() - ref, 2.0 ** -24
    error, bias = float(diff.norm() / ref.norm()), float(diff.mean() / ref.abs().mean())
    print(f"error {error / u:.2f} u, bias {bias / u:.3f} u")
    if mean:
        assert error < 2 * u and abs(bias) < u / 2
    else:
        assert error < 5 * u
