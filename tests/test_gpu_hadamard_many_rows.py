"""The Hadamard transform and quantizer for more rows than SMs (256 threads per row, neighbouring coefficients in pairs)
against calls of at most 148 rows (1024 threads per row, coefficients singly; checked against the CPU oracle in
test_gpu_hadamard.py).  Every coefficient goes through the same additions in the same order, so the bits agree."""
import pytest
import torch

import synth
from tests.gpu_util import bf16_to_dev, host

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("T, K, r", [
    (149, 224, 0), (150, 896, 64),          # three index bits, five
    (153, 1536, 0), (149, 1536, 32),        # 12 * 2^7
    (149, 1792, 32), (301, 3584, 448),      # 28 * 2^6 = 3 + 3 bits, a segment border inside a group; 2^7 = 4 + 3
    (150, 3072, 384), (149, 12288, 1536),   # 12 * 2^8, 2^10
    (299, 14336, 0), (149, 14336, 1792), (149, 28672, 3584),
])
def test_many_rows_are_the_rows_one_by_one(T, K, r):
    import paper_2412_14363_b200 as resq
    X = bf16_to_dev(synth.f32_to_bf16_bits(synth.activations(T, K, "t4", seed=700 + T)))
    X[T - 1] = 0
    out = []
    for step in (T, 100):
        x8 = torch.full((T, max(r, 1)), 77, dtype=torch.int8, device="cuda")
        x4 = torch.zeros((T, (K - r) // 2), dtype=torch.uint8, device="cuda")
        x4e = torch.zeros((T, K - r), dtype=torch.int8, device="cuda")
        s8, s4 = (torch.full((T,), float("nan"), device="cuda") for _ in range(2))
        for t in range(0, T, step):
            n = slice(t, min(T, t + step))
            parts = [x[n].clone() for x in (x8, x4, s8, s4, x4e)]  # 16-byte aligned
            resq.resq_hadamard_quantize(X[n].clone(), r, *parts)
            for whole, part in zip((x8, x4, s8, s4, x4e), parts):
                whole[n] = part
        assert resq.resq_device_status() == resq.OK
        out.append([host(x) for x in (x8, x4, x4e, s8, s4)])
    for a, b in zip(*out):
        assert a.tobytes() == b.tobytes()
