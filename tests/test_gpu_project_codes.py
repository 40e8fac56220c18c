"""Projected rows of few tokens, summed and quantized in one kernel: the codes and scales of the coefficients that resq_project gives, at the edges
of the chunks that a CTA of the row's cluster takes, for all-zero rows and rows of one value."""
import pytest
import torch


@pytest.mark.gpu
@pytest.mark.parametrize("asym", [False, True])
@pytest.mark.parametrize("T,K,r", [(1, 512, 64), (3, 14336, 1792), (1, 1056, 32), (8, 2080, 0), (17, 4096, 512), (64, 1024, 992), (33, 8192, 1024),
                                   (2, 16416, 2048), (5, 640, 320)])
def test_codes_of_projected_rows(T, K, r, asym):
    import paper_2412_14363_b200 as resq

    g = torch.Generator(device="cuda").manual_seed(T + K)
    X = torch.randn(T, K, device="cuda", generator=g).to(torch.bfloat16)
    P = (torch.randn(K, K, device="cuda", generator=g) / K ** 0.5).to(torch.bfloat16)
    if T > 2:
        X[1] = 0
        X[2], P[5] = 0, 0.5
        X[2, 5] = 3.0  # a row of one value
    # the workspace of a layer holds the projected rows and the partial sums behind them
    desc = resq.layer_desc(K, 8, r)
    ws = (resq.alloc_workspace_asym if asym else resq.alloc_workspace)(desc, T, True, True)
    C = torch.empty((T, K), dtype=torch.float32, device="cuda")
    resq.resq_project(X, P, C, torch.empty(int(resq.lib.resq_project_workspace_bytes()), dtype=torch.uint8, device="cuda"))
    z = lambda shape, dt: torch.full(shape if isinstance(shape, tuple) else (shape,), 99, dtype=dt, device="cuda")
    s8, s4, z8, z4 = (z(T, torch.float32) for _ in range(4))
    it = torch.uint8 if asym else torch.int8
    q8, q4, q4e = z((T, r), it) if r else None, z((T, (K - r) // 2), torch.uint8), z((T, K - r), it)
    if asym:
        resq.resq_project_quantize_asym(X, P, r, q8, q4, s8, s4, z8, z4, q4e, workspace=ws)
    else:
        resq.resq_project_quantize(X, P, r, q8, q4, s8, s4, q4e, workspace=ws)
    assert resq.resq_device_status() == resq.OK
    for seg, q, s, zp, top in ((C[:, :r], q8, s8, z8, 255 if asym else 127), (C[:, r:], q4e, s4, z4, 15 if asym else 7)):
        if seg.shape[1] == 0:
            assert (s == 0).all() and (not asym or (zp == 0).all())
            continue
        lo = seg.amin(1) if asym else torch.zeros(T, device="cuda")
        # fp32 throughout, the divisor on the device too: the definition's own roundings
        want_s = (seg.amax(1) - lo if asym else seg.abs().amax(1)) / torch.full((T,), float(top), device="cuda")
        assert torch.equal(s, want_s)
        if asym:
            assert torch.equal(zp, lo)
        want = torch.round((seg - lo[:, None]) / want_s[:, None]) if asym else torch.round(seg / want_s[:, None])
        want = torch.where(want_s[:, None] > 0, want, torch.zeros_like(want))
        assert torch.equal(q.float(), want)
    lohi = q4e.to(torch.int16) & 15
    assert torch.equal(q4.to(torch.int16), lohi[:, ::2] | lohi[:, 1::2] << 4)


@pytest.mark.gpu
@pytest.mark.parametrize("T,K", [(65, 264), (300, 1024), (1300, 4096), (257, 2056)])
def test_projected_rows_anywhere(T, K):
    """The same coefficients on 32 bytes (stores of 32) and 16 behind (stores of 16), and nothing behind the last row."""
    import paper_2412_14363_b200 as resq

    g = torch.Generator(device="cuda").manual_seed(T + K)
    X = torch.randn(T, K, device="cuda", generator=g).to(torch.bfloat16)
    P = (torch.randn(K, K, device="cuda", generator=g) / K ** 0.5).to(torch.bfloat16)
    ws = torch.empty(int(resq.lib.resq_project_workspace_bytes()), dtype=torch.uint8, device="cuda")
    outs = []
    for skip in (0, 4):
        buf = torch.full((skip + (T + 1) * K,), 9.0, device="cuda")
        C = buf[skip:].view(T + 1, K)
        resq.resq_project(X, P, C[:T], ws)
        assert resq.resq_device_status() == resq.OK
        assert (C[T] == 9).all() and (buf[:skip] == 9).all()
        outs.append(C[:T])
    assert torch.equal(*outs)
    want = X.double() @ P.double()
    size = X.double().abs() @ P.double().abs()
    assert ((outs[0].double() - want).abs() <= K * 2.0 ** -23 * size).all()  # fp32 sums of exact products


@pytest.mark.gpu
@pytest.mark.parametrize("T,K,r", [(1000, 16416, 2048), (700, 28672, 0)])
def test_many_wide_rows(T, K, r):
    """Rows too wide for two stages, more of them than CTAs fit: the codes of the same rows a hundred at a time."""
    import paper_2412_14363_b200 as resq

    g = torch.Generator(device="cuda").manual_seed(K)
    X = torch.randn(T, K, device="cuda", generator=g).to(torch.bfloat16)

    def run(X):
        n = X.shape[0]
        z = lambda shape, dt: torch.full(shape, 77, dtype=dt, device="cuda")
        o = [z((n, r), torch.int8) if r else None, z((n, (K - r) // 2), torch.uint8), z((n,), torch.float32), z((n,), torch.float32),
             z((n, K - r), torch.int8)]
        resq.resq_project_quantize(X, None, r, *o)
        assert resq.resq_device_status() == resq.OK
        return [t for t in o if t is not None]

    parts = [run(X[i:i + 100]) for i in range(0, T, 100)]
    for i, got in enumerate(run(X)):
        assert torch.equal(got, torch.cat([p[i] for p in parts]))
