"""Bilinear upsampling of a dense grid in 16-byte pieces (and, beside it, of token
rows that are no whole pieces), bit-exact against the oracle: grids of one row,
one column and one token, widths around the step of a CTA's warps."""
import numpy as np
import pytest

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("dtype,C", [("bf16", 2), ("bf16", 3), ("bf16", 8), ("bf16", 10),
                                     ("bf16", 16), ("f32", 1), ("f32", 5)])
@pytest.mark.parametrize("gh,gw", [(1, 1), (1, 7), (6, 1), (2, 2), (9, 17), (8, 33)])
def test_bilinear_pieces(gh, gw, dtype, C):
    import torch
    import oracle
    import paper_2608_17995_gb300 as av
    from paper_2608_17995_gb300.pipeline import to_device, to_numpy
    av.build()
    B, M = 2, gh * gw
    k = max(1, M // 3)
    rng = np.random.default_rng(M * 100 + C)
    A, V = rng.random((2, B, M)).astype(np.float32)
    _, mask, off = oracle.topk(oracle.fuse(A, V, 0.5), k)
    lat = rng.standard_normal((B, M, C * 4)).astype(np.float32)
    if dtype == "bf16":
        lat = (lat.view(np.uint32) >> 16).astype(np.uint16)
    want = oracle.selective_upsample(lat, gh, gw, mask, mode="bilinear")
    n = M + 3 * k
    i32 = dict(dtype=torch.int32, device="cuda")
    tdt = torch.bfloat16 if dtype == "bf16" else torch.float32

    def outputs():
        return (torch.zeros(B, n, C * 4, dtype=tdt, device="cuda"), torch.zeros(B, n, 2, **i32),
                torch.zeros(B, n, **i32), torch.zeros(B, n, **i32),
                torch.zeros(B, n, dtype=torch.int8, device="cuda"))

    sel, o = torch.zeros(B, k, **i32), torch.zeros(B, M, **i32)
    m = torch.zeros(B, M, dtype=torch.uint8, device="cuda")
    one, two = outputs(), outputs()
    latd = to_device(lat, dtype)
    av.avits_select_upsample(to_device(A, "f32"), to_device(V, "f32"), 0.5, k, sel, o, m, latd, gh,
                             gw, *one, mode=av.BILINEAR)
    av.avits_selective_upsample(latd, gh, gw, m, o, k, *two, mode=av.BILINEAR)
    assert av.avits_device_status() == 0
    assert np.array_equal(to_numpy(m), mask) and np.array_equal(to_numpy(o), off)
    for got in (one, two):
        for g, w in zip(got, want):
            assert np.array_equal(to_numpy(g), w)
