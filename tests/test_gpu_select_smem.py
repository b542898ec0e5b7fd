"""The one-launch selection + upsample where its dynamic shared memory alone is
just below the 48 KB that need no opt-in (its static arrays come on top)."""
import numpy as np
import pytest

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("B,gh,gw", [(64, 16, 40), (76, 18, 36)])
def test_shared_memory_just_below_the_default_limit(B, gh, gw):
    import torch
    import oracle
    import paper_2608_17995_gb300 as av
    from paper_2608_17995_gb300.pipeline import to_device, to_numpy
    av.build()
    M, C, k = gh * gw, 16, 100
    parts = max(1, min((M + 15) // 16, 152 // B))
    smem = 16 * ((9 * M + 15) // 16) + -(-M // parts) * C * 4 * 2
    assert 43 * 1024 < smem <= 48 * 1024
    rng = np.random.default_rng(B)
    A, V = rng.random((2, B, M)).astype(np.float32)
    _, mask, off = oracle.topk(oracle.fuse(A, V, 0.5), k)
    lat = rng.integers(0, 0x4000, (B, M, C * 4)).astype(np.uint16)
    want = oracle.selective_upsample(lat, gh, gw, mask)
    n = M + 3 * k
    i32 = dict(dtype=torch.int32, device="cuda")
    sel, o = torch.zeros(B, k, **i32), torch.zeros(B, M, **i32)
    m = torch.zeros(B, M, dtype=torch.uint8, device="cuda")
    out = torch.zeros(B, n, C * 4, dtype=torch.bfloat16, device="cuda")
    pos, span, tok = torch.zeros(B, n, 2, **i32), torch.zeros(B, n, **i32), torch.zeros(B, n, **i32)
    sub = torch.zeros(B, n, dtype=torch.int8, device="cuda")
    av.avits_select_upsample(to_device(A, "f32"), to_device(V, "f32"), 0.5, k, sel, o, m,
                             to_device(lat, "bf16"), gh, gw, out, pos, span, tok, sub)
    assert av.avits_device_status() == 0
    assert np.array_equal(to_numpy(m), mask) and np.array_equal(to_numpy(o), off)
    assert np.array_equal(to_numpy(out), want[0])
    for g, w in zip((pos, span, tok, sub), want[1:]):
        assert np.array_equal(to_numpy(g), w)
