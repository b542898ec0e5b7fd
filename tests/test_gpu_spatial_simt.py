"""GPU parity of the CUDA-core spatial score at the edges of its tiles: rows
per CTA (16 or 32), 128-key tiles, 32-column chunks, and heads whose key tiles
straddle the CTAs of a cluster.

Tolerance: the products, exponentials (ex2.approx, 2 ulp) and sums are fp32.  A
logit x (log2 units) is a sum of d products in four chains; its error is below
(d / 4 + 4) 2^-24 |q||k| scale log2(e), ~2e-6 at the sizes and values here, so a
mass is off by at most ~4e-6 of itself and A by less.  1e-5 is allowed.
"""
import math

import numpy as np
import pytest

pytestmark = pytest.mark.gpu

TOL = 1e-5


@pytest.fixture(scope="module")
def av():
    import torch
    assert torch.cuda.is_available(), "GPU tests need a CUDA device"
    import paper_2608_17995_gb300 as av
    av.build()
    av.lib()
    return av


@pytest.mark.parametrize("dtype,B,H,M,L,R,d,mask", [
    ("f32", 1, 1, 1, 1, 0, 1, False),          # one query, one key, one column
    ("f32", 1, 1, 15, 3, 112, 31, False),      # below every tile; 130 keys: a tile of two
    ("f32", 2, 3, 17, 111, 0, 33, False),      # 128 keys exactly, a second row tile of one
    ("f32", 1, 5, 33, 96, 0, 36, True),        # 129 keys, a last chunk of four columns
    ("f32", 1, 2, 300, 77, 640, 40, False),    # 8 key tiles x 2 heads over 8 CTAs
    ("f32", 1, 1, 64, 50, 1500, 64, True),     # one head over every CTA of the cluster
    ("f32", 1, 7, 100, 60, 0, 128, False),     # heads straddle CTAs at every boundary
    ("f32", 3, 24, 700, 33, 0, 64, False),     # 32-row tiles, the last of 28 rows
    ("f32", 1, 2, 40, 20, 0, 256, False),      # the widest head
    ("bf16", 1, 3, 129, 5, 0, 41, False),      # element-wise loads
    ("bf16", 2, 4, 96, 64, 97, 96, True),
    ("bf16", 1, 260, 20, 13, 0, 64, False),    # more heads than the tensor-core path takes
])
def test_simt_edges(av, dtype, B, H, M, L, R, d, mask):
    import torch
    import oracle
    from paper_2608_17995_gb300.pipeline import to_device, to_numpy
    from paper_2608_17995_gb300.workloads import to_bf16_bits
    rng = np.random.default_rng(B * 7919 + H * 31 + M * d + L)
    N = L + M + R
    c = math.sqrt(2.0)
    q = (rng.standard_normal((B, H, M, d)) * c).astype(np.float32)
    k = (rng.standard_normal((B, H, N, d)) * c).astype(np.float32)
    if dtype == "bf16":
        q, k = to_bf16_bits(q), to_bf16_bits(k)
    tm = (rng.random((B, N)) < 0.3).astype(np.uint8) if mask else None
    if mask:
        tm[:, 0] = 1
    qd, kd = to_device(q, dtype), to_device(k, dtype)
    A = torch.full((B, M), 0.5, device="cuda")
    lse = torch.zeros(B, H, M, 2, device="cuda")
    scale = 1.0 / math.sqrt(d)
    av.avits_score_spatial(qd, kd, L, scale, A, weight=0.5, accumulate=True, lse=lse,
                           text_mask=None if tm is None else torch.from_numpy(tm).cuda())
    assert av.avits_device_status() == 0
    A_o, _, lse_o = oracle.score_spatial(q, k, L, scale, weight=0.5,
                                         A_in=np.full((B, M), 0.5, np.float32), text_mask=tm)
    np.testing.assert_allclose(to_numpy(A), A_o, rtol=TOL, atol=1e-7)
    np.testing.assert_allclose(to_numpy(lse), lse_o, rtol=TOL, atol=2e-5)
    # a strided (token-major) and a misaligned view take the other load path
    if dtype == "f32" and d > 1:
        buf = torch.zeros(B, N, H, d + 1, device="cuda")[..., 1:]
        buf.copy_(kd.transpose(1, 2))
        A2 = torch.full((B, M), 0.5, device="cuda")
        av.avits_score_spatial(qd, buf.transpose(1, 2), L, scale, A2, weight=0.5, accumulate=True,
                               text_mask=None if tm is None else torch.from_numpy(tm).cuda())
        assert av.avits_device_status() == 0
        assert torch.equal(A, A2)   # the same sums in the same order


@pytest.mark.parametrize("B,H,M,L,R,d", [
    (1, 1, 1, 1, 0, 8),             # one row, one vector
    (1, 1, 64, 36, 0, 256),         # one key tile of 100
    (2, 3, 17, 111, 0, 40),         # a last chunk of one vector
    (1, 2, 300, 77, 640, 96),
    (3, 24, 700, 33, 0, 32),        # 32-row tiles, the last of 28 rows
    (16, 1, 70, 26, 0, 264 - 16),   # eight chunks, the last of three vectors
])
def test_simt_bf16_vectors(av, B, H, M, L, R, d):
    """bf16 in 16-byte loads: the oracle's values, and the bits of the
    element-wise loads that a misaligned view takes."""
    import torch
    import oracle
    from paper_2608_17995_gb300.pipeline import to_numpy
    g = torch.Generator(device="cuda").manual_seed(M + d)
    N, scale = L + M + R, 1.0 / math.sqrt(d)
    q = (math.sqrt(2.0) * torch.randn(B, H, M, d, generator=g, device="cuda")).bfloat16()
    k = (math.sqrt(2.0) * torch.randn(B, H, N, d, generator=g, device="cuda")).bfloat16()
    A, A2 = torch.zeros(B, M, device="cuda"), torch.zeros(B, M, device="cuda")
    av.avits_score_spatial(q, k, L, scale, A)
    buf = torch.zeros(B, N, H, d + 1, device="cuda", dtype=torch.bfloat16)[..., 1:]
    buf.copy_(k.transpose(1, 2))
    av.avits_score_spatial(q, buf.transpose(1, 2), L, scale, A2)
    assert av.avits_device_status() == 0
    assert torch.equal(A, A2)
    # token-major rows of whole vectors keep the 16-byte loads
    av.avits_score_spatial(q, k.transpose(1, 2).contiguous().transpose(1, 2), L, scale, A2)
    assert av.avits_device_status() == 0
    assert torch.equal(A, A2)
    want = oracle.score_spatial(to_numpy(q), to_numpy(k), L, scale)[0]
    np.testing.assert_allclose(to_numpy(A), want, rtol=TOL, atol=1e-7)


def test_simt_no_finite_key(av):
    """NaN and infinite logits give NaN for their rows alone."""
    import torch
    q = torch.ones(1, 2, 40, 32, device="cuda")
    k = torch.ones(1, 2, 140, 32, device="cuda")
    q[0, 1, 3, 0] = float("nan")
    q[0, 0, 35, 5] = float("inf")
    A = torch.zeros(1, 40, device="cuda")
    av.avits_score_spatial(q, k, 70, 0.1, A)
    assert av.avits_device_status() == 0
    bad = torch.isnan(A[0]).nonzero()[:, 0].tolist()
    assert bad == [3, 35]
    good = torch.ones(40, dtype=torch.bool, device="cuda")
    good[[3, 35]] = False
    torch.testing.assert_close(A[0][good], torch.full_like(A[0][good], 0.5), rtol=1e-6, atol=0)
