"""GPU parity of the temporal kernels over row widths: the step variance where
the number of threads per token changes (rows of 8, 16 and 128 16-byte
vectors), and the relative change beside the spatial kernel where several
narrow rows share a copy and several rounds of blocks share the work.

Tolerance: fp32 sums of at most 4096 squares against fp64, each chain at most
(4096 / 8) terms before the tree: below 512 * 2^-24 = 3e-5 in the worst case
and ~2e-6 for random signs of the rounding; 1e-5 as for every fp32 score.
"""
import math

import numpy as np
import pytest

pytestmark = pytest.mark.gpu


@pytest.fixture(scope="module")
def av():
    import torch
    assert torch.cuda.is_available(), "GPU tests need a CUDA device"
    import paper_2608_17995_gb300 as av
    av.build()
    av.lib()
    return av


@pytest.mark.parametrize("dtype,vectors", [(t, v) for t in ("f32", "bf16")
                                           for v in (1, 8, 9, 16, 17, 127, 128, 129)])
@pytest.mark.parametrize("n_t,N", [(2, 1), (5, 17), (9, 33)])
def test_variance_row_widths(av, dtype, vectors, n_t, N):
    import torch
    import oracle
    from paper_2608_17995_gb300.pipeline import to_device, to_numpy
    from paper_2608_17995_gb300.workloads import to_bf16_bits
    D = vectors * (4 if dtype == "f32" else 8)
    rng = np.random.default_rng(D + n_t)
    snaps = [rng.standard_normal((3, N, D)).astype(np.float32) for _ in range(n_t)]
    if dtype == "bf16":
        snaps = [to_bf16_bits(s) for s in snaps]
    V = torch.full((3, N), float("nan"), device="cuda")
    av.avits_score_temporal_var([to_device(s, dtype) for s in snaps], V)
    assert av.avits_device_status() == 0
    np.testing.assert_allclose(to_numpy(V), oracle.score_temporal_var(snaps), rtol=1e-5, atol=1e-7)


@pytest.mark.parametrize("dtype,vectors", [("bf16", 1), ("bf16", 16), ("bf16", 33), ("bf16", 96),
                                           ("f32", 127), ("bf16", 127), ("bf16", 128)])
@pytest.mark.parametrize("n_t", [2, 3, 6, 16])
def test_variance_many_tokens(av, dtype, vectors, n_t):
    """More tokens than the widest of the rules for few, and a few of them alone,
    against the oracle.  The two sum a row's 16-byte vectors in another order for
    33 to 127 of them and in the same one for all other widths."""
    import torch
    import oracle
    from paper_2608_17995_gb300.pipeline import to_numpy
    D, N = vectors * (4 if dtype == "f32" else 8), 4500
    g = torch.Generator(device="cuda").manual_seed(D + n_t)
    snaps = [torch.randn(1, N, D, generator=g, device="cuda").to(
        torch.bfloat16 if dtype == "bf16" else torch.float32) for _ in range(n_t)]
    V, few = torch.full((1, N), float("nan"), device="cuda"), torch.full((1, 70), float("nan"), device="cuda")
    av.avits_score_temporal_var(snaps, V)
    av.avits_score_temporal_var([s[:, -70:].contiguous() for s in snaps], few)
    assert av.avits_device_status() == 0
    if not 32 < vectors < 128:
        assert torch.equal(V[:, -70:], few)
    want = oracle.score_temporal_var([to_numpy(s) for s in snaps])
    np.testing.assert_allclose(to_numpy(V), want, rtol=1e-5, atol=1e-7)
    np.testing.assert_allclose(to_numpy(few), want[:, -70:], rtol=1e-5, atol=1e-7)


@pytest.mark.parametrize("dtype,B,H,M,L,D", [
    ("bf16", 1, 1, 130, 20, 8),        # fewer rows than SMs: two per copy
    ("bf16", 1, 1, 12000, 20, 8),      # 64 rows of 16 bytes per copy, a ragged last one
    ("bf16", 1, 1, 1000, 20, 128),     # seven rows per copy
    ("bf16", 3, 2, 257, 40, 128),
    ("bf16", 2, 1, 4000, 24, 3072),    # several rounds beside a short spatial kernel
    ("bf16", 1, 1, 900, 16, 8192),     # one row per copy
    ("f32h", 1, 2, 300, 30, 768),      # fp32: after the CUDA-core spatial kernel
])
def test_temporal_beside_spatial(av, dtype, B, H, M, L, D):
    """The same V as the separate call, bit for bit, and the oracle's."""
    import torch
    import oracle
    from paper_2608_17995_gb300.pipeline import to_numpy
    g = torch.Generator(device="cuda").manual_seed(M + D)
    d = 64
    q = torch.randn(B, H, M, d, generator=g, device="cuda").bfloat16()
    k = torch.randn(B, H, L + M, d, generator=g, device="cuda").bfloat16()
    hd = torch.float32 if dtype == "f32h" else torch.bfloat16
    if hd != torch.bfloat16:   # the call takes one type: fp32 goes the CUDA-core way
        q, k = q.float(), k.float()
    hp = torch.randn(B, M, D, generator=g, device="cuda")
    ht = (hp + 0.3 * torch.randn(B, M, D, generator=g, device="cuda")).to(hd)
    hp = hp.to(hd)
    A, V, V2 = torch.empty(B, M, device="cuda"), torch.empty(B, M, device="cuda"), torch.empty(B, M, device="cuda")
    for _ in range(2):
        V.fill_(float("nan"))
        av.avits_score_spatiotemporal(q, k, L, 1 / math.sqrt(d), A, ht, hp, V)
        av.avits_score_temporal(ht, hp, V2)
        assert av.avits_device_status() == 0
        assert torch.equal(V, V2)
    np.testing.assert_allclose(to_numpy(V), oracle.score_temporal(to_numpy(ht), to_numpy(hp)), rtol=1e-5,
                               atol=1e-7)
