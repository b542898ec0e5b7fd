"""GPU parity of the joint-attention forward where its 64-key steps and units
can go wrong: the reference of the exponentials moving in the first or the
second half of a key tile (O rescaled between its two products), key counts
around a half tile, and one key tile per unit with several units per block.

Tolerances as in test_gpu_attention (P and O rounded to bf16 once each).
"""
import math

import numpy as np
import pytest

from test_gpu_attention import _bf16, _compare, _f32, _rand_qkv, _run, av, orc  # noqa: F401

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("d", [64, 128])
@pytest.mark.parametrize("cols", [(70, 71), (128, 192), (200, 201), (300, 301), (64, 128)])
def test_reference_moves_in_either_half(av, orc, d, cols):  # noqa: F811
    """One run of keys with logits far above the rest (their exponentials pass
    2^32 against the earlier reference), in the first or second half.  Their
    logits have a standard deviation of 3 * 5 nats = 21.6 log2 units: 1.5 of
    these pass 2^32, and 5.5 would be needed to take the text keys' sum below
    the normal range (2^-126 of the row's largest term), where lse_txt is -inf
    by the interface."""
    B, H, Mq, Nk, L = 1, 2, 140, 310, 75
    q, k, v = _rand_qkv(31 + cols[0] + d, B, H, Mq, Nk, d)
    kf = _f32(k)
    kf[:, :, cols[0]:cols[1]] *= 5.0
    k = _bf16(kf)
    scale = 1.0 / math.sqrt(d)
    o, lse, A = _run(av, q, k, v, L, scale)
    _compare(orc, q, k, v, L, scale, o, lse, A)


@pytest.mark.parametrize("Nk,L", [(63, 10), (64, 64), (65, 1), (128, 100), (129, 127), (192, 64)])
def test_key_counts_around_a_half_tile(av, orc, Nk, L):  # noqa: F811
    q, k, v = _rand_qkv(Nk, 1, 3, 257, Nk, 128)
    scale = 1.0 / math.sqrt(128)
    o, lse, A = _run(av, q, k, v, L, scale)
    _compare(orc, q, k, v, L, scale, o, lse, A)


@pytest.mark.parametrize("d", [64, 128])
def test_one_key_tile_per_unit(av, orc, d):  # noqa: F811
    """400 units of one key tile: every step ends a unit, so Q, K and V of the
    next one, its S product and this one's epilogue follow each other."""
    B, H, Mq, Nk, L = 2, 100, 300, 100, 30
    q, k, v = _rand_qkv(77 + d, B, H, Mq, Nk, d)
    scale = 1.0 / math.sqrt(d)
    o, lse, A = _run(av, q, k, v, L, scale)
    _compare(orc, q, k, v, L, scale, o, lse, A)


@pytest.mark.parametrize("d", [64, 128])
@pytest.mark.parametrize("what", ["nan", "small", "large"])
def test_rows_stay_alone(av, d, what):  # noqa: F811
    """A row's results are its own: another row of its warp that holds a NaN, or
    whose logits pass the sums from which P's rounding is made up for (2^6) and
    from which the reference moves (2^16), changes none of their bits."""
    import torch
    torch.manual_seed(d)
    q, k, v = (torch.randn(1, 2, 333, d, device="cuda").bfloat16() for _ in range(3))
    one, two = [(torch.empty_like(q), torch.empty(1, 2, 333, 2, device="cuda")) for _ in range(2)]
    scale = 1.0 / math.sqrt(d)
    av.avits_attention_forward(q, k, v, 40, scale, one[0], lse=one[1])
    rows = [5, 40, 331]
    if what == "nan":
        q[0, 1, rows, 3] = float("nan")
    else:   # a logit of 9 or 18 nats at a key of the second tile: ~2^9, ~2^18 above the first
        u = k[0, 1, 200].float()
        q[0, 1, rows] = (u * ((9.0 if what == "small" else 18.0) / (scale * u.dot(u)))).bfloat16()
    av.avits_attention_forward(q, k, v, 40, scale, two[0], lse=two[1])
    assert av.avits_device_status() == 0
    other = torch.ones(2, 333, dtype=torch.bool, device="cuda")
    other[1, rows] = False
    for x, y in zip(one, two):
        assert torch.equal(x[0][other], y[0][other])


def test_nan_rows_stay_alone(av):  # noqa: F811
    import torch
    q = torch.randn(1, 2, 300, 128, device="cuda").bfloat16()
    k, v = (torch.randn(1, 2, 333, 128, device="cuda").bfloat16() for _ in range(2))
    o, o2 = torch.empty_like(q), torch.empty_like(q)
    av.avits_attention_forward(q, k, v, 40, 0.09, o)
    q[0, 1, 5, 3] = float("nan")
    av.avits_attention_forward(q, k, v, 40, 0.09, o2)
    assert av.avits_device_status() == 0
    assert torch.isnan(o2[0, 1, 5]).all()
    o[0, 1, 5] = 0
    o2[0, 1, 5] = 0
    # the other rows of the warp take the step again: the same terms
    assert torch.equal(o2, o)
    assert np.isfinite(o2.float().cpu().numpy()).all()
