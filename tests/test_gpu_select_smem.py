"""The selection kernels where their dynamic shared memory alone is just below
the 48 KB that need no opt-in (their static arrays come on top)."""
import os
import subprocess
import sys

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


def select_at(gh, gw, entry):
    """One selection of gh x gw tokens through `entry`, against the oracle."""
    import torch
    import oracle
    import paper_2608_17995_gb300 as av
    from paper_2608_17995_gb300.pipeline import to_device, to_numpy
    av.build()
    M, C, k = gh * gw, 4, gh * gw // 3
    rng = np.random.default_rng(M)
    A, V = rng.random((2, 1, M)).astype(np.float32)
    _, mask, off = oracle.topk(oracle.fuse(A, V, 0.5), k)
    i32 = dict(dtype=torch.int32, device="cuda")
    sel, o = torch.zeros(1, k, **i32), torch.zeros(1, M, **i32)
    m = torch.zeros(1, M, dtype=torch.uint8, device="cuda")
    Ad, Vd = to_device(A, "f32"), to_device(V, "f32")
    if entry == "select":
        av.avits_fuse_select(Ad, Vd, 0.5, k, sel, o, sel_mask=m)
    else:
        lat = rng.standard_normal((1, M, C * 4)).astype(np.float32)
        pos = span = None
        if entry == "mixed":   # span-1 tokens in raster order
            pos = np.stack(np.divmod(np.arange(M), gw), 1).astype(np.int32)[None]
            span = np.ones((1, M), np.int32)
        want = oracle.selective_upsample(lat, gh, gw, mask, pos_in=pos, span_in=span)
        n = M + 3 * k
        out = [torch.zeros(1, n, C * 4, device="cuda"), torch.zeros(1, n, 2, **i32),
               torch.zeros(1, n, **i32), torch.zeros(1, n, **i32),
               torch.zeros(1, n, dtype=torch.int8, device="cuda")]
        mixed = {} if pos is None else dict(pos_in=to_device(pos, "i32"), span_in=to_device(span, "i32"))
        av.avits_select_upsample(Ad, Vd, 0.5, k, sel, o, m, to_device(lat, "f32"), gh, gw, *out, **mixed)
        for g, w in zip(out, want):
            assert np.array_equal(to_numpy(g), w)
    assert av.avits_device_status() == 0
    assert np.array_equal(to_numpy(m), mask) and np.array_equal(to_numpy(o), off)


@pytest.mark.parametrize("entry", ["select", "upsample", "mixed"])
@pytest.mark.parametrize("gh,gw", [(108, 110), (96, 128)])
def test_large_selection_in_a_fresh_process(gh, gw, entry):
    """11,880 and 12,288 tokens (46 and 48 KB of keys) as a process's first
    call: the kernel's limit is raised once for good, so an earlier and larger
    selection would hide a missing opt-in."""
    root = os.path.dirname(os.path.dirname(os.path.abspath(__file__)))
    code = "import sys; sys.path[:0] = [%r, %r]; import test_gpu_select_smem as t; t.select_at(%d, %d, %r)" % (
        root, os.path.join(root, "tests"), gh, gw, entry)
    r = subprocess.run([sys.executable, "-c", code], cwd=root, capture_output=True, text=True, timeout=300)
    assert r.returncode == 0, r.stdout[-2000:] + r.stderr[-2000:]
