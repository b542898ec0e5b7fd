"""GPU parity (bit-exact) of the two-pass merge: batches of more tokens than
one pass takes in nearest mode, and the bilinear merge, over token widths that
are and are not whole 16-byte pieces, spans of every kind, and tilings that do
not cover the frame, with one workspace used by both modes in turn."""
import numpy as np
import pytest

pytestmark = pytest.mark.gpu

NEAREST, BILINEAR = 0, 1


@pytest.fixture(scope="module")
def av():
    import torch
    assert torch.cuda.is_available(), "GPU tests need a CUDA device"
    import paper_2608_17995_gb300 as av
    av.build()
    av.lib()
    return av


def _tiling(rng, B, fh, fw, block, spans):
    """pos [B,N,2], span [B,N]: blocks of block x block cells cut into tokens of
    one span each, the same spans in every element but in other places and
    another token order."""
    cells = [(y, x) for y in range(0, fh, block) for x in range(0, fw, block)]
    kinds = rng.choice(spans, size=len(cells))
    pos, span = [], []
    for _ in range(B):
        p, s = [], []
        for (y, x), k in zip(cells, rng.permutation(kinds)):
            for u in range(0, block, k):
                for v in range(0, block, k):
                    p.append((y + u, x + v))
                    s.append(k)
        order = rng.permutation(len(s))
        pos.append(np.array(p, np.int32)[order])
        span.append(np.array(s, np.int32)[order])
    return np.ascontiguousarray(np.stack(pos)), np.ascontiguousarray(np.stack(span))


def _latent(rng, B, N, C, dtype):
    from paper_2608_17995_gb300.workloads import to_bf16_bits
    x = rng.standard_normal((B, N, C * 4)).astype(np.float32)
    return to_bf16_bits(x) if dtype == "bf16" else x


def _call(av, mixed, dtype, pos, span, fh, fw, mode, ws):
    import torch
    from paper_2608_17995_gb300.pipeline import to_device, to_numpy
    B, _, T = mixed.shape
    out = torch.full((B, fh * fw, T), 7.0, device="cuda",
                     dtype=torch.bfloat16 if dtype == "bf16" else torch.float32)
    av.avits_merge_final(to_device(mixed, dtype), to_device(pos, "i32"), to_device(span, "i32"),
                         fh, fw, out, mode=mode, workspace=ws)
    return to_numpy(out), av.avits_device_status()


def _same(a, b):
    v = np.uint16 if a.dtype == np.uint16 else np.uint32
    return np.array_equal(a.view(v), b.view(v))


@pytest.mark.parametrize("mode", [NEAREST, BILINEAR])
@pytest.mark.parametrize("dtype,C,B,fh,fw", [
    ("bf16", 16, 41, 24, 36), ("bf16", 1, 60, 24, 24), ("bf16", 3, 37, 12, 60), ("f32", 1, 45, 24, 36),
    ("f32", 5, 40, 36, 24), ("bf16", 16, 3, 84, 108)])
def test_merge_two_pass_bit_exact(av, mode, dtype, C, B, fh, fw):
    import torch
    import oracle
    rng = np.random.default_rng(C * 1000 + B + mode)
    block, spans = (12, [1, 2, 3, 4, 6, 12]) if mode == NEAREST else (4, [1, 2, 4])
    if mode == BILINEAR and C == 16:
        spans = [1, 2]   # the common schedule: no level-2 pixels
    ws = torch.zeros(av.avits_merge_final_workspace(mode, B, fh, fw), dtype=torch.uint8, device="cuda")
    for _ in range(2):   # the second call finds the first one's map
        pos, span = _tiling(rng, B, fh, fw, block, spans)
        mixed = _latent(rng, B, pos.shape[1], C, dtype)
        got, st = _call(av, mixed, dtype, pos, span, fh, fw, mode, ws)
        want, cover = oracle.merge_final(mixed, pos, span, fh, fw,
                                         mode="nearest" if mode == NEAREST else "bilinear")
        assert st == 0 and np.all(cover == 1)
        assert _same(got, want)


@pytest.mark.parametrize("spans", [[1, 2], [1, 3, 4], [1, 6, 12]])
@pytest.mark.parametrize("dtype,C,B", [
    ("bf16", 1, 20), ("bf16", 3, 20), ("bf16", 4, 20), ("f32", 1, 20),     # 8 lanes per token
    ("bf16", 1, 90), ("bf16", 3, 90)])                                     # two passes
def test_merge_nearest_routes(av, spans, dtype, C, B):
    """Small tokens on both sides of the lines between one pass and two, with
    spans whose cells are up to nine rounds of a token's eight lanes, a call with
    a hole and one with a cell covered twice among good ones."""
    import torch
    import oracle
    rng = np.random.default_rng(C + B + sum(spans))
    fh, fw = 36, 24
    ws = torch.zeros(av.avits_merge_final_workspace(NEAREST, B, fh, fw), dtype=torch.uint8, device="cuda")
    # a span-1 block in every frame: at least 144 tokens an element
    pos, span = _tiling(rng, B, fh, fw, 12, spans)
    while pos.shape[1] < 144:
        pos, span = _tiling(rng, B, fh, fw, 12, spans)
    mixed = _latent(rng, B, pos.shape[1], C, dtype)
    want, cover = oracle.merge_final(mixed, pos, span, fh, fw)
    assert np.all(cover == 1)
    for bad in (None, "hole", "twice", None):
        p, s = pos.copy(), span.copy()
        if bad == "hole":
            s[B - 1, 3] = 0
        elif bad == "twice":
            one = np.flatnonzero(s[0] == 1)[:2]
            p[0, one[1]] = p[0, one[0]]
        got, st = _call(av, mixed, dtype, p, s, fh, fw, NEAREST, ws)
        assert st == (0 if bad is None else 6)
        if bad is None:
            assert _same(got, want)


@pytest.mark.parametrize("mode", [NEAREST, BILINEAR])
@pytest.mark.parametrize("dtype,C,B", [("bf16", 16, 1), ("bf16", 4, 20), ("bf16", 16, 20), ("bf16", 3, 20),
                                       ("bf16", 3, 80)])
def test_positions_and_spans_beyond_the_integers(av, mode, dtype, C, B):
    """A token whose last row or column does not fit an int is outside the frame
    like any other: reported, its cells are holes, and the next call is right."""
    import torch
    import oracle
    rng = np.random.default_rng(C + B)
    fh, fw, top = 24, 24, 2 ** 31 - 1
    pos, span = _tiling(rng, B, fh, fw, 4, [1, 2])
    mixed = _latent(rng, B, pos.shape[1], C, dtype)
    want, _ = oracle.merge_final(mixed, pos, span, fh, fw, mode="nearest" if mode == NEAREST else "bilinear")
    ws = torch.zeros(av.avits_merge_final_workspace(mode, B, fh, fw), dtype=torch.uint8, device="cuda")
    for at, s in (([top, 0], None), ([0, top], None), ([top - 1, top - 1], None), ([1, 0], top),
                  ([top, top], top), ([-top - 1, 3], top)):
        p, sp = pos.copy(), span.copy()
        p[B - 1, 5] = at
        if s is not None:
            sp[B - 1, 5] = s
        assert _call(av, mixed, dtype, p, sp, fh, fw, mode, ws)[1] == 6
    got, st = _call(av, mixed, dtype, pos, span, fh, fw, mode, ws)
    assert st == 0 and _same(got, want)


@pytest.mark.parametrize("first", [NEAREST, BILINEAR])
def test_merge_two_pass_reports_bad_tilings(av, first):
    import torch
    import oracle
    rng = np.random.default_rng(5)
    B, fh, fw = 48, 24, 24
    pos, span = _tiling(rng, B, fh, fw, 4, [1, 2])
    mixed = _latent(rng, B, pos.shape[1], 4, "f32")
    N = pos.shape[1]
    ws = torch.zeros(av.avits_merge_final_workspace(NEAREST, B, fh, fw), dtype=torch.uint8, device="cuda")
    want = {m: oracle.merge_final(mixed, pos, span, fh, fw,
                                  mode="nearest" if m == NEAREST else "bilinear")[0]
            for m in (NEAREST, BILINEAR)}

    def bad():
        two = np.flatnonzero(span[B - 1] == 1)[:2]
        moved = pos.copy()
        moved[B - 1, two[1]] = pos[B - 1, two[0]]       # a cell twice, another not at all
        yield moved, span
        empty = span.copy()
        empty[0, N // 2] = 0                            # a token of no cells
        yield pos, empty
        far = pos.copy()
        far[B // 2, 0] = [fh - 1, fw]                   # outside the frame
        yield far, span

    for p, s in bad():
        for m in (first, 1 - first):
            assert _call(av, mixed, "f32", p, s, fh, fw, m, ws)[1] == 6
            got, st = _call(av, mixed, "f32", pos, span, fh, fw, m, ws)
            assert st == 0 and _same(got, want[m])


@pytest.mark.parametrize("spans", [[1, 2], [1, 2, 4]])
@pytest.mark.parametrize("dtype,C", [("bf16", 1), ("bf16", 3), ("bf16", 16), ("f32", 1), ("f32", 4)])
def test_a_hole_shows_nothing_of_earlier_calls(av, dtype, C, spans):
    """A bilinear merge with holes on a workspace that a merge of more tokens
    used before: reported, and the cells around a hole draw on zeros, not on
    what the old words name (tokens beyond this call's, here among the NaNs
    around the sequence, or tokens elsewhere in it)."""
    import torch
    import oracle
    from paper_2608_17995_gb300.pipeline import to_device, to_numpy
    rng = np.random.default_rng(C + len(spans))
    B, fh, fw = 3, 40, 24   # one token per cell: enough for the nearest merge's two passes
    pos, span = _tiling(rng, B, fh, fw, 4, spans)
    N, T = pos.shape[1], 4 * C
    mixed = _latent(rng, B, N, C, dtype)
    for b in range(B):   # two holes of every span, the frame's last token among them
        last = np.flatnonzero((pos[b] + span[b][:, None] == [fh, fw]).all(1))
        holes = np.concatenate([rng.choice(np.flatnonzero(span[b] == s), 2) for s in spans] + [last])
        span[b, holes] *= -1
        mixed[b, holes] = 0
    out = np.zeros((B, fh, fw), bool)   # cells of holes
    for b, t in zip(*np.nonzero(span < 0)):
        y, x, s = *pos[b, t], -span[b, t]
        out[b, y:y + s, x:x + s] = True
    out = out.reshape(B, fh * fw)
    tdt = torch.bfloat16 if dtype == "bf16" else torch.float32
    n = B * N * T + -B * N * T % 8   # the sequence starts on 16 bytes
    wide = torch.full((3 * n,), float("nan"), dtype=tdt, device="cuda")
    view = wide[n:n + B * N * T].view(B, N, T)
    view.copy_(to_device(mixed, dtype))
    dense = np.stack([np.stack(np.divmod(np.arange(fh * fw), fw), 1)] * B).astype(np.int32)
    ones = np.ones((B, fh * fw), np.int32)
    got = []
    for first in (None, NEAREST, BILINEAR):
        ws = torch.zeros(av.avits_merge_final_workspace(BILINEAR, B, fh, fw), dtype=torch.uint8,
                         device="cuda")
        if first is not None:   # one token per cell, in raster order
            assert _call(av, _latent(rng, B, fh * fw, C, dtype), dtype, dense, ones, fh, fw, first,
                         ws)[1] == 0
        full = torch.full((B, fh * fw, T), 7.0, dtype=tdt, device="cuda")
        av.avits_merge_final(view, to_device(pos, "i32"), to_device(span, "i32"), fh, fw, full,
                             mode=BILINEAR, workspace=ws)
        assert av.avits_device_status() == 6
        got.append(to_numpy(full))
    assert _same(got[0], got[1]) and _same(got[0], got[2])
    assert not got[0][out].any()
    if spans == [1, 2]:   # elsewhere: as if the missing tokens were zeros
        want, _ = oracle.merge_final(mixed, pos, np.abs(span), fh, fw, mode="bilinear")
        assert _same(got[0][~out], want[~out])


@pytest.mark.parametrize("dtype,C,gh,gw,k", [
    ("bf16", 16, 9, 13, 40), ("f32", 4, 16, 16, 0), ("f32", 1, 8, 30, 240), ("bf16", 2, 33, 8, 100),
    ("bf16", 1, 8, 8, 30), ("bf16", 16, 1, 20, 7), ("bf16", 16, 20, 1, 7)])
def test_bilinear_children_bit_exact(av, dtype, C, gh, gw, k):
    """The bilinear children of a dense grid, at its edges and corners, through
    both upsample entry points (one grid row or column included)."""
    import torch
    import oracle
    from paper_2608_17995_gb300.pipeline import to_device, to_numpy
    rng = np.random.default_rng(gh * 100 + gw)
    B, M = 3, gh * gw
    lat = _latent(rng, B, M, C, dtype)
    A, V = rng.random((2, B, M)).astype(np.float32)
    S = oracle.fuse(A, V, 0.5)
    _, mask, off = oracle.topk(S, k)
    want = oracle.selective_upsample(lat, gh, gw, mask, mode="bilinear")
    tdt = torch.bfloat16 if dtype == "bf16" else torch.float32
    n = M + 3 * k

    def outs():
        return (torch.zeros(B, n, C * 4, dtype=tdt, device="cuda"),
                torch.zeros(B, n, 2, dtype=torch.int32, device="cuda"),
                torch.zeros(B, n, dtype=torch.int32, device="cuda"),
                torch.zeros(B, n, dtype=torch.int32, device="cuda"),
                torch.zeros(B, n, dtype=torch.int8, device="cuda"))
    ld = to_device(lat, dtype)
    one, two = outs(), outs()
    av.avits_selective_upsample(ld, gh, gw, to_device(mask, "u8"), to_device(off, "i32"), k, *one,
                                mode=BILINEAR)
    sel = torch.zeros(B, max(k, 1), dtype=torch.int32, device="cuda")
    o = torch.zeros(B, M, dtype=torch.int32, device="cuda")
    m = torch.zeros(B, M, dtype=torch.uint8, device="cuda")
    av.avits_select_upsample(to_device(A, "f32"), to_device(V, "f32"), 0.5, k, sel, o, m, ld, gh, gw,
                             *two, mode=BILINEAR)
    assert av.avits_device_status() == 0
    for got in (one, two):
        assert _same(to_numpy(got[0]), want[0])
        for g, w in zip(got[1:], want[1:]):
            assert np.array_equal(to_numpy(g), w)
