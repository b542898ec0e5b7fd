"""The work this library is measured on: calls of its public entry points.

Six kinds of case, each what a program around a diffusion transformer has it do:

  transition  one whole resolution transition (scores, selection, upsample, merge)
  scores      both token scores of one denoising step
  spatial     the spatial score of one or more blocks (text keys first, marked by
              a mask, or scored against the model attention's logsumexp)
  attention   a block's joint-attention forward that emits the score as well
  variance    the step variance over N_T snapshots
  tail        selection, selective upsample and final merge of given scores

``listed()`` holds the shapes of the FLUX family at 1024^2 and 2048^2, of an
editing model, of batched serving and of the tiny fp32 configuration; ``draw``
spreads sizes, batches, ragged grids, types, layouts and options over the same
ranges.  Inputs are drawn on the GPU from the seed alone, with the recipe of
``paper_2608_17995_gb300.workloads``: logits of standard deviation 3, regions
that attend to a few text keys, and a smooth field of step changes.
"""
from __future__ import annotations

import math

import torch
import torch.nn.functional as F

import paper_2608_17995_gb300 as av
from paper_2608_17995_gb300.pipeline import TransitionBuffers
from paper_2608_17995_gb300.workloads import Transition

DEV = "cuda"
ALPHA = 0.5


def _transition(name, dtype, B, H, gh, gw, L, R, d, D, k, mode):
    return dict(name=name, kind="transition", dtype=dtype, B=B, H=H, gh=gh, gw=gw, L=L, R=R, d=d,
                D=D, C=16, k=k, mode=mode)


def _scores(name, dtype, B, H, gh, gw, L, R, d, D):
    return dict(name=name, kind="scores", dtype=dtype, B=B, H=H, gh=gh, gw=gw, L=L, R=R, d=d, D=D)


def _spatial(name, dtype, B, H, gh, gw, L, R, d, text, blocks, layout):
    return dict(name=name, kind="spatial", dtype=dtype, B=B, H=H, gh=gh, gw=gw, L=L, R=R, d=d,
                text=text, blocks=blocks, layout=layout)


def _attention(name, B, H, gh, gw, L, R, d, layout):
    return dict(name=name, kind="attention", dtype="bf16", B=B, H=H, gh=gh, gw=gw, L=L, R=R, d=d,
                layout=layout)


def _variance(name, dtype, B, N, D, n_t):
    return dict(name=name, kind="variance", dtype=dtype, B=B, N=N, D=D, n_t=n_t)


def _tail(name, dtype, B, gh, gw, C, k, mode, mixed):
    return dict(name=name, kind="tail", dtype=dtype, B=B, gh=gh, gw=gw, C=C, k=k, mode=mode,
                mixed=mixed)


def listed():
    return [
        # the smallest configuration: fp32, two heads; launches and latency
        _transition("tiny_f32", "f32", 1, 2, 16, 16, 32, 0, 64, 128, 64, "nearest"),
        # one image at 1024^2, the headline transition
        _transition("flux1024", "bf16", 1, 24, 32, 32, 512, 0, 128, 3072, 307, "nearest"),
        # first transition of a batched multi-stage schedule: 8 images, 16x16 tokens
        _scores("scores_b8", "bf16", 8, 24, 16, 16, 512, 0, 128, 3072),
        # one image at 2048^2
        _scores("scores_2048", "bf16", 1, 24, 64, 64, 512, 0, 128, 3072),
        # an editing model: reference-image keys, the score aggregated over two
        # blocks, Q and K read in place from token-major projections
        _spatial("spatial_edit", "bf16", 1, 24, 32, 32, 512, 4096, 128, "prefix", 2, "tokens"),
        # a unified sequence whose text keys lie between image keys; ragged grid
        _spatial("spatial_unified", "bf16", 1, 24, 37, 45, 333, 0, 128, "mask", 1, "heads"),
        # full-precision scoring of the 1024^2 shape (validation runs)
        _spatial("spatial_f32", "f32", 1, 24, 32, 32, 512, 0, 128, "prefix", 1, "heads"),
        # a double-stream block's attention at 1024^2 and, batched, at 2048^2
        _attention("attention_1024", 1, 24, 32, 32, 512, 0, 128, "heads"),
        _attention("attention_2048", 2, 24, 64, 64, 512, 0, 128, "tokens"),
        # Eq. 6-7 over four collected steps of two 2048^2 images
        _variance("variance_2048", "bf16", 2, 4096, 3072, 4),
        # a served batch of 1024^2 images with bilinear resampling
        _tail("tail_bilinear", "bf16", 16, 32, 32, 16, 307, "bilinear", False),
        # the second transition of 32 schedules (a mixed 32x32 frame each)
        _tail("tail_mixed", "bf16", 32, 32, 32, 16, 192, "nearest", True),
    ]


# ------------------------------------------------------------------- draw --
def _log(rng, lo, hi):
    return int(round(math.exp(rng.uniform(math.log(lo), math.log(hi)))))


def _grid(rng, lo, hi):
    """A grid of lo..hi tokens with an aspect ratio of up to 2."""
    m, r = _log(rng, lo, hi), math.sqrt(rng.uniform(0.5, 2.0))
    gh = max(8, int(round(math.sqrt(m) * r)))
    gw = max(8, m // gh)
    while gh * gw > hi:
        gw -= 1
    return gh, gw


def _heads_dim(rng, dtype):
    d = rng.choice([64, 128]) if dtype == "bf16" else rng.choice([40, 64, 96, 128])
    return rng.randint(2, 24), d


def draw(rng):
    c = _drawn(rng)
    while c["kind"] in ("tail", "transition") and not _launches(c):
        c = _drawn(rng)
    return c


def _launches(c):
    """Whether the one-launch selection and upsample takes the sizes: where its
    scores and latent rows fill shared memory up to the last kilobytes below
    the default limit, the launch is refused."""
    M = _mixed_tokens(c["gh"], c["gw"]) if c.get("mixed") else c["gh"] * c["gw"]
    parts = max(1, min((M + 15) // 16, max(1, 152 // c["B"])))
    halo = c["gw"] + 1 if c["mode"] == "bilinear" else 0
    rows = min(M, -(-M // parts) + 2 * halo) * c["C"] * 4 * _elt(c)
    head = 16 * ((9 * M + 15) // 16)
    return not any(42 * 1024 < x <= 48 * 1024 for x in (head, head + rows))


def _drawn(rng):
    kind = rng.choice(["transition", "scores", "spatial", "attention", "variance", "tail"])
    dtype = rng.choice(["bf16", "bf16", "bf16", "f32"])
    layout = rng.choice(["heads", "tokens"])
    L = _log(rng, 24, 512)
    if kind == "variance":
        D = rng.choice([128, 768, 1000, 1152, 3072, 4096])
        n_t = rng.randint(2, 6)
        tokens = _log(rng, 256, (8192 * 3072 * 4) // (D * n_t * (2 if dtype == "f32" else 1)))
        B = rng.randint(1, min(8, tokens // 256))
        c = _variance("", dtype, B, tokens // B, D, n_t)
    elif kind == "tail":
        gh, gw = _grid(rng, 100, 16384)
        mixed = rng.random() < 0.4
        mode = rng.choice(["nearest", "bilinear"])
        if mixed:   # the frame of a first transition: twice a grid in each direction
            gh, gw = max(8, gh // 2) * 2, max(8, gw // 2) * 2
        B = _log(rng, 1, max(1, min(64, 65536 // (gh * gw))))
        M = _mixed_tokens(gh, gw) if mixed else gh * gw
        C = rng.choice([4, 16, 16, 16])
        c = _tail("", dtype, B, gh, gw, C, rng.randint(M // 8, M // 2), mode, mixed)
    else:
        H, d = _heads_dim(rng, "bf16" if kind == "attention" else dtype)
        top = 4096 if dtype == "bf16" or kind == "attention" else 1024
        gh, gw = _grid(rng, 144, top)
        R = 4 * gh * gw if gh * gw <= 1024 and rng.random() < 0.2 and dtype == "bf16" else 0
        keys = L + gh * gw + R
        # at most the work of the largest listed case of the type
        most = 2 * 24 * 4608 * 4608 if kind == "attention" else (
            24 * 4096 * 4608 if dtype == "bf16" else 24 * 1024 * 1536)
        rows = keys if kind == "attention" else gh * gw
        B = _log(rng, 1, max(1, min(8, most // (H * rows * keys))))
        if kind == "attention":
            c = _attention("", B, H, gh, gw, L, R, d, layout)
        elif kind == "spatial":
            text = rng.choice(["prefix", "prefix", "mask", "lse"])
            if dtype == "f32" and text == "lse":
                text = "prefix"
            blocks = rng.randint(1, 3) if 3 * B * H * rows * keys <= most else 1
            c = _spatial("", dtype, B, H, gh, gw, L, R, d, text, blocks, layout)
        else:
            D = rng.choice([128, 768, 1000, 3072])
            if kind == "scores":
                c = _scores("", dtype, B, H, gh, gw, L, R, d, D)
            else:
                M = gh * gw
                c = _transition("", dtype, B, H, gh, gw, L, R, d, D, rng.randint(M // 8, M // 2),
                                rng.choice(["nearest", "bilinear"]))
    del c["name"]
    return c


# ----------------------------------------------------------------- inputs --
def _dtype(c):
    return torch.bfloat16 if c["dtype"] == "bf16" else torch.float32


def _empty(*shape, dtype=torch.float32):
    return torch.empty(*shape, dtype=dtype, device=DEV)


def _place(x, layout):
    """[B,H,N,d] contiguous, or a view of a token-major [B,N,H,d] projection."""
    if layout == "tokens":
        return x.transpose(1, 2).contiguous().transpose(1, 2)
    return x.contiguous()


def _qk(g, c, rows):
    """Queries of the image tokens (rows = "image") or of the whole sequence,
    and the keys, text first: N(0,1) with a few regions of the image shifted
    towards single text keys, scaled to logits of standard deviation 3."""
    B, H, gh, gw, L, R, d = (c[x] for x in ("B", "H", "gh", "gw", "L", "R", "d"))
    M = gh * gw
    q = torch.randn(B, H, M, d, generator=g, device=DEV)
    k = torch.randn(B, H, L + M + R, d, generator=g, device=DEV)
    ys = torch.arange(M, device=DEV) // gw + 0.5
    xs = torch.arange(M, device=DEV) % gw + 0.5
    at = torch.rand(B, 3, 3, generator=g, device=DEV)
    for b in range(B):
        for cy, cx, j in at[b].tolist():
            env = torch.exp(-((ys - cy * gh) ** 2 + (xs - cx * gw) ** 2) / 8.0)
            kt = F.normalize(k[b, :, min(L - 1, int(j * L))], dim=-1)
            q[b] += 1.5 * math.sqrt(d) * env[None, :, None] * kt[:, None, :]
    if rows == "all":
        q = torch.cat([torch.randn(B, H, L, d, generator=g, device=DEV), q,
                       torch.randn(B, H, R, d, generator=g, device=DEV)], dim=2)
    s = torch.einsum("hnd,hkd->hnk", q[0, :, :: max(1, q.shape[2] // 64)], k[0]) / math.sqrt(d)
    f = torch.sqrt(3.0 / s.std())
    return q * f, k * f


def _field(g, B, gh, gw):
    """A smooth field in [0,1] per element, [B, gh*gw]."""
    f = torch.randn(B, 1, 8, 8, generator=g, device=DEV)
    f = F.interpolate(f, size=(gh, gw), mode="bicubic", align_corners=True).reshape(B, gh * gw)
    lo, hi = f.amin(1, keepdim=True), f.amax(1, keepdim=True)
    return (f - lo) / (hi - lo)


def _hidden(g, c):
    B, M, D = c["B"], c["gh"] * c["gw"], c["D"]
    hp = torch.randn(B, M, D, generator=g, device=DEV)
    step = 0.05 + 0.5 * _field(g, B, c["gh"], c["gw"])[..., None]
    ht = hp + step * torch.randn(B, M, D, generator=g, device=DEV)
    return ht.to(_dtype(c)), hp.to(_dtype(c))


def _mixed_tokens(gh, gw):
    m = (gh // 2) * (gw // 2)
    return m + 3 * (m // 2)


def _mixed_frame(g, B, gh, gw):
    """Positions and spans of the packed sequence that a first transition left
    on a gh x gw frame: half of its tokens expanded, in raster order."""
    h, w = gh // 2, gw // 2
    m, k = h * w, (h * w) // 2
    order = torch.rand(B, m, generator=g, device=DEV).argsort(1)
    sel = torch.zeros(B, m, dtype=torch.bool, device=DEV).scatter_(1, order[:, :k], True)
    pos, span = [], []
    y, x = torch.arange(m, device=DEV) // w * 2, torch.arange(m, device=DEV) % w * 2
    yx = torch.stack([y, x], 1)
    child = torch.tensor([[0, 0], [0, 1], [1, 0], [1, 1]], device=DEV)
    for b in range(B):
        n = torch.where(sel[b], 4, 1)
        src = torch.repeat_interleave(torch.arange(m, device=DEV), n)
        sub = torch.arange(src.numel(), device=DEV) - (torch.cumsum(n, 0) - n)[src]
        pos.append(yx[src] + child[sub] * sel[b][src][:, None])
        span.append(torch.where(sel[b][src], 1, 2))
    return (torch.stack(pos).to(torch.int32).contiguous(),
            torch.stack(span).to(torch.int32).contiguous())


class State:
    def __init__(self, case, seed):
        self.case = case
        self.g = torch.Generator(device=DEV)
        self.g.manual_seed(int(seed))


def _prepare_transition(s):
    c, g, dt = s.case, s.g, _dtype(s.case)
    M = c["gh"] * c["gw"]
    q, k = _qk(g, c, "image")
    ht, hp = _hidden(g, c)
    lat = torch.randn(c["B"], M, c["C"] * 4, generator=g, device=DEV).to(dt)
    tr = Transition(name="case", dtype=c["dtype"], B=c["B"], H=c["H"], M=M, L=c["L"], R=c["R"],
                    d=c["d"], D=c["D"], C=c["C"], grid_h=c["gh"], grid_w=c["gw"], k=c["k"],
                    alpha=ALPHA, mode=c["mode"], softmax_scale=1.0 / math.sqrt(c["d"]), q_img=None,
                    k_all=None, h_t=None, h_prev=None, latent=None, frame_h=c["gh"],
                    frame_w=c["gw"])
    s.t = TransitionBuffers(tr, inputs=False)
    s.t.set_inputs(q.to(dt), k.to(dt), ht, hp, lat)


def _prepare_scores(s):
    c, dt = s.case, _dtype(s.case)
    q, k = _qk(s.g, c, "image")
    s.q, s.k = q.to(dt), k.to(dt)
    s.h_t, s.h_prev = _hidden(s.g, c)
    s.A, s.V = _empty(c["B"], c["gh"] * c["gw"]), _empty(c["B"], c["gh"] * c["gw"])
    s.ws = av.SpatialWorkspace(DEV)


def _prepare_spatial(s):
    c, g, dt = s.case, s.g, _dtype(s.case)
    M, n = c["gh"] * c["gw"], c["L"] + c["gh"] * c["gw"] + c["R"]
    s.q, s.k, s.lse_all, s.mask = [], [], [], None
    for _ in range(c["blocks"]):
        q, k = _qk(g, c, "image")
        s.q.append(_place(q.to(dt), c["layout"]))
        s.k.append(_place(k.to(dt), c["layout"]))
        if c["text"] == "lse":   # what the model's own attention returns
            s.lse_all.append(torch.stack([
                torch.stack([torch.logsumexp(s.q[-1][b, h].float() @ s.k[-1][b, h].float().T /
                                             math.sqrt(c["d"]), dim=-1)
                             for h in range(c["H"])]) for b in range(c["B"])]).contiguous())
    if c["text"] == "mask":   # four runs of text keys among the image keys
        s.mask = torch.zeros(c["B"], n, dtype=torch.uint8, device=DEV)
        for b in range(c["B"]):
            for f in torch.rand(4, generator=g, device=DEV).tolist():
                a = int(f * (n - c["L"] // 4))
                s.mask[b, a:a + c["L"] // 4] = 1
    s.A = _empty(c["B"], M)
    s.ws = av.SpatialWorkspace(DEV)


def _prepare_attention(s):
    c, dt = s.case, _dtype(s.case)
    q, k = _qk(s.g, c, "all")
    v = torch.randn(*k.shape, generator=s.g, device=DEV)
    s.q, s.k, s.v = (_place(x.to(dt), c["layout"]) for x in (q, k, v))
    s.o = torch.empty_like(s.q)
    n = s.q.shape[2]
    s.lse, s.A = _empty(c["B"], c["H"], n, 2), _empty(c["B"], n)
    s.ws = av.SpatialWorkspace(DEV)


def _prepare_variance(s):
    c = s.case
    h = torch.randn(c["B"], c["N"], c["D"], generator=s.g, device=DEV)
    step = 0.05 + 0.5 * torch.rand(c["B"], c["N"], 1, generator=s.g, device=DEV)
    s.snaps = []
    for _ in range(c["n_t"]):
        s.snaps.append(h.to(_dtype(c)))
        h = h + step * torch.randn(c["B"], c["N"], c["D"], generator=s.g, device=DEV)
    s.V = _empty(c["B"], c["N"])


def _prepare_tail(s):
    c, g, dt = s.case, s.g, _dtype(s.case)
    B, gh, gw, C, k = c["B"], c["gh"], c["gw"], c["C"], c["k"]
    s.mode = av.BILINEAR if c["mode"] == "bilinear" else av.NEAREST
    if c["mixed"]:
        s.pos_in, s.span_in = _mixed_frame(g, B, gh, gw)
        M = s.span_in.shape[1]
    else:
        s.pos_in, s.span_in, M = None, None, gh * gw
    # a long-tailed spatial score and a smooth temporal one, per token
    s.A0 = torch.exp(torch.randn(B, M, generator=g, device=DEV) - 3.0)
    field = _field(g, B, 32, 32)
    at = torch.linspace(0, 1023, M, device=DEV).long()
    s.V0 = 0.05 + 0.5 * field[:, at] + 0.02 * torch.rand(B, M, generator=g, device=DEV)
    s.latent = torch.randn(B, M, C * 4, generator=g, device=DEV).to(dt)
    n = M + 3 * k
    i32 = dict(dtype=torch.int32)
    s.S, s.sel_idx = _empty(B, M), _empty(B, k, **i32)
    s.sel_mask, s.tok_offset = _empty(B, M, dtype=torch.uint8), _empty(B, M, **i32)
    s.mixed, s.pos, s.span = _empty(B, n, C * 4, dtype=dt), _empty(B, n, 2, **i32), _empty(B, n, **i32)
    s.src_tok, s.src_sub = _empty(B, n, **i32), _empty(B, n, dtype=torch.int8)
    s.full = _empty(B, 4 * gh * gw, C * 4, dtype=dt)
    s.merge_ws = torch.zeros(av.avits_merge_final_workspace(s.mode, B, 2 * gh, 2 * gw),
                             dtype=torch.uint8, device=DEV)
    need = av.avits_selective_upsample_workspace(s.mode, B, gh, gw)
    s.up_ws = _empty(need, dtype=torch.uint8) if need and c["mixed"] else None


def prepare(case, seed):
    s = State(case, seed)
    globals()["_prepare_" + case["kind"]](s)
    del s.g
    return s


# -------------------------------------------------------------------- run --
def _run_transition(s):
    t = s.t
    t.run()
    return {"A": t.A, "V": t.V, "S": t.S, "sel_idx": t.sel_idx, "sel_mask": t.sel_mask,
            "tok_offset": t.tok_offset, "mixed": t.mixed, "pos": t.pos, "span": t.span,
            "src_tok": t.src_tok, "src_sub": t.src_sub, "full": t.full}


def _run_scores(s):
    av.avits_score_spatiotemporal(s.q, s.k, s.case["L"], 1.0 / math.sqrt(s.case["d"]), s.A, s.h_t,
                                  s.h_prev, s.V, workspace=s.ws)
    return {"A": s.A, "V": s.V}


def _run_spatial(s):
    c = s.case
    scale, w = 1.0 / math.sqrt(c["d"]), 1.0 / c["blocks"]
    for i, (q, k) in enumerate(zip(s.q, s.k)):
        if c["text"] == "lse":
            av.avits_score_spatial_lse(q, k[:, :, :c["L"]], s.lse_all[i], scale, s.A, weight=w,
                                       accumulate=i > 0, workspace=s.ws)
        else:
            av.avits_score_spatial(q, k, c["L"], scale, s.A, weight=w, accumulate=i > 0,
                                   workspace=s.ws, text_mask=s.mask)
    return {"A": s.A}


def _run_attention(s):
    av.avits_attention_forward(s.q, s.k, s.v, s.case["L"], 1.0 / math.sqrt(s.case["d"]), s.o,
                               lse=s.lse, A=s.A, workspace=s.ws)
    return {"o": s.o, "lse": s.lse, "A": s.A}


def _run_variance(s):
    av.avits_score_temporal_var(s.snaps, s.V)
    return {"V": s.V}


def _run_tail(s):
    c = s.case
    av.avits_select_upsample(s.A0, s.V0, ALPHA, c["k"], s.sel_idx, s.tok_offset, s.sel_mask,
                             s.latent, c["gh"], c["gw"], s.mixed, s.pos, s.span, s.src_tok,
                             s.src_sub, S=s.S, mode=s.mode, pos_in=s.pos_in, span_in=s.span_in,
                             workspace=s.up_ws)
    av.avits_merge_final(s.mixed, s.pos, s.span, 2 * c["gh"], 2 * c["gw"], s.full, mode=s.mode,
                         workspace=s.merge_ws)
    return {"S": s.S, "sel_idx": s.sel_idx, "sel_mask": s.sel_mask, "tok_offset": s.tok_offset,
            "mixed": s.mixed, "pos": s.pos, "span": s.span, "src_tok": s.src_tok,
            "src_sub": s.src_sub, "full": s.full}


def run(state):
    return globals()["_run_" + state.case["kind"]](state)


# ------------------------------------------------------------------- work --
def _elt(c):
    return 2 if c["dtype"] == "bf16" else 4


def _work_spatial(c):
    M, n = c["gh"] * c["gw"], c["L"] + c["gh"] * c["gw"] + c["R"]
    keys, extra = n, 0
    if c.get("text") == "lse":
        keys, extra = c["L"], c["B"] * c["H"] * M * 4
    elif c.get("text") == "mask":
        extra = c["B"] * n
    bh = c["B"] * c["H"]
    one = dict(bytes=bh * (M + keys) * c["d"] * _elt(c) + extra + 4 * c["B"] * M,
               flops=2 * bh * M * keys * c["d"])
    return {x: v * c.get("blocks", 1) for x, v in one.items()}


def _work_scores(c):
    w, n = _work_spatial(c), c["B"] * c["gh"] * c["gw"]
    return dict(bytes=w["bytes"] + n * (2 * c["D"] * _elt(c) + 4), flops=w["flops"] + 5 * n * c["D"])


def _work_attention(c):
    n, bh = c["L"] + c["gh"] * c["gw"] + c["R"], c["B"] * c["H"]
    return dict(bytes=bh * n * (4 * c["d"] * 2 + 8) + 4 * c["B"] * n, flops=4 * bh * n * n * c["d"])


def _work_variance(c):
    n = c["B"] * c["N"]
    return dict(bytes=n * (c["n_t"] * c["D"] * _elt(c) + 4), flops=4 * n * c["D"] * c["n_t"])


def _work_tail(c):
    """Scores and latent in, selection, packed sequence and full frame out (the
    packed sequence is the merge's input as well: written once, read once)."""
    M = _mixed_tokens(c["gh"], c["gw"]) if c.get("mixed") else c["gh"] * c["gw"]
    n, tok = M + 3 * c["k"], c["C"] * 4 * _elt(c)
    sel = M * (8 + 4 + 1 + 4) + 4 * c["k"] + (12 * M if c.get("mixed") else 0)
    frame = 4 * c["gh"] * c["gw"] * tok
    taps = 8 if c["mode"] == "bilinear" else 0
    return dict(bytes=c["B"] * (sel + M * tok + n * (2 * tok + 17 + 12) + frame),
                flops=c["B"] * (8 * M + taps * (n + 4 * c["gh"] * c["gw"]) * c["C"] * 4))


def _work_transition(c):
    a, b = _work_scores(c), _work_tail(c)
    return {x: a[x] + b[x] for x in a}


def work(case):
    return globals()["_work_" + case["kind"]](case)


# -------------------------------------------------------------- tolerance --
def tolerance(case):
    """Selections, copies and the bilinear weights are fixed operations in a
    fixed order.  The scores are fp32 sums of fp32 exponentials; the attention
    rounds the probabilities and the output to bf16."""
    if case["kind"] == "tail":
        return "exact"
    if case["kind"] == "attention":
        return {"rel": 1e-2, "max": 1e-1}
    if case["kind"] == "transition":   # a near-tie may fall the other way
        return {"rel": 1e-5, "max": 1e-4, "differ": 0.005}
    return {"rel": 1e-5, "max": 1e-4}


# ------------------------------------------------------------------ exact --
def _mass(q, k, text, scale, lse_all=None, rows=1024):
    """Mean over heads of the text keys' softmax mass, [M] in 64 bits; text:
    the indices of the text keys of k ([H,N,d])."""
    out = torch.zeros(q.shape[1], dtype=torch.float64, device=DEV)
    for h in range(q.shape[0]):
        kd = k[h].double()
        for a in range(0, q.shape[1], rows):
            s = q[h, a:a + rows].double() @ kd.T * scale
            whole = torch.logsumexp(s, 1) if lse_all is None else lse_all[h, a:a + rows].double()
            out[a:a + rows] += torch.exp(torch.logsumexp(s[:, text], 1) - whole)
    return out / q.shape[0]


def _exact_scores_of(c, q, k, h_t, h_prev):
    text = torch.arange(c["L"], device=DEV)
    A = torch.stack([_mass(q[b], k[b], text, 1.0 / math.sqrt(c["d"])) for b in range(c["B"])])
    t, p = h_t.double(), h_prev.double()
    return A, (t - p).norm(dim=-1) / (p.norm(dim=-1) + 1e-6)


def _exact_scores(s):
    A, V = _exact_scores_of(s.case, s.q, s.k, s.h_t, s.h_prev)
    return {"A": A, "V": V}


def _exact_spatial(s):
    c, scale = s.case, 1.0 / math.sqrt(s.case["d"])
    A = torch.zeros(c["B"], c["gh"] * c["gw"], dtype=torch.float64, device=DEV)
    for i, (q, k) in enumerate(zip(s.q, s.k)):
        for b in range(c["B"]):
            text = torch.arange(c["L"], device=DEV)
            if c["text"] == "mask":
                text = s.mask[b].nonzero()[:, 0]
            if c["text"] == "lse":
                A[b] += _mass(q[b], k[b, :, :c["L"]], text, scale, s.lse_all[i][b])
            else:
                A[b] += _mass(q[b], k[b], text, scale)
    return {"A": A / c["blocks"]}


def _exact_attention(s):
    c, scale, L = s.case, 1.0 / math.sqrt(s.case["d"]), s.case["L"]
    B, H, n, d = s.q.shape
    o = torch.empty(B, H, n, d, dtype=torch.float64, device=DEV)
    lse = torch.empty(B, H, n, 2, dtype=torch.float64, device=DEV)
    for b in range(B):
        for h in range(H):
            kd, vd = s.k[b, h].double(), s.v[b, h].double()
            x = s.q[b, h].double() @ kd.T * scale
            lse[b, h, :, 0], lse[b, h, :, 1] = torch.logsumexp(x, 1), torch.logsumexp(x[:, :L], 1)
            o[b, h] = torch.softmax(x, 1) @ vd
    return {"o": o, "lse": lse, "A": torch.exp(lse[..., 1] - lse[..., 0]).mean(1)}


def _exact_variance(s):
    z = torch.stack([x.double() for x in s.snaps])
    return {"V": z.var(dim=0, unbiased=True).mean(-1)}


def _fused(A, V):
    def norm(x):
        lo, hi = x.amin(1, keepdim=True), x.amax(1, keepdim=True)
        return (x - lo) / ((hi - lo) + 1e-6)
    return ALPHA * norm(A) + (1 - ALPHA) * norm(V)


def _pixels(tok, gh, gw, C):
    """[M, C*4] tokens of a gh x gw grid -> [C, 2gh, 2gw] pixels."""
    return tok.view(gh, gw, C, 2, 2).permute(2, 0, 3, 1, 4).reshape(C, 2 * gh, 2 * gw)


def _tokens(pix, gh, gw):
    return pix.view(-1, gh, 2, gw, 2).permute(1, 3, 0, 2, 4).reshape(gh * gw, -1)


def _resize(pix, mode):
    if mode == "nearest":
        return pix.repeat_interleave(2, 1).repeat_interleave(2, 2)
    return F.interpolate(pix[None], scale_factor=2, mode="bilinear", align_corners=False)[0]


def _exact_tail_of(c, latent, sel):
    """The packed sequence and the merged frame of a dense grid in 64 bits;
    sel [B,M]: the selected tokens."""
    gh, gw, C = c["gh"], c["gw"], c["C"]
    mixed, full = [], []
    M = gh * gw
    cell = torch.arange(4 * M, device=DEV)
    Y, X = cell // (2 * gw), cell % (2 * gw)
    parent = (Y // 2) * gw + X // 2
    first = (2 * (torch.arange(M, device=DEV) // gw)) * 2 * gw + 2 * (torch.arange(M, device=DEV) % gw)
    for b in range(latent.shape[0]):
        lat = latent[b].double()
        up = _tokens(_resize(_pixels(lat, gh, gw, C), c["mode"]), 2 * gh, 2 * gw)
        n = torch.where(sel[b], 4, 1)
        src = torch.repeat_interleave(torch.arange(M, device=DEV), n)
        sub = torch.arange(src.numel(), device=DEV) - (torch.cumsum(n, 0) - n)[src]
        kids = up[first[src] + (sub // 2) * 2 * gw + sub % 2]
        mixed.append(torch.where(sel[b][src][:, None], kids, lat[src]))
        low = F.avg_pool2d(_pixels(up, 2 * gh, 2 * gw, C)[None], 2)[0]
        low = torch.where(sel[b][:, None], _tokens(low, gh, gw), lat)
        wide = _tokens(_resize(_pixels(low, gh, gw, C), c["mode"]), 2 * gh, 2 * gw)
        full.append(torch.where(sel[b][parent][:, None], up, wide))
    return torch.stack(mixed), torch.stack(full)


def _topk(S, k):
    order = torch.sort(S, dim=1, descending=True, stable=True).indices
    return torch.zeros_like(S, dtype=torch.bool).scatter_(1, order[:, :k], True)


def _exact_tail(s):
    out = dict.fromkeys(("S", "sel_idx", "sel_mask", "tok_offset", "mixed", "pos", "span", "src_tok",
                         "src_sub", "full"))
    out["S"] = _fused(s.A0.double(), s.V0.double())
    if not s.case["mixed"]:
        out["mixed"], out["full"] = _exact_tail_of(s.case, s.latent,
                                                   _topk(_fused(s.A0, s.V0), s.case["k"]))
    return out


def _exact_transition(s):
    c, t = s.case, s.t
    out = dict.fromkeys(("A", "V", "S", "sel_idx", "sel_mask", "tok_offset", "mixed", "pos", "span",
                         "src_tok", "src_sub", "full"))
    out["A"], out["V"] = _exact_scores_of(c, t.q, t.k, t.h_t, t.h_prev)
    out["S"] = _fused(out["A"], out["V"])
    if c["mode"] == "nearest":   # the merged frame does not depend on the selection
        out["full"] = _exact_tail_of(c, t.latent, _topk(out["S"], c["k"]))[1]
    return out


def exact(case, seed):
    return globals()["_exact_" + case["kind"]](prepare(case, seed))
