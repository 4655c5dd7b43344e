"""Performance cases of the Q-Render library: what a user's program has it do,
through its public entry points, over the range of scene sizes, image sizes,
feature widths, storage formats and select rules it is used with.

Eight kinds of work (a case's "kind"):

  frame      one whole Q-Render frame (qr_render) into buffers kept from frame
             to frame, as a viewer or an evaluation loop renders
  select     one select rule (qr_select / qr_select_rule) on a frame that is
             already projected and sorted, as a comparison of rules runs it
  dense      the Eq. 1 blend of every intersecting Gaussian (qr_dense)
  backward   cosine loss and its gradients of a rendered frame (qr_cosine_backward)
  train      one differentiable training step with the Eq. 2 loss through
             autograd (quantile_render, qr_contrastive_loss, backward)
  relevance  open-vocabulary scores of a view against text queries, with the
             map written (qr_relevance) or not (qr_blend_relevance)
  views      many views of several scenes in one launch, with scores (Batch.step)
  table      storing a feature table at lower precision (qr_quantize_*)

Scenes are the repository's synthetic stand-ins (scenes.py): the tiny test
scene, the indoor room (few distinct rows, dense lists) and the object seen
from outside (many distinct rows, long lists at the silhouette).
"""
import math

import numpy as np
import torch

from paper_2512_20927_gb300 import autograd as qa
from paper_2512_20927_gb300 import batch as qb
from paper_2512_20927_gb300 import qrender as q
from paper_2512_20927_gb300 import scenes

RULES = {"quantile": q.QR_RULE_QUANTILE, "topk": q.QR_RULE_TOPK,
         "stratified": q.QR_RULE_STRATIFIED, "riemann": q.QR_RULE_RIEMANN}


def listed():
    return [
        # the smallest call: a few thousand Gaussians into a thumbnail with
        # short features; launches and latency are all there is
        dict(name="frame-tiny", kind="frame", scene="tiny", n=2000, width=128, height=128,
             channels=16, dtype="f32", K=8),
        # the headline frame: an indoor room at VGA with 512-D FP32 features
        dict(name="frame-room", kind="frame", scene="room", n=500_000, width=640, height=480,
             channels=512, dtype="f32", K=8),
        # an object-centric frame: long per-tile lists, a distinct row for
        # nearly every pixel
        dict(name="frame-object", kind="frame", scene="object", n=500_000, width=640, height=480,
             channels=512, dtype="f32", K=8),
        # the largest single frame: 1M Gaussians at ScanNet's full resolution,
        # FP8 feature table
        dict(name="frame-large-fp8", kind="frame", scene="room", n=1_000_000, width=1296,
             height=968, channels=512, dtype="fp8", K=8),
        # the paper's alternative rules: Stratified-K on the room ...
        dict(name="select-stratified", kind="select", scene="room", n=500_000, width=640,
             height=480, K=8, rule="stratified"),
        # ... and top-K with more kept Gaussians, on a ragged view of the object
        dict(name="select-topk-ragged", kind="select", scene="object", n=200_000, width=517,
             height=389, K=16, rule="topk"),
        # the plain method every frame is compared with
        dict(name="dense-room", kind="dense", scene="room", n=500_000, width=640, height=480,
             channels=512, dtype="f32"),
        # loss and gradients of a rendered training view, BF16 features
        dict(name="backward-cosine", kind="backward", scene="room", n=300_000, width=640,
             height=480, channels=512, dtype="bf16", K=8),
        # a whole training step with the paper's contrastive loss over 32 patches
        dict(name="train-eq2", kind="train", scene="room", n=300_000, width=640, height=480,
             channels=512, dtype="bf16", K=8, masks=32),
        # scores of a view against 64 text queries without writing the map
        dict(name="relevance-fused", kind="relevance", scene="room", n=500_000, width=640,
             height=480, channels=512, dtype="f32", K=8, queries=64, fused=True),
        # evaluation of several scenes: views of many sizes in one launch, with scores
        dict(name="views", kind="views", scenes=2, n=200_000, views=8, seed_views=0,
             channels=512, dtype="bf16", K=8, queries=64),
        # compressing a scene's feature table
        dict(name="table-fp8", kind="table", n=500_000, channels=512, dtype="fp8"),
    ]


def _log(rng, lo, hi):
    return int(round(math.exp(rng.uniform(math.log(lo), math.log(hi)))))


def draw(rng):
    kind = rng.choice(["frame", "frame", "frame", "select", "dense", "backward", "train",
                       "relevance", "views", "table"])
    scene = rng.choice(["room", "object"])
    width = _log(rng, 97, 800)
    height = max(61, int(width * rng.uniform(0.6, 1.0)))
    n = _log(rng, 10_000, 600_000)
    dtype = rng.choice(["f32", "bf16", "fp8"])
    if kind == "frame":
        if rng.random() < 0.3:
            return dict(kind=kind, scene="tiny", n=_log(rng, 500, 20_000),
                        width=rng.randint(40, 200), height=rng.randint(40, 200),
                        channels=rng.choice([16, 32, 64, 128]), dtype=dtype,
                        K=rng.choice([1, 4, 8, 16]))
        return dict(kind=kind, scene=scene, n=n, width=width, height=height,
                    channels=rng.choice([64, 256, 512, 512]), dtype=dtype,
                    K=rng.choice([4, 8, 8, 16, 32]))
    if kind == "select":
        return dict(kind=kind, scene=scene, n=n, width=width, height=height,
                    K=rng.choice([2, 4, 8, 8, 16, 32]), rule=rng.choice(sorted(RULES)))
    if kind == "dense":
        return dict(kind=kind, scene=scene, n=min(n, 300_000), width=min(width, 640),
                    height=min(height, 480), channels=rng.choice([64, 128, 256, 512, 512]),
                    dtype=dtype)
    if kind in ("backward", "train"):
        c = dict(kind=kind, scene=scene, n=min(n, 300_000), width=min(width, 640),
                 height=min(height, 480), channels=rng.choice([128, 256, 512]),
                 dtype=rng.choice(["f32", "bf16"]), K=rng.choice([4, 8, 8, 16]))
        return c if kind == "backward" else dict(c, masks=rng.randint(2, 48))
    if kind == "relevance":
        return dict(kind=kind, scene=scene, n=n, width=width, height=height,
                    channels=rng.choice([128, 256, 512]), dtype=dtype, K=rng.choice([4, 8]),
                    queries=rng.choice([16, 32, 64, 128]), fused=rng.random() < 0.5)
    if kind == "views":
        return dict(kind=kind, scenes=rng.randint(1, 2), n=_log(rng, 50_000, 200_000),
                    views=rng.randint(2, 6), seed_views=rng.randint(1, 1000),
                    channels=512 if dtype == "fp8" else rng.choice([256, 512]), dtype=dtype,
                    K=rng.choice([4, 8, 16]), queries=rng.choice([32, 64]))
    return dict(kind="table", n=_log(rng, 1000, 500_000),
                channels=rng.choice([16, 128, 384, 512]), dtype=rng.choice(["bf16", "fp8"]))


# ---------------------------------------------------------------- inputs
def _features(n, channels, seed, unit=True):
    """CLIP-like rows: N(0, 1), unit length (drawn on the GPU)."""
    gen = torch.Generator(device="cuda").manual_seed(seed)
    f = torch.randn((n, channels), generator=gen, device="cuda")
    return torch.nn.functional.normalize(f, dim=1) if unit else f


def _store(f, dtype):
    """(table, scale) of a float32 table: scale is None but for FP8."""
    if dtype == "f32":
        return f, None
    if dtype == "bf16":
        return f.to(torch.bfloat16), None
    s = f.abs().amax(1) / 448.0
    s = torch.where(s > 0, s, torch.ones_like(s))
    return (f / s[:, None]).clamp(-448, 448).to(torch.float8_e4m3fn).view(torch.uint8), s


def _gaussians(scene, n, seed):
    rng = np.random.default_rng(seed)
    if scene == "tiny":
        return scenes.tiny_scene(seed, n, 1)[0]
    if scene == "room":
        return scenes.room_gaussians(rng, n)
    return scenes.object_scene(seed, n, 1)[0]


def _camera(scene, width, height):
    return {"tiny": scenes.tiny_camera, "room": scenes.room_camera,
            "object": scenes.object_camera}[scene](width, height)


class _Inputs:
    """What both the library and the plain evaluation below start from."""

    def __init__(self, case, seed):
        g = _gaussians(case["scene"], case["n"], seed)
        self.cam = _camera(case["scene"], case["width"], case["height"])
        self.g = tuple(torch.from_numpy(np.ascontiguousarray(a, np.float32)).cuda()
                       for a in (g.mean, g.log_scale, g.quat, g.opacity))
        self.P = case["width"] * case["height"]
        self.table = self.scale = None
        if "channels" in case:
            f = _features(case["n"], case["channels"], seed + 1, case["scene"] != "tiny")
            self.table, self.scale = _store(f, case["dtype"])
        m = case.get("masks", 24)
        if case["kind"] in ("backward", "train"):
            self.mask = torch.from_numpy(scenes.patch_masks(case["width"], case["height"], m,
                                                            seed)).cuda()
            self.targets = _features(m, case["channels"], seed + 2)
        if case["kind"] == "backward":
            # every pixel is pulled towards its patch's embedding
            self.target = self.targets[self.mask.clamp(min=0).long()].contiguous()
        if case["kind"] == "relevance":
            self.queries = _features(case["queries"], case["channels"], seed + 3).to(torch.bfloat16)


def _frame(inp, K):
    """A frame with room for a quarter more intersections than the view has."""
    params = q.default_params(K)
    n = int(inp.g[0].shape[0])
    found = q.render_frame(inp.g, None, inp.cam, K=K)["n_isect"]
    fr = q.frame_create(n, inp.cam, params, int(found * 1.25) + 4096)
    q.qr_project(fr, *inp.g)
    q.qr_sort(fr)
    return fr


def _selection(fr):
    return (torch.empty((fr.pixels, fr.K), dtype=torch.int32, device="cuda"),
            torch.empty((fr.pixels, fr.K), dtype=torch.float32, device="cuda"),
            torch.empty(fr.pixels, dtype=torch.uint8, device="cuda"))


def prepare(case, seed):
    kind = case["kind"]
    s = {"case": case}
    if kind == "table":
        s["x"] = _features(case["n"], case["channels"], seed)
        return s
    if kind == "views":
        made = []
        for i in range(case["scenes"]):
            n = case["n"] * (i + 1)
            g = _gaussians("room", n, seed + 10 * i)
            table, scale = _store(_features(n, case["channels"], seed + 10 * i + 1), case["dtype"])
            made.append(qb.Scene(q.gaussians_to_device(g),
                                 table if scale is None else (table, scale)))
        views = scenes.batched_views(case["seed_views"], case["views"], case["scenes"])
        qs = _features(case["queries"], case["channels"], seed + 3).to(torch.bfloat16)
        s["batch"] = qb.Batch(made, views, K=case["K"], queries=qs.view(torch.int16))
        return s
    inp = s["in"] = _Inputs(case, seed)
    if kind == "train":
        s["features"] = inp.table.requires_grad_(True)
        s["opacity"] = inp.g[3].clone().requires_grad_(True)
        return s
    fr = s["frame"] = _frame(inp, case.get("K", 8))
    if kind == "dense":
        s["out"] = torch.empty((inp.P, case["channels"]), device="cuda")
        s["T"] = torch.empty(inp.P, device="cuda")
        return s
    ids, w, cnt = s["sel"] = _selection(fr)
    if kind == "select":
        s["tau"] = (torch.empty((inp.P, fr.K), device="cuda") if case["rule"] == "stratified"
                    else None)
        return s
    if kind != "frame":
        q.qr_select(fr, ids, w, cnt)
    if kind != "relevance" or not case["fused"]:
        s["out"] = torch.empty((inp.P, case["channels"]), device="cuda")
        if kind != "frame":
            q.qr_blend(inp.table, inp.scale, ids, w, cnt, s["out"])
    return s


def run(s):
    case = s["case"]
    kind = case["kind"]
    if kind == "table":
        return (q.qr_quantize_bf16(s["x"]) if case["dtype"] == "bf16"
                else q.qr_quantize_fp8(s["x"]))
    if kind == "views":
        b = s["batch"]
        b.step()
        return {"out": b.out, "ids": b.ids, "weights": b.weights, "counts": b.counts,
                "scores": b.scores}
    inp = s["in"]
    if kind == "train":
        mean, log_scale, quat, _ = inp.g
        fmap, counts = qa.quantile_render(mean, log_scale, quat, s["opacity"], s["features"],
                                          inp.cam, K=case["K"])
        loss, grad = q.qr_contrastive_loss(fmap.detach().view(inp.P, -1), inp.targets, inp.mask)
        gf, go = torch.autograd.grad(fmap, (s["features"], s["opacity"]), grad.view_as(fmap))
        return {"map": fmap.detach(), "counts": counts, "loss": loss, "grad_features": gf,
                "grad_opacity": go}
    fr = s["frame"]
    if kind == "dense":
        q.qr_dense(fr, inp.table, inp.scale, s["out"], s["T"])
        return {"out": s["out"], "T": s["T"]}
    ids, w, cnt = s["sel"]
    if kind == "select":
        if case["rule"] == "quantile":
            q.qr_select(fr, ids, w, cnt)
        else:
            q.qr_select_rule(fr, RULES[case["rule"]], ids, w, cnt, s["tau"])
        return {"ids": ids, "weights": w, "counts": cnt, "tau": s["tau"]}
    if kind == "frame":
        q.qr_render(fr, *inp.g, inp.table, inp.scale, ids, w, cnt, s["out"])
        return {"out": s["out"], "ids": ids, "weights": w, "counts": cnt}
    if kind == "backward":
        loss, gmap, gf, ga, gc = q.qr_cosine_backward(fr, inp.table, inp.scale, ids, w, cnt,
                                                      s["out"], inp.target)
        return {"loss": loss, "grad_map": gmap, "grad_features": gf, "grad_opacity": ga,
                "grad_conic": gc}
    if case["fused"]:
        return {"scores": q.qr_blend_relevance(inp.table, inp.scale, ids, w, cnt, inp.queries,
                                               width=case["width"])[0]}
    return {"scores": q.qr_relevance(s["out"], inp.queries)[0]}


# Distinct feature rows a frame's pixels select, as a share of the Gaussians
# (measured: 840 of 500k for the room, 49,658 of 500k for the object at VGA).
ROWS = {"tiny": 0.5, "room": 0.002, "object": 0.1}
# Blended Gaussians per pixel of the dense walk (measured: 68 for the room).
MEMBERS = 68


def work(case):
    kind = case["kind"]
    es = {"f32": 4, "bf16": 2, "fp8": 1}[case.get("dtype", "f32")]
    C, K = case.get("channels", 0), case.get("K", 8)
    if kind == "table":
        n = case["n"] * C
        return {"bytes": n * (4 + es), "flops": n}
    if kind == "views":
        px = [v.width * v.height for _, v in
              scenes.batched_views(case["seed_views"], case["views"], case["scenes"])]
        P, Q = sum(px), case["queries"]
        n = case["n"] * case["views"] * (case["scenes"] + 1) / 2
        # every Gaussian's parameters and the map's write and read by the scores
        return {"bytes": 44 * n + P * (8 * C + 8 * K + 1 + 4 * Q), "flops": 2.0 * P * C * (K + Q)}
    P, n = case["width"] * case["height"], case["n"]
    rows = ROWS[case["scene"]] * n * C * es
    if kind == "frame":
        return {"bytes": 44 * n + rows + P * (4 * C + 8 * K + 1), "flops": 2.0 * P * C * K}
    if kind == "select":
        # the projected records of the Gaussians on screen (a tenth of the room)
        seen = n if case["scene"] == "object" else n // 10
        return {"bytes": 44 * seen + P * (8 * K + 1), "flops": 30.0 * P * MEMBERS}
    if kind == "dense":
        return {"bytes": rows * 10 + P * (4 * C + 4), "flops": 2.0 * P * C * MEMBERS}
    if kind == "relevance":
        Q = case["queries"]
        read = rows + P * (8 * K + 1) if case["fused"] else 4.0 * P * C
        return {"bytes": read + 4.0 * P * Q, "flops": 2.0 * P * C * (Q + (K if case["fused"] else 0))}
    # every gradient row is written, the map's gradient too
    grads = n * (4 * C + 16) + rows
    if kind == "backward":
        return {"bytes": P * (12 * C + 8 * K + 1) + grads, "flops": 4.0 * P * C * K}
    # train: the map and its gradient written, each read once more
    return {"bytes": 44 * n + P * (16 * C + 16 * K + 1) + grads + n * C * es,
            "flops": P * C * (6.0 * K + 4.0 * case["masks"])}


# ---------------------------------------------------------------- 64-bit evaluation
# Plain torch in float64: projection, tile lists, the walks of Eq. 1 and of the
# select rules, blend, losses and their gradients.
ALPHA_MIN, ALPHA_MAX = float(np.float32(1.0 / 255.0)), float(np.float32(0.99))
T_MIN, DILATION = float(np.float32(1e-4)), float(np.float32(0.3))
TILE = 16


class _Exact:
    """Projection and depth-ordered tile lists of one view."""

    def __init__(self, g, cam):
        mean, log_scale, quat, opacity = (x.detach().double() for x in g)
        c = torch.from_numpy(cam.as_array().astype(np.float64)).cuda()
        R, t, fx, fy, cx, cy, near = c[:9].view(3, 3), c[9:12], *c[12:17].tolist()
        self.W, self.H = cam.width, cam.height
        p = mean @ R.T + t
        keep = (p[:, 2] > near) & (opacity >= ALPHA_MIN)
        gid = keep.nonzero()[:, 0]
        p, log_scale, quat, opacity = p[gid], log_scale[gid], quat[gid], opacity[gid]
        w, x, y, z = torch.nn.functional.normalize(quat, dim=1).unbind(1)
        rot = torch.stack([1 - 2 * (y * y + z * z), 2 * (x * y - w * z), 2 * (x * z + w * y),
                           2 * (x * y + w * z), 1 - 2 * (x * x + z * z), 2 * (y * z - w * x),
                           2 * (x * z - w * y), 2 * (y * z + w * x), 1 - 2 * (x * x + y * y)],
                          1).view(-1, 3, 3)
        half = rot * log_scale.exp()[:, None, :]
        iz = 1.0 / p[:, 2]
        J = torch.zeros((len(gid), 2, 3), dtype=torch.float64, device="cuda")
        J[:, 0, 0], J[:, 0, 2] = fx * iz, -fx * p[:, 0] * iz * iz
        J[:, 1, 1], J[:, 1, 2] = fy * iz, -fy * p[:, 1] * iz * iz
        M = J @ R @ half
        S = M @ M.transpose(1, 2)
        s00, s01, s11 = S[:, 0, 0] + DILATION, S[:, 0, 1], S[:, 1, 1] + DILATION
        det = s00 * s11 - s01 * s01
        mx, my = fx * p[:, 0] * iz + cx, fy * p[:, 1] * iz + cy
        r = (2 * (opacity / ALPHA_MIN).log()).clamp(min=0).sqrt()
        ex, ey = r * s00.sqrt() + 1, r * s11.sqrt() + 1
        on = (mx + ex >= 0) & (mx - ex <= self.W) & (my + ey >= 0) & (my - ey <= self.H)
        on = on.nonzero()[:, 0]
        # depth order, equal depths by id
        on = on[torch.argsort(p[on, 2].float(), stable=True)]
        self.gid, self.mean = gid[on], torch.stack([mx, my], 1)[on]
        self.conic = torch.stack([s11 / det, -s01 / det, s00 / det], 1)[on]
        self.alpha = opacity[on]
        tx_n, ty_n = -(-self.W // TILE), -(-self.H // TILE)
        x0 = ((mx - ex)[on] / TILE).floor().clamp(0, tx_n - 1).long()
        x1 = ((mx + ex)[on] / TILE).floor().clamp(0, tx_n - 1).long()
        y0 = ((my - ey)[on] / TILE).floor().clamp(0, ty_n - 1).long()
        y1 = ((my + ey)[on] / TILE).floor().clamp(0, ty_n - 1).long()
        wide, per = x1 - x0 + 1, (x1 - x0 + 1) * (y1 - y0 + 1)
        who = torch.repeat_interleave(torch.arange(len(on), device="cuda"), per)
        at = torch.arange(len(who), device="cuda") - (per.cumsum(0) - per)[who]
        tile = (y0[who] + at // wide[who]) * tx_n + x0[who] + at % wide[who]
        tile, order = torch.sort(tile, stable=True)
        self.entry = who[order]
        length = torch.bincount(tile, minlength=tx_n * ty_n)
        start = length.cumsum(0) - length
        # the longest lists first, so the tiles still walking are a prefix
        length, by = torch.sort(length, descending=True)
        self.start, self.length = start[by], length.tolist()
        i = torch.arange(TILE * TILE, device="cuda")
        px = (by % tx_n * TILE)[:, None] + i % TILE
        py = (by // tx_n * TILE)[:, None] + i // TILE
        self.inside = (px < self.W) & (py < self.H)
        self.pix = (py * self.W + px)[self.inside]
        self.ux, self.uy = px + 0.5, py + 0.5

    def image(self, x):
        out = torch.empty((self.W * self.H,) + x.shape[2:], dtype=x.dtype, device="cuda")
        out[self.pix] = x[self.inside]
        return out

    def steps(self, done):
        """(entries, alpha' or 0, tiles still walking), list position by position."""
        n, i = len(self.length), 0
        while True:
            while n and self.length[n - 1] <= i:
                n -= 1
            if not n or (i % 32 == 0 and bool(done[:n].all())):
                return
            e = self.entry[self.start[:n] + i]
            dx = self.ux[:n] - self.mean[e, 0][:, None]
            dy = self.uy[:n] - self.mean[e, 1][:, None]
            A = self.conic[e][:, None, :]
            qq = A[..., 0] * dx * dx + 2 * A[..., 1] * dx * dy + A[..., 2] * dy * dy
            a = (self.alpha[e][:, None] * torch.exp(-0.5 * qq)).clamp(max=ALPHA_MAX)
            yield e, torch.where(a >= ALPHA_MIN, a, torch.zeros_like(a)), n
            i += 1

    def new(self, *more, fill=0.0, dtype=torch.float64):
        return torch.full(self.inside.shape + more, fill, dtype=dtype, device="cuda")

    def dense(self, visit):
        """Eq. 1's walk: visit(entries, weights, T, blended, n) at each position; the last T."""
        T, done = self.new(fill=1.0), ~self.inside
        for e, a, n in self.steps(done):
            Tt = T[:n] * (1 - a)
            live = (a > 0) & ~done[:n]
            stop = live & (Tt < T_MIN)
            live &= ~stop
            done[:n] |= stop
            w = torch.where(live, T[:n] * a, torch.zeros_like(a))
            T[:n] = torch.where(live, Tt, T[:n])
            visit(e, w, T, live, n)
        return T

    def quantile(self, K, tau=None, count=False):
        """Algorithm 1 with boundaries tau [.., K]: entries [.., K] (-1 padded), weights."""
        if tau is None:
            tau = (1 - torch.arange(1, K + 1, dtype=torch.float64, device="cuda") / (K + 1))
            tau = tau.expand(self.inside.shape + (K,))
        T, TQ, done = self.new(fill=1.0), self.new(fill=1.0), ~self.inside
        k, m = self.new(fill=0, dtype=torch.long), self.new(fill=0, dtype=torch.long)
        ent, wts = self.new(K + 1, fill=-1, dtype=torch.long), self.new(K + 1)
        for e, a, n in self.steps(done):
            Tt = T[:n] * (1 - a)
            live = (a > 0) & ~done[:n]
            nk = (Tt[..., None] < tau[:n]).sum(-1)
            hit = live & (nk > k[:n])
            # entries that are not kept go to the spare last column
            at = torch.where(hit, m[:n], torch.full_like(m[:n], K))[..., None]
            ent[:n].scatter_(2, at, e[:, None, None].expand_as(at))
            wts[:n].scatter_(2, at, ((nk - k[:n]).double() if count else TQ[:n] * a)[..., None])
            m[:n] += hit
            k[:n] = torch.where(hit, nk, k[:n])
            TQ[:n] = torch.where(hit, TQ[:n] * (1 - a), TQ[:n])
            T[:n] = torch.where(live, Tt, T[:n])
            done[:n] |= live & (Tt < tau[:n, :, K - 1])
        D = k.double() if count else 1 - TQ
        return self._kept(ent[..., :K], wts[..., :K], m, D)

    def _kept(self, ent, wts, m, D):
        has = torch.arange(ent.shape[-1], device="cuda") < m[..., None]
        w = torch.where(has, wts / torch.where(m > 0, D, torch.ones_like(D))[..., None],
                        torch.zeros_like(wts))
        return self.image(torch.where(has, ent, torch.full_like(ent, -1))), self.image(w)

    def topk(self, K):
        wts, at = self.new(K), self.new(K, fill=-1, dtype=torch.long)
        ent, i = self.new(K, fill=-1, dtype=torch.long), [0]

        def visit(e, w, T, live, n):
            low, j = wts[:n].min(-1, keepdim=True)
            put = live[..., None] & (w[..., None] > low)
            for x, v in ((wts, w[..., None]), (ent, e[:, None, None].expand_as(j)),
                         (at, torch.full_like(j, i[0]))):
                x[:n].scatter_(2, j, torch.where(put, v, x[:n].gather(2, j)))
            i[0] += 1
        self.dense(visit)
        order = torch.where(at < 0, torch.full_like(at, 1 << 40), at).argsort(-1)
        wts, ent = wts.gather(2, order), ent.gather(2, order)
        return self._kept(ent, wts, (ent >= 0).sum(-1), wts.sum(-1))

    def stratified(self, K):
        s1, s2, nb = self.new(), self.new(), self.new()

        def visit(e, w, T, live, n):
            x = torch.where(live, T[:n], torch.zeros_like(w))
            s1[:n] += x
            s2[:n] += x * x
            nb[:n] += live
        self.dense(visit)
        u = 1 - torch.arange(1, K + 1, dtype=torch.float64, device="cuda") / (K + 1)
        mu = s1 / nb
        sd = (s2 / nb - mu * mu).clamp(min=0).sqrt()
        lo, hi = torch.special.ndtr(-mu / sd), torch.special.ndtr((1 - mu) / sd)
        tau = mu[..., None] + sd[..., None] * torch.special.ndtri(
            lo[..., None] + (hi - lo)[..., None] * u)
        tau = torch.where((nb >= 2)[..., None], tau, u.expand_as(tau))
        ent, w = self.quantile(K, tau)
        return ent, w, self.image(tau)

    def pixel_terms(self, ent):
        """alpha exp(-q/2) parts of kept entries [P, K]: (G, alpha G, dx, dy)."""
        p = torch.arange(self.W * self.H, device="cuda")[:, None]
        e = ent.clamp(min=0)
        dx, dy = p % self.W + 0.5 - self.mean[e, 0], p // self.W + 0.5 - self.mean[e, 1]
        A = self.conic[e]
        G = torch.exp(-0.5 * (A[..., 0] * dx * dx + 2 * A[..., 1] * dx * dy + A[..., 2] * dy * dy))
        return G, self.alpha[e] * G, dx, dy


class _Rows:
    """The feature rows of a view's entries, decoded to float64."""

    def __init__(self, table, scale, gid):
        self.table, self.scale, self.gid = table.detach(), scale, gid

    def __call__(self, e):
        g = self.gid[e.clamp(min=0)]
        if self.scale is None:
            return self.table[g].double()
        return (self.table[g].view(torch.float8_e4m3fn).double() * self.scale[g][..., None].double())


def _blend(rows, ent, w):
    return sum(w[:, j, None] * rows(ent[:, j]) for j in range(ent.shape[1]))


def _gradients(v, rows, ent, g, n):
    """Gradients of the blend of the kept entries: features [n, C], opacity, conic."""
    K, C = ent.shape[1], g.shape[1]
    has = ent >= 0
    G, raw, dx, dy = v.pixel_terms(ent)
    a = torch.where(has, raw.clamp(max=ALPHA_MAX), torch.zeros_like(raw))
    s = torch.stack([(g * rows(ent[:, j])).sum(1) for j in range(K)], 1)
    P = torch.cat([torch.ones_like(a[:, :1]), (1 - a).cumprod(1)], 1)
    TQ, P = P[:, -1:], P[:, :-1]
    D = 1 - TQ
    ps = torch.where(has, a * P * s, torch.zeros_like(s))
    after = ps.flip(1).cumsum(1).flip(1) - ps
    gF = ps.sum(1, keepdim=True) / D
    da = (P * s - after / (1 - a)) / D - gF * TQ / ((1 - a) * D)
    da = torch.where(has & (raw < ALPHA_MAX), da, torch.zeros_like(da))
    gid = v.gid[ent.clamp(min=0)]
    gf = torch.zeros((n, C), dtype=torch.float64, device="cuda")
    ga = torch.zeros(n, dtype=torch.float64, device="cuda")
    gc = torch.zeros((n, 3), dtype=torch.float64, device="cuda")
    h = -0.5 * a * da
    for j in range(K):
        on = has[:, j]
        i = gid[on, j]
        # rows summed per Gaussian by a sparse product (few Gaussians, many pixels)
        who, back = torch.unique(i, return_inverse=True)
        pick = torch.sparse_coo_tensor(torch.stack([back, on.nonzero()[:, 0]]),
                                       (a * P / D)[on, j], (len(who), g.shape[0]))
        gf[who] += torch.sparse.mm(pick, g)
        ga.index_add_(0, i, (da * G)[on, j])
        gc.index_add_(0, i, torch.stack([h * dx * dx, 2 * h * dx * dy, h * dy * dy], 2)[on, j])
    return gf, ga, gc


def _cosine(F, t, on):
    nf, nt = F.norm(dim=1, keepdim=True).clamp(min=1e-8), t.norm(dim=1, keepdim=True).clamp(min=1e-8)
    cs, n = (F * t).sum(1, keepdim=True) / (nf * nt), on.sum().clamp(min=1)
    g = -(t / (nf * nt) - F * cs / (nf * nf)) / n
    return ((1 - cs[:, 0]) * on).sum() / n, g * on[:, None]


def _eq2(F, targets, mask):
    t = targets.double()
    t = t / t.norm(dim=1, keepdim=True).clamp(min=1e-8)
    raw = F.norm(dim=1, keepdim=True)
    nf = raw.clamp(min=1e-8)
    s = F @ t.T / nf
    on = mask >= 0
    n = on.sum().clamp(min=1)
    own = torch.nn.functional.one_hot(mask.clamp(min=0).long(), len(t)).bool()
    e = torch.where(own, torch.zeros_like(s), s.exp())
    Z = e.sum(1, keepdim=True)
    c = torch.where(own, -torch.ones_like(s), e / Z)
    g = (c @ t) / nf - torch.where(raw > 1e-8, (c * s).sum(1, keepdim=True) * F / (nf * nf),
                                   torch.zeros_like(F))
    terms = torch.where(on, Z[:, 0].log() - s.gather(1, mask.clamp(min=0).long()[:, None])[:, 0],
                        torch.zeros_like(Z[:, 0]))
    return terms.sum() / n, g * on[:, None] / n


def exact(case, seed):
    kind = case["kind"]
    if kind == "table":
        x = _features(case["n"], case["channels"], seed).double()
        return x if case["dtype"] == "bf16" else (None, x.abs().amax(1) / 448.0)
    if kind == "views":
        outs = []
        views = scenes.batched_views(case["seed_views"], case["views"], case["scenes"])
        qs = _features(case["queries"], case["channels"], seed + 3).to(torch.bfloat16).double()
        for i in range(case["scenes"]):
            n = case["n"] * (i + 1)
            g = _gaussians("room", n, seed + 10 * i)
            g = tuple(torch.from_numpy(np.ascontiguousarray(a, np.float32)).cuda()
                      for a in (g.mean, g.log_scale, g.quat, g.opacity))
            table, scale = _store(_features(n, case["channels"], seed + 10 * i + 1), case["dtype"])
            for si, cam in views:
                if si == i:
                    v = _Exact(g, cam)
                    ent, w = v.quantile(case["K"])
                    out = _blend(_Rows(table, scale, v.gid), ent, w)
                    outs.append((out.float(), w, out @ qs.T))
        # the maps of several views at full resolution: rounded once to 32 bits
        out, w, scores = (torch.cat(x) for x in zip(*outs))
        return {"out": out, "ids": None, "weights": w, "counts": None, "scores": scores}
    inp = _Inputs(case, seed)
    v = _Exact(inp.g, inp.cam)
    K = case.get("K", 8)
    if kind == "select":
        tau = None
        if case["rule"] == "topk":
            _, w = v.topk(K)
        elif case["rule"] == "stratified":
            _, w, tau = v.stratified(K)
        else:
            _, w = v.quantile(K, count=case["rule"] == "riemann")
        return {"ids": None, "weights": w, "counts": None, "tau": tau}
    rows = _Rows(inp.table, inp.scale, v.gid)
    if kind == "dense":
        out = v.new(case["channels"])
        ws, es = [], []

        def flush():
            if ws:
                n = max(len(e) for e in es)
                W = torch.stack([torch.nn.functional.pad(x, (0, 0, 0, n - len(x))) for x in ws], 2)
                E = torch.stack([torch.nn.functional.pad(x, (0, n - len(x))) for x in es], 1)
                out[:n] += W @ rows(E)
                ws.clear()
                es.clear()

        def visit(e, w, T, live, n):
            ws.append(w)
            es.append(e)
            if len(ws) == 32:
                flush()
        T = v.dense(visit)
        flush()
        return {"out": v.image(out), "T": v.image(T)}
    ent, w = v.quantile(K)
    out = _blend(rows, ent, w)
    if kind == "frame":
        return {"out": out, "ids": None, "weights": w, "counts": None}
    if kind == "relevance":
        return {"scores": out @ inp.queries.double().T}
    if kind == "backward":
        loss, g = _cosine(out, inp.target.double(), (ent >= 0).any(1))
        gf, ga, gc = _gradients(v, rows, ent, g, case["n"])
        return {"loss": loss, "grad_map": g, "grad_features": gf, "grad_opacity": ga,
                "grad_conic": gc}
    loss, g = _eq2(out, inp.targets, inp.mask)
    gf, ga, _ = _gradients(v, rows, ent, g, case["n"])
    return {"map": out.view(case["height"], case["width"], -1), "counts": None, "loss": loss,
            "grad_features": gf, "grad_opacity": ga}
