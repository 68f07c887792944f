"""The work that a program using this library has it do, as measurable cases.

Every case goes through the public entry points: `pipeline.Renderer` for whole
frames (project, intersect, sort, composite, adjoint) and the `psi` calls for
the query decode, the cross-attention, the label and geometry tables, the
storage conversion and the per-surfel training terms. Scenes are the plane-structured synthetic
scenes of `scenegen` (same planes, distributions and cameras), drawn on the
GPU so that a new input is made quickly.

Kinds of case:
  frame   one or more views of a map: project, intersect, sort, composite;
          optionally the query decode and the adjoint
  maps    depth and normal maps: the per-surfel geometry table, its dense
          composite, and both adjoints
  labels  the per-surfel instance-label table and its composite with the
          per-pixel argmax fused in
  attn    the frustum-constrained cross-attention and its adjoint
  terms   the per-surfel part of a training step: quaternion frames and their
          adjoint, the regularisers, and the storage form of the features
"""
from __future__ import annotations

import math

import numpy as np
import torch

from paper_2604_10982_gb300 import pipeline as pl, psi, scenegen as sg

DTYPES = {"f32": psi.F32, "bf16": psi.BF16, "fp8": psi.FP8_E4M3}
MODES = {"sphere": psi.SPHERE, "aabb": psi.AABB, "exact": psi.EXACT}
ESIZE = {"f32": 4, "bf16": 2, "fp8": 1}
# a case as `listed` and `draw` give it is completed from these
FRAME = dict(kind="frame", scene="street", n=200_000, views=1, width=1280, height=720, cam_y=2.0, D=64, feat="bf16",
             out="bf16", K=8, mode="exact", opacity_radius=True, lowpass=False, scale_median=0.05, queries=0,
             adjoint=False, graph=False)
# uneven resolutions of a multi-view batch, in shares of the case's largest one
VIEW_SHARES = (1 / 3, 1 / 2, 2 / 3, 5 / 6, 1)


def listed():
    f = lambda **kw: dict(FRAME, **kw)  # noqa: E731
    return [
        # a preview or a unit of an interactive tool: a small map, one small
        # view; launches and host work are what it costs
        f(name="tiny_box_fwd", scene="box", n=2000, width=128, height=128, D=16, feat="f32", out="f32"),
        # one view of a street map in plain FP32 with a large selection
        f(name="street_720p_fwd", n=200_000, D=64, feat="f32", out="f32", K=16, opacity_radius=False),
        # a training step on FP32 features: frame, upstream gradients, adjoint
        f(name="grad_540p_train", n=500_000, width=960, height=540, cam_y=5.0, D=128, feat="f32", out="f32", K=16,
          opacity_radius=False, adjoint=True),
        # many views of uneven resolution in one launch per stage, FP8 storage,
        # replayed as a CUDA graph
        f(name="batch16_fp8_fwd", n=1_000_000, views=16, width=1920, height=1080, D=128, feat="fp8", out="f32",
          graph=True),
        # full panoptic inference: composite and decode against 100 queries
        f(name="panoptic_1080p_infer", n=3_000_000, width=1920, height=1080, cam_y=5.0, D=128, queries=100),
        # the full training step on the same map
        f(name="panoptic_1080p_train", n=3_000_000, width=1920, height=1080, cam_y=20.0, D=128, queries=100,
          adjoint=True),
        # a ragged view of a dense indoor map with the low-pass filter, with
        # its adjoint (2DGS-compatible training)
        f(name="box_lowpass_train", scene="box", n=20_000, width=333, height=211, D=32, lowpass=True,
          scale_median=0.08, adjoint=True),
        # depth and normal supervision of a 700k-surfel map at an odd size
        dict(name="maps_ragged_train", kind="maps", scene="street", n=700_000, width=1237, height=701, cam_y=5.0,
             opacity_radius=True, scale_median=0.05),
        # the instance-label table of a map and one labelled view of it
        dict(name="labels_1M_540p", kind="labels", scene="street", n=1_000_000, width=960, height=540, cam_y=10.0,
             D=128, queries=100, K=8, scale_median=0.05),
        # queries attending to the surfels of a view, with the adjoint
        dict(name="attn_3M_train", kind="attn", scene="street", n=3_000_000, width=1920, height=1080, cam_y=5.0, D=128,
             d=128, queries=100),
        # the same for a small map and few queries
        dict(name="attn_40k_train", kind="attn", scene="street", n=40_001, width=960, height=540, cam_y=5.0, D=64, d=64,
             queries=20),
        # the per-surfel terms of a training step over a whole map
        dict(name="terms_1M", kind="terms", scene="street", n=1_000_003, D=128, feat="fp8"),
    ]


def _log(rng, lo, hi):
    return math.exp(rng.uniform(math.log(lo), math.log(hi)))


def _map_size(rng, pixels, most):
    """Surfels of a map seen by a view of so many pixels: at most two per pixel
    (a far denser map is thinned out before it is shown that small)."""
    return int(_log(rng, 1_000, max(1_500, min(most, 2 * pixels))))


def draw(rng):
    """One more case of the same ranges."""
    kind = rng.choices(["frame", "maps", "labels", "attn", "terms"], [10, 1, 1, 2, 1])[0]
    w = max(33, int(_log(rng, 64, 1921)))
    h = max(17, min(1080, int(w * rng.uniform(0.4, 1.0))))
    if kind == "attn":
        return dict(kind=kind, scene="street", n=int(_log(rng, 1_000, 3_000_000)), width=w, height=h,
                    cam_y=rng.uniform(2, 40), D=rng.choice([64, 128]), d=rng.choice([32, 64, 128, 256]),
                    queries=rng.randint(1, 128))
    if kind == "terms":
        return dict(kind=kind, scene="street", n=int(_log(rng, 1_000, 1_000_000)), D=rng.choice([16, 48, 64, 128]),
                    feat=rng.choice(["bf16", "fp8"]))
    if kind == "maps":
        w, h = min(w, 1237), min(h, 701)
        return dict(kind=kind, scene="street", n=_map_size(rng, w * h, 700_000), width=w, height=h,
                    cam_y=rng.uniform(2, 40), opacity_radius=True, scale_median=0.05)
    if kind == "labels":
        return dict(kind=kind, scene="street", n=_map_size(rng, w * h, 1_000_000), width=w, height=h,
                    cam_y=rng.uniform(2, 40), D=rng.choice([64, 128]), queries=rng.randint(1, 128),
                    K=rng.choice([1, 4, 8]), scale_median=0.05)
    scene = rng.choices(["street", "box"], [4, 1])[0]
    feat = rng.choice(["f32", "bf16", "bf16", "fp8"])
    K = rng.choices([8, 16, 0, rng.randint(1, 32)], [6, 2, 1, 2])[0]
    D = rng.choice([16, 32, 48, 64, 128, 128, 256])
    views = rng.choice([1, 1, 1, 1, 2, 3, 5])
    adjoint = rng.random() < 0.5
    if K == 0:
        D, w, h = rng.choice([16, 32]), min(w, 320 if adjoint else 640), min(h, 180 if adjoint else 360)
    if K > 8 or D > 128 or views > 1:
        w, h = min(w, 960), min(h, 540)
    mode = rng.choices(["exact", "aabb", "sphere"], [6, 1, 1])[0]
    n = _map_size(rng, w * h if mode == "exact" else w * h // 4, 20_000 if scene == "box" else 3_000_000)
    lowpass = rng.random() < 0.2
    out = "bf16" if rng.random() < 0.5 else "f32"
    queries = rng.randint(1, 128) if (D in (64, 128) and out == "bf16") else 0
    return dict(FRAME, scene=scene, n=n, views=views, width=w, height=h,
                cam_y=rng.uniform(2, 40) if scene == "street" else 0.0, D=D, feat=feat, out=out, K=K,
                mode=mode, opacity_radius=rng.random() < 0.7,
                lowpass=lowpass, scale_median=0.05 if scene == "street" else rng.uniform(0.05, 0.12), queries=queries,
                adjoint=adjoint, graph=rng.random() < 0.2 and not adjoint)


# ------------------------------------------------------------------ inputs
def _cameras(case):
    w, h, views = case["width"], case["height"], case.get("views", 1)
    if case["scene"] == "box":
        return [sg.look_camera((0.5 * math.sin(v), -6.0, 1.5), 0.1 * v, w, h, 0.86 * w) for v in range(views)]
    if views == 1:
        return [sg.look_camera((0.0, case["cam_y"], 1.5), 0.0, w, h, w / 2.0)]
    cams = []
    for v in range(views):
        s = VIEW_SHARES[v % len(VIEW_SHARES)]
        vw, vh = max(16, round(w * s)), max(16, round(h * s))
        yaw = (0.0 if v % 2 == 0 else math.pi) + 0.17 * math.sin(2.3 * v)
        cams.append(sg.look_camera((0.0, 60.0 * v / (views - 1), 1.5), yaw, vw, vh, vw / 2.0))
    return cams


def _surfels(case, g):
    """The scene generator's plane-structured surfels, drawn on the GPU."""
    n = case["n"]
    planes = sg.box_planes() if case["scene"] == "box" else sg.street_planes()
    dev = "cuda"
    U = lambda *s: torch.rand(*s, generator=g, device=dev, dtype=torch.float64)  # noqa: E731
    N = lambda *s: torch.randn(*s, generator=g, device=dev, dtype=torch.float64)  # noqa: E731
    area = torch.tensor([p.area for p in planes], dtype=torch.float64, device=dev)
    pick = torch.searchsorted(torch.cumsum(area, 0) / area.sum(), U(n), right=True).clamp(max=len(planes) - 1)
    col = lambda a: torch.tensor([getattr(p, a) for p in planes], dtype=torch.float64, device=dev)[pick]  # noqa: E731
    e1, e2 = col("e1"), col("e2")
    nrm = torch.linalg.cross(e1, e2)
    mu = (col("origin") + (U(n) * col("l1"))[:, None] * e1 + (U(n) * col("l2"))[:, None] * e2 +
          (0.02 * N(n))[:, None] * nrm)
    phi = 2.0 * math.pi * U(n)
    axis = torch.cos(phi)[:, None] * e1 + torch.sin(phi)[:, None] * e2
    th = math.radians(5.0) * N(n)
    n2 = nrm * torch.cos(th)[:, None] + torch.linalg.cross(axis, nrm) * torch.sin(th)[:, None]
    b2 = torch.linalg.cross(n2, axis)
    rot = 2.0 * math.pi * U(n)
    tu = torch.cos(rot)[:, None] * axis + torch.sin(rot)[:, None] * b2
    tv = torch.linalg.cross(n2, tu)
    scale = torch.exp(math.log(case.get("scale_median", 0.05)) + 0.5 * N(n, 2))
    return [t.float().contiguous() for t in (mu, tu, tv, scale, torch.sigmoid(N(n)), U(n, 3))]


def _normal(g, *shape):
    return torch.randn(*shape, generator=g, device="cuda")


def _draw(case, seed):
    """Every random input of the case, from the seed alone."""
    g = torch.Generator(device="cuda")
    g.manual_seed(seed * 7919 + 17)
    x = {"surfels": _surfels(case, g)}
    n, D, kind = case["n"], case.get("D", 0), case["kind"]
    if kind == "frame":
        P = sum(c.width * c.height for c in _cameras(case))
        x["feat"] = _normal(g, n, D)
        x["queries"] = (_normal(g, max(case["queries"], 1), D) / math.sqrt(D)).to(torch.bfloat16)
        if case["adjoint"]:
            x["gC"], x["gF"], x["gT"] = _normal(g, 3, P), _normal(g, P, D), _normal(g, P)
    elif kind == "maps":
        P = case["width"] * case["height"]
        x["gC"], x["gF"], x["gT"] = _normal(g, 3, P), _normal(g, P, 16), _normal(g, P)
        x["gF"][:, 4:] = 0.0  # the table's padding columns carry no loss
    elif kind == "labels":
        q = case["queries"]
        x["feat"] = _normal(g, n, D)
        x["queries"] = (_normal(g, q, D) / math.sqrt(D)).to(torch.bfloat16)
        r = torch.rand(q, 3, generator=g, device="cuda")
        x["q_mu"] = r * torch.tensor([16.0, 60.0, 12.0], device="cuda") - torch.tensor([8.0, 0.0, 0.0], device="cuda")
        a = _normal(g, q, 3).double()  # a random orthonormal frame per query
        b = torch.linalg.cross(a, _normal(g, q, 3).double())
        a = torch.stack([v / v.norm(dim=1, keepdim=True) for v in (a, b, torch.linalg.cross(a, b))], 2)
        s = 0.5 + 2.5 * torch.rand(q, 3, generator=g, device="cuda").double()
        x["q_cov"] = (a @ torch.diag_embed(s * s) @ a.transpose(1, 2)).float().contiguous()
    elif kind == "attn":
        q, d = case["queries"], case["d"]
        x["feat"] = _normal(g, n, D)
        x["Q"] = _normal(g, q, D)
        x["W"] = [_normal(g, D, d) / math.sqrt(D) for _ in range(3)]
        x["gO"] = _normal(g, q, d)
    else:  # terms
        x["feat"] = _normal(g, n, D)
        x["quat"] = _normal(g, n, 4)
        x["gtu"], x["gtv"] = _normal(g, n, 3), _normal(g, n, 3)
        nodes = 64
        x["node_of"] = torch.randint(-1, nodes, (n,), generator=g, device="cuda", dtype=torch.int32)
        x["node_mu"] = _normal(g, nodes, 3) * 5.0
        nn = _normal(g, nodes, 3)
        x["node_n"] = (nn / nn.norm(dim=1, keepdim=True)).contiguous()
    return x


def _scene(x, q=None, qscale=None, dtype=psi.F32):
    s = pl.DeviceScene(sg.Surfels(*(t.cpu().numpy() for t in x["surfels"])))
    if q is not None:
        s.q, s.qscale, s.feat_dtype, s.D = q, qscale, dtype, int(q.shape[1])
    return s


def _grads(n, D):
    z = lambda *s: torch.zeros(*s, device="cuda")  # noqa: E731
    d = dict(mu=z(n, 3), tu=z(n, 3), tv=z(n, 3), scale=z(n, 2), opacity=z(n), rgb=z(n, 3), feat=z(n, D) if D else None)
    return d, psi.PsiGrads(*(psi._ptr(d[k]) for k in ("mu", "tu", "tv", "scale", "opacity", "rgb", "feat")))


def prepare(case, seed):
    x = _draw(case, seed)
    ctx = psi.Context(0)
    st = dict(case=case, ctx=ctx, x=x)
    kind, n, D = case["kind"], case["n"], case.get("D", 0)
    if kind == "frame":
        dt = DTYPES[case["feat"]]
        q, qs = pl.quantize_features(x.pop("feat"), dt, ctx)
        st["scene"] = sc = _scene(x, q, qs, dt)
        opts = psi.default_opts(mode=MODES[case["mode"]], top_k=case["K"], opacity_radius=int(case["opacity_radius"]),
                                lowpass=int(case["lowpass"]))
        st["r"] = r = pl.make_renderer(ctx, sc, _cameras(case), opts, D=D, F_dtype=DTYPES[case["out"]])
        if case["queries"]:
            st["ids"] = torch.empty(r.n_pix, dtype=torch.int32, device="cuda")
        if case["adjoint"]:
            st["grads"], st["gs"] = _grads(n, D)
        if case["graph"]:
            _forward(st)
            torch.cuda.synchronize()
            st["graph"] = torch.cuda.CUDAGraph()
            with torch.cuda.graph(st["graph"], capture_error_mode="relaxed"):
                _forward(st)
    elif kind == "maps":
        st["scene"] = sc = _scene(x)
        opts = psi.default_opts(top_k=0, opacity_radius=int(case["opacity_radius"]))
        st["cam"] = _cameras(case)[0]
        st["r"] = pl.make_renderer(ctx, sc, [st["cam"]], opts, D=16)
        st["grads"], st["gs"] = _grads(n, 16)
    elif kind == "labels":
        q, qs = pl.quantize_features(x.pop("feat"), psi.BF16, ctx)
        st["scene"] = sc = _scene(x, q, qs, psi.BF16)
        opts = psi.default_opts(top_k=case["K"], opacity_radius=1)
        st["r"] = pl.make_renderer(ctx, sc, _cameras(case), opts, D=0)
    elif kind == "attn":
        q, _ = pl.quantize_features(x.pop("feat"), psi.BF16, ctx)
        st["scene"] = _scene(x, q, None, psi.BF16)
        st["cam"] = psi.cameras(_cameras(case))[0]
        st["grads"], st["gs"] = _grads(n, D)
        e = lambda *s: torch.empty(*s, device="cuda")  # noqa: E731
        nq, d = case["queries"], case["d"]
        st["out"] = dict(O=e(nq, d), gQ=e(nq, D), gWQ=e(D, d), gWK=e(D, d), gWV=e(D, d))
        st["ws"] = torch.empty(psi.attention_workspace_size(n, D, d, nq), dtype=torch.uint8, device="cuda")
    else:
        st["scene"] = _scene(x)
        st["grads"], st["gs"] = _grads(n, 0)
        st["gq"] = torch.zeros(n, 4, device="cuda")
        st["losses"] = torch.empty(2, dtype=torch.float64, device="cuda")
    return st


# ------------------------------------------------------------------ one pass
def _forward(st):
    r, case = st["r"], st["case"]
    r.frame(st["scene"])
    if case["queries"]:
        psi.psi_decode_queries(st["ctx"], r.F, r.n_pix, case["D"], st["x"]["queries"], case["queries"], r.T, st["ids"])


def run(st):
    case, ctx, x, sc = st["case"], st["ctx"], st["x"], st["scene"]
    kind = case["kind"]
    if kind == "frame":
        r = st["r"]
        if case["graph"]:
            st["graph"].replay()
        else:
            _forward(st)
        out = dict(rgb=r.rgb, T=r.T, F=r.F, n_last=r.n_last, topk_ids=r.topk_ids, topk_w=r.topk_w)
        if case["queries"]:
            out["ids"] = st["ids"]
        if case["adjoint"]:
            psi.psi_grads_zero(ctx, st["gs"], case["n"], case["D"])
            out["grads"] = r.backward(sc, x["gC"], x["gF"], x["gT"], grads=st["grads"])
        return out
    if kind == "maps":
        r = st["r"]
        ts = pl.label_scene(sc, pl.surfel_geometry(ctx, sc, st["cam"]))
        r.frame(ts)
        psi.psi_grads_zero(ctx, st["gs"], case["n"], 16)
        gr = r.backward(ts, x["gC"], x["gF"], x["gT"], grads=st["grads"])
        psi.psi_surfel_geometry_bwd(ctx, sc.surfels_struct(), psi.cameras([st["cam"]]), gr["feat"], 16, st["gs"])
        return dict(rgb=r.rgb, T=r.T, F=r.F, grads=gr)
    if kind == "labels":
        r = st["r"]
        table = pl.surfel_labels(ctx, sc, x["queries"], x["q_mu"], x["q_cov"])
        ls = pl.label_scene(sc, table)
        r.project(ls)
        r.intersect()
        r.sort()
        r.render(ls, want_F=False, argmax=True)
        return dict(table=table, ids=r.argmax, rgb=r.rgb, T=r.T)
    if kind == "attn":
        o, nq, d = st["out"], case["queries"], case["d"]
        s, f = sc.surfels_struct(), sc.features_struct()
        psi.psi_grads_zero(ctx, st["gs"], case["n"], case["D"])
        psi.psi_frustum_attention(ctx, s, f, st["cam"], 0.2, x["Q"], nq, *x["W"], d, o["O"], st["ws"])
        psi.psi_frustum_attention_bwd(ctx, s, f, x["Q"], nq, *x["W"], d, x["gO"], o["gQ"], o["gWQ"], o["gWK"], o["gWV"],
                                      st["gs"], st["ws"])
        return dict(o, g_feat=st["grads"]["feat"], g_mu=st["grads"]["mu"])
    n = case["n"]
    gr = st["grads"]
    psi.psi_grads_zero(ctx, st["gs"], n, 0)
    psi.psi_quat_frames(ctx, x["quat"], n, sc.tu, sc.tv)
    s = sc.surfels_struct()
    psi.psi_surfel_regularisers(ctx, s, x["node_of"], x["node_mu"], x["node_n"], 64, 0.5, 0.1, 0.01, st["losses"],
                                st["gs"])
    st["gq"].zero_()
    psi.psi_quat_frames_bwd(ctx, x["quat"], n, x["gtu"], x["gtv"], st["gq"])
    q, qs = pl.quantize_features(x["feat"], DTYPES[case["feat"]], ctx)
    return dict(tu=sc.tu, tv=sc.tv, losses=st["losses"], g_mu=gr["mu"], g_tu=gr["tu"], g_tv=gr["tv"],
                g_scale=gr["scale"], gq=st["gq"], q=q.view(torch.uint8), qscale=qs)


def work(case):
    """Bytes and operations of one pass: inputs read once, outputs written
    once; of the feature rows, those that a pixel can select; of the
    operations, the contractions with the features."""
    n, D, kind = case["n"], case.get("D", 0), case["kind"]
    if kind == "attn":
        nq = case["queries"]
        return {"bytes": n * (2 * D + 20) * 2 + n * (D + 3) * 4, "flops": 14.0 * nq * n * D}
    if kind == "terms":
        return {"bytes": n * (44 + 4 + 44 + 16 + 24 + 24 + 16) + n * D * (4 + ESIZE[case["feat"]]), "flops": 200.0 * n}
    P = sum(c.width * c.height for c in _cameras(case))
    if kind == "labels":
        q = case["queries"]
        ld = (q + 15) // 16 * 16
        return {"bytes": n * (60 + 2 * D + 2 * ld) + min(n, P * case["K"]) * 2 * ld + P * (16 + 4 + 4),
                "flops": 2.0 * n * q * D + 2.0 * P * case["K"] * ld}
    if kind == "maps":
        D, K, es, eo, adj, q = 16, 0, 4, 4, True, 0
    else:
        K, es, eo, adj, q = case["K"], ESIZE[case["feat"]], ESIZE[case["out"]], case["adjoint"], case["queries"]
    rows = min(n, P * K) if K else n
    b = n * 60 + rows * D * es + P * (20 + 8 * K) + P * D * eo + (P * 4 if q else 0)
    f = 2.0 * P * (K or 16) * D + 2.0 * P * q * D
    if adj:
        b += P * 16 + P * D * 4 + n * (15 + D) * 4
        f += 4.0 * P * (K or 16) * D
    return {"bytes": b, "flops": f}


# ------------------------------------------------------------------ 64 bits
def _stored(f, feat):
    """The stored feature values in 64 bits."""
    if feat == "f32":
        return f.double()
    if feat == "bf16":
        return f.to(torch.bfloat16).double()
    s = f.abs().amax(0).clamp(min=1e-30) / 448.0
    return (f / s).clamp(-448, 448).to(torch.float8_e4m3fn).double() * s.double()


def _composite(case, x, opts, table, gC=None, gF=None, gT=None, D=0, K=0):
    """Brute force over every surfel at every pixel, by automatic
    differentiation: (rgb, F, T) of each view and the gradients."""
    leaves = [t.double().requires_grad_(gC is not None) for t in x["surfels"]]
    mu, tu, tv, sc, op, col = leaves
    P_tot = sum(c.width * c.height for c in _cameras(case))
    f64 = dict(dtype=torch.float64, device="cuda")
    C, F, T = torch.zeros(3, P_tot, **f64), torch.zeros(P_tot, D, **f64), torch.zeros(P_tot, **f64)
    feat = table.detach().requires_grad_(gC is not None) if table is not None else None
    base = 0
    for cam in _cameras(case):
        R = torch.tensor(np.asarray(cam.R, np.float32), device="cuda").double()
        t = torch.tensor(np.asarray(cam.t, np.float32), device="cuda").double()
        f_, cx, cy = float(np.float32(cam.fx)), float(np.float32(cam.cx)), float(np.float32(cam.cy))
        r2 = torch.full_like(op, 9.0)
        if opts["opacity_radius"]:
            r2 = torch.minimum(r2, 2.0 * torch.log(255.0 * op.detach().clamp(min=1e-9)) + 1e-3)
        with torch.no_grad():
            z = mu @ R[2] + t[2]
            nab = torch.sqrt((sc[:, 0] * (tu @ R[2])) ** 2 + (sc[:, 1] * (tv @ R[2])) ** 2)
            keep = (op >= 1.0 / 255.0) & (z - torch.sqrt(r2.clamp(min=0) * (1 + 2.0 ** -10)) * nab > float(np.float32(0.2)))
            idx = torch.nonzero(keep)[:, 0]
            idx = idx[torch.sort(z[idx].float(), stable=True)[1]]
        P = cam.width * cam.height
        step = max(64, 4_000_000 // max(int(idx.numel()), 1))
        for p0 in range(0, P, step):
            p = torch.arange(p0, min(p0 + step, P), device="cuda")
            px, py = (p % cam.width).double() + 0.5, (p // cam.width).double() + 0.5
            proj = lambda v: torch.stack([f_ * v[:, 0] + cx * v[:, 2], f_ * v[:, 1] + cy * v[:, 2], v[:, 2]], 1)  # noqa: E731
            m0 = proj((sc[idx, :1] * tu[idx]) @ R.T)
            m1 = proj((sc[idx, 1:] * tv[idx]) @ R.T)
            m2 = proj(mu[idx] @ R.T + t)
            rows = [torch.linalg.cross(m1, m2), torch.linalg.cross(m2, m0), torch.linalg.cross(m0, m1)]
            q = [r[:, 0] * px[:, None] + r[:, 1] * py[:, None] + r[:, 2] for r in rows]
            d2 = (q[0] ** 2 + q[1] ** 2) / (q[2] ** 2).clamp(min=1e-300)
            rr = r2[idx]
            if opts["lowpass"]:
                ell = (d2 <= rr) & (q[2] ** 2 > 0)
                rho = 2.0 * ((px[:, None] - m2[:, 0] / m2[:, 2]) ** 2 + (py[:, None] - m2[:, 1] / m2[:, 2]) ** 2)
                filt = (rho < d2) | ~ell
                d2 = torch.where(filt, rho, d2)
            a = torch.clamp(op[idx] * torch.exp(-0.5 * d2.clamp(max=100.0)), max=0.99)
            hit = (d2 <= rr) & (a >= 1.0 / 255.0)
            a = torch.where(hit, a, torch.zeros_like(a))
            lg = torch.log1p(-a)
            Tb = torch.exp(torch.cumsum(lg, 1) - lg)
            live = hit & (Tb.detach() >= float(np.float32(1e-4)))
            w = torch.where(live, a * Tb, torch.zeros_like(a))
            Tf = torch.exp(torch.where(live, lg, torch.zeros_like(lg)).sum(1))
            c = w @ col[idx]
            sl = slice(base + p0, base + p0 + p.numel())
            loss = 0.0
            if D:
                if K:
                    wk, ik = torch.topk(w, min(K, w.shape[1]), dim=1)
                    Fp = torch.einsum("pk,pkd->pd", wk, feat[idx[ik]])
                else:
                    Fp = w @ feat[idx]
                F[sl] = Fp.detach()
                if gC is not None:
                    loss = (gF[sl].double() * Fp).sum()
            C[:, sl], T[sl] = c.detach().T, Tf.detach()
            if gC is not None:
                loss = loss + (gC[:, sl].double().T * c).sum() + (gT[sl].double() * Tf).sum()
                loss.backward()
        base += P
    return C, F, T, leaves, feat


def exact(case, seed):
    kind, n = case["kind"], case["n"]
    if kind in ("frame", "maps", "labels"):
        P = sum(c.width * c.height for c in _cameras(case))
        if n * P > 3_000_000_000 and kind != "labels":
            return None
    x = _draw(case, seed)
    mu, tu, tv, sc, op, col = (t.double() for t in x["surfels"])
    if kind == "frame":
        adj = case["adjoint"]
        C, F, T, lv, feat = _composite(case, x, case, _stored(x["feat"], case["feat"]), *([x["gC"], x["gF"], x["gT"]] if adj else [None] * 3),
                                       D=case["D"], K=case["K"])
        out = dict(rgb=C, T=T, F=F, n_last=None, topk_ids=None, topk_w=None, ids=None)
        if adj:
            out["grads"] = dict(zip(("mu", "tu", "tv", "scale", "opacity", "rgb"), (v.grad for v in lv)), feat=feat.grad)
        return out
    if kind == "maps":
        cam = _cameras(case)[0]
        R = torch.tensor(np.asarray(cam.R, np.float32), device="cuda").double()
        t = torch.tensor(np.asarray(cam.t, np.float32), device="cuda").double()

        def table(m, u, v):
            xc = m @ R.T + t
            nc = torch.linalg.cross(u, v)
            nc = (nc / nc.norm(dim=1, keepdim=True)) @ R.T
            nc = torch.where(((nc * xc).sum(1) > 0)[:, None], -nc, nc)
            return torch.cat([xc[:, 2:], nc, torch.zeros(n, 12, dtype=torch.float64, device="cuda")], 1)

        C, F, T, lv, tb = _composite(case, x, dict(opacity_radius=case["opacity_radius"], lowpass=False),
                                     table(mu, tu, tv).float().double(), x["gC"], x["gF"], x["gT"], D=16, K=0)
        grads = dict(zip(("mu", "tu", "tv", "scale", "opacity", "rgb"), (v.grad.clone() for v in lv)), feat=tb.grad)
        for v in lv:
            v.grad = None
        table(*lv[:3]).backward(tb.grad)
        for k, v in zip(("mu", "tu", "tv"), lv):
            grads[k] += v.grad
        return dict(rgb=C, T=T, F=F, grads=grads)
    if kind == "labels":
        f = x["feat"].to(torch.bfloat16).double()
        s = torch.sigmoid(f @ x["queries"].double().T)
        prec = torch.from_numpy(np.linalg.inv(x["q_cov"].double().cpu().numpy())).cuda()
        for q in range(case["queries"]):
            d = mu - x["q_mu"][q].double()
            s[:, q] *= torch.exp(-0.5 * ((d @ prec[q]) * d).sum(1))
        tab = torch.softmax(s, 1)
        ld = (case["queries"] + 15) // 16 * 16
        return dict(table=torch.nn.functional.pad(tab, (0, ld - case["queries"])), ids=None, rgb=None, T=None)
    if kind == "attn":
        C, d = case["D"], case["d"]
        f = x["feat"].to(torch.bfloat16).double().requires_grad_(True)
        m = mu.clone().requires_grad_(True)
        Q = x["Q"].double().requires_grad_(True)
        WQ, WK, WV = (w.double().requires_grad_(True) for w in x["W"])
        c = torch.arange(C, device="cuda")
        tt = c // 3
        arg = m[:, c % 3] * (10000.0 ** (-6.0 * (tt // 2).double() / C))
        Kf = f + torch.where(tt % 2 == 0, torch.sin(arg), torch.cos(arg))
        with torch.no_grad():
            cam = _cameras(case)[0]
            R = torch.tensor(np.asarray(cam.R, np.float32), device="cuda").double()
            t = torch.tensor(np.asarray(cam.t, np.float32), device="cuda").double()
            xc = mu @ R.T + t
            fx, cx, cy, W, H = cam.fx, cam.cx, cam.cy, cam.width, cam.height
            z = xc[:, 2]
            dist = torch.stack([z - float(np.float32(0.2)), (fx * xc[:, 0] + cx * z) / math.hypot(fx, cx),
                                (-fx * xc[:, 0] + (W - cx) * z) / math.hypot(fx, W - cx),
                                (fx * xc[:, 1] + cy * z) / math.hypot(fx, cy),
                                (-fx * xc[:, 1] + (H - cy) * z) / math.hypot(fx, H - cy)]).amin(0)
            act = dist + math.sqrt(-2.0 * math.log(0.01)) * sc.amax(1) >= 0
        if not bool(act.any()):
            return None
        e = ((Q @ WQ) @ WK.T / math.sqrt(d)) @ Kf.T
        p = torch.softmax(e.masked_fill(~act, -math.inf), 1)
        O = (p @ f) @ WV
        (O * x["gO"].double()).sum().backward()
        return dict(O=O.detach(), gQ=Q.grad, gWQ=WQ.grad, gWK=WK.grad, gWV=WV.grad, g_feat=f.grad, g_mu=m.grad)
    q = x["quat"].double().requires_grad_(True)
    u = q / q.norm(dim=1, keepdim=True)
    w_, x_, y_, z_ = u.unbind(1)
    a = torch.stack([1 - 2 * (y_ * y_ + z_ * z_), 2 * (x_ * y_ + w_ * z_), 2 * (x_ * z_ - w_ * y_)], 1)
    b = torch.stack([2 * (x_ * y_ - w_ * z_), 1 - 2 * (x_ * x_ + z_ * z_), 2 * (y_ * z_ + w_ * x_)], 1)
    ((a * x["gtu"].double()).sum() + (b * x["gtv"].double()).sum()).backward()
    m, u_, v_, s_ = (t.detach().clone().requires_grad_(True) for t in (mu, a, b, sc))
    k = x["node_of"].long()
    on = k >= 0
    nh, nm = x["node_n"].double()[k[on]], x["node_mu"].double()[k[on]]
    c = torch.linalg.cross(u_, v_)[on]
    c = c / c.norm(dim=1, keepdim=True)
    geo = (((m[on] - nm) * nh).sum(1).abs() + 0.5 * (1 - (c * nh).sum(1).abs())).sum()
    iso = ((s_[:, 0] - s_[:, 1]) ** 2).sum()
    w_geo, w_iso = float(np.float32(0.1)), float(np.float32(0.01))
    (w_geo * geo + w_iso * iso).backward()
    return dict(tu=a.detach(), tv=b.detach(), losses=torch.stack([geo, iso]).detach(), g_mu=m.grad, g_tu=u_.grad,
                g_tv=v_.grad, g_scale=s_.grad, gq=q.grad, q=None, qscale=None)
