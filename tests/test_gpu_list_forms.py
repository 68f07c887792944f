"""Forms of the list walks that change with the tile shape, the launch shape
and the features, at the list lengths where the staging changes over (needs a
GPU). Bars: those of the parity suites -- forward values as check_values, or
bit for bit between launch shapes; gradients 1e-5 relative L2 between two
forms (only the order of float32 additions differs)."""
import numpy as np
import pytest

torch = pytest.importorskip("torch")

from oracle import oracle as orc
from paper_2604_10982_gb300 import scenegen as sg

from .gpu_common import check_values, opts_of
from .test_gpu_list_edges import _stack

pytestmark = pytest.mark.gpu

GRADS = ("mu", "tu", "tv", "scale", "opacity", "rgb", "feat")


@pytest.fixture(scope="module")
def ctx():
    if not torch.cuda.is_available():
        pytest.skip("no CUDA device")
    from paper_2604_10982_gb300 import psi
    return psi.Context(0)


def _upstream(P, D):
    g = torch.Generator(device="cpu").manual_seed(11)
    return [torch.randn(*s, generator=g).cuda() for s in ((3, P), (P, D), (P,))]


def _close(a, b, what):
    for k in GRADS:
        x, y = a[k].double(), b[k].double()
        assert torch.linalg.norm(x - y).item() <= 1e-5 * torch.linalg.norm(y).item(), (what, k)


@pytest.mark.parametrize("K,lowpass", [(8, False), (16, False), (8, True)])
def test_warps_leave_the_walk_at_different_batches(ctx, K, lowpass):
    """Lists of up to 900 records, half of them opaque and a few pixels wide,
    half faint and wide: some warps are saturated early, some late, some never,
    so the producer is stopped or waited for at any batch.
    Launched over and over, one tile per CTA and persistent."""
    from paper_2604_10982_gb300 import pipeline as pl, psi
    w = _stack(900, 16)
    w.surfels.opacity[:] = np.where(np.arange(900) % 2 == 0, 0.006, 0.9).astype(np.float32)
    cam = w.cameras[0]
    o = orc.Opts(mode=orc.EXACT, top_k=K, opacity_radius=True, lowpass=lowpass)
    scene = pl.DeviceScene(w.surfels, w.features)
    r = pl.make_renderer(ctx, scene, [cam], opts_of(o), D=16)
    r.frame(scene)
    up = _upstream(r.n_pix, 16)
    ref = orc.render(w.surfels, cam, o, feat=w.features.astype(np.float64))
    assert (ref["T"] < 1e-4).any() and (ref["T"] > 0.5).any()
    check_values(r.rgb.cpu().numpy().astype(np.float64).T, r.T.cpu().numpy().astype(np.float64),
                 r.F.cpu().numpy().astype(np.float64), ref, cam, fmax=np.abs(w.features).max())
    first = [t.clone() for t in (r.rgb, r.T, r.n_last, r.F, r.topk_ids, r.topk_w)]
    g0 = r.backward(scene, *up)
    try:
        for shape in (0, 4):
            for which, saved in ((0, 0), (1, 1), (1, 0)):
                psi.psi_ctx_set_render_shape(ctx, which, r.opts, psi.F32, saved, shape)
            for _ in range(100):
                r.render(scene)
                for a, b in zip(first, (r.rgb, r.T, r.n_last, r.F, r.topk_ids, r.topk_w)):
                    assert torch.equal(a, b), shape
            for _ in range(20):
                _close(r.backward(scene, *up), g0, shape)
                _close(r.backward(scene, *up, recompute=True), g0, shape)
    finally:
        for which, saved in ((0, 0), (1, 1), (1, 0)):
            psi.psi_ctx_set_render_shape(ctx, which, r.opts, psi.F32, saved, 0)
    assert ctx.status_fetch() == (0, 0)


FORMS = {  # options, feature dim, forward shape, adjoint shapes from saved state, recomputing
    "tile8": (dict(top_k=8, tile_h=8), 32, 0, (0, 4), (0, 4)),
    "tile8_k3": (dict(top_k=3, tile_h=8), 32, 4, (0,), (0,)),
    "tile8_pair": (dict(top_k=8, tile_h=8), 32, 0, (8, 12), (0,)),
    "alternative": (dict(top_k=8), 32, 1, (1,), (1,)),
    "alternative_persistent": (dict(top_k=8), 32, 5, (5, 13), (5,)),
    "lowpass": (dict(top_k=8, lowpass=True), 32, 1, (0, 1, 8), (0,)),
    "dense32": (dict(top_k=0), 32, 0, (0, 1), (0,)),
}


@pytest.mark.parametrize("n", [127, 129, 257, 513, 900])
@pytest.mark.parametrize("form", list(FORMS))
def test_forms_at_list_lengths(ctx, form, n):
    """Forward against the oracle (this input excuses no pixel), bit for bit
    against the default shape; every adjoint form against the default one."""
    from paper_2604_10982_gb300 import pipeline as pl, psi
    kw, D, fwd, saved_shapes, re_shapes = FORMS[form]
    w = _stack(n, D)
    cam = w.cameras[0]
    o = orc.Opts(mode=orc.EXACT, opacity_radius=True, **kw)
    scene = pl.DeviceScene(w.surfels, w.features)
    base = pl.make_renderer(ctx, scene, [cam], opts_of(orc.Opts(mode=orc.EXACT, opacity_radius=True,
                                                                **{k: v for k, v in kw.items() if k != "tile_h"})), D=D)
    base.frame(scene)
    up = _upstream(base.n_pix, D)
    g0 = base.backward(scene, *up)
    r = pl.make_renderer(ctx, scene, [cam], opts_of(o), D=D)
    try:
        psi.psi_ctx_set_render_shape(ctx, 0, r.opts, psi.F32, 0, fwd)
        r.frame(scene)
        ref = orc.render(w.surfels, cam, o, feat=w.features.astype(np.float64))
        check_values(r.rgb.cpu().numpy().astype(np.float64).T, r.T.cpu().numpy().astype(np.float64),
                     r.F.cpu().numpy().astype(np.float64), ref, cam, max_excused=0, fmax=np.abs(w.features).max())
        for name in ("rgb", "T", "F") + (("topk_ids", "topk_w") if kw["top_k"] else ()):
            assert torch.equal(getattr(r, name), getattr(base, name)), name
        for saved, shapes in ((1, saved_shapes), (0, re_shapes)):
            for shape in shapes:
                psi.psi_ctx_set_render_shape(ctx, 1, r.opts, psi.F32, saved, shape)
                _close(r.backward(scene, *up, recompute=not saved), g0, (saved, shape))
    finally:
        for which, saved in ((0, 0), (1, 1), (1, 0)):
            psi.psi_ctx_set_render_shape(ctx, which, r.opts, psi.F32, saved, 0)
    assert ctx.status_fetch() == (0, 0)
