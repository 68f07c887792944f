"""Host threads with a context and a stream each, calling the same entry point
with sizes that share one kernel but not its amount of shared memory (needs a
GPU): no call disturbs another's launch, every one returns PSI_OK."""
import ctypes
import sys
import threading

import pytest

torch = pytest.importorskip("torch")

from paper_2604_10982_gb300 import scenegen as sg

pytestmark = pytest.mark.gpu

CALLS = 4000


def _render_call(K, dim, adjoint, stream):
    from paper_2604_10982_gb300 import pipeline as pl, psi
    ctx = psi.Context(0)
    w = sg.dense_box(n=50, d=dim, width=16, height=16)
    scene = pl.DeviceScene(w.surfels, w.features)
    r = pl.make_renderer(ctx, scene, w.cameras, psi.default_opts(mode=psi.EXACT, top_k=K, opacity_radius=1), D=dim)
    r.frame(scene)
    P, feats, s = r.n_pix, scene.features_struct(), scene.surfels_struct()
    out = psi.PsiFwdOut(*(psi._ptr(t) for t in (r.rgb, r.T, r.n_last, r.F)), psi.F32, psi._ptr(r.topk_ids),
                        psi._ptr(r.topk_w), None)
    keep = [ctx, scene, r, feats, s, out]
    frame = (psi._ptr(r.records), psi._ptr(r.vals), psi._ptr(r.ranges), r.cams, r.V)
    opts, st = ctypes.byref(r.opts), psi._stream(stream)
    if not adjoint:
        args = (ctx.handle, ctypes.byref(feats), *frame, r.n, opts, ctypes.byref(out), st)
        return psi.lib().psi_render_fwd, args, keep
    up = [torch.ones(3, P, device="cuda"), torch.ones(P, dim, device="cuda"), torch.ones(P, device="cuda")]
    grads = r.backward(scene, *up)
    gs = psi.PsiGrads(*(psi._ptr(grads[k]) for k in ("mu", "tu", "tv", "scale", "opacity", "rgb", "feat")))
    keep += [up, grads, gs]
    args = (ctx.handle, ctypes.byref(s), ctypes.byref(feats), *frame, opts, *(psi._ptr(t) for t in up),
            ctypes.byref(out), ctypes.byref(gs), psi._ptr(r.ws_bwd), r.ws_bwd.numel(), st)
    return psi.lib().psi_render_bwd, args, keep


def _decode_call(n_q, stream):
    from paper_2604_10982_gb300 import psi
    ctx = psi.Context(0)
    F, Q = (torch.ones(n, 128, device="cuda", dtype=torch.bfloat16) for n in (64, n_q))
    T, ids = torch.zeros(64, device="cuda"), torch.empty(64, dtype=torch.int32, device="cuda")
    args = (ctx.handle, psi._ptr(F), 64, 128, psi._ptr(Q), n_q, psi._ptr(T), psi._ptr(ids), None, psi._stream(stream))
    return psi.lib().psi_decode_queries, args, [ctx, F, Q, T, ids]


@pytest.mark.parametrize("what,sizes", [("render", (1, 4, 7, 8)), ("render", (9, 12, 13, 16)), ("render", (17, 24, 29, 32)),
                                        ("adjoint", (20, 24, 28, 32)), ("decode", (10, 40, 100, 128))])
def test_threads_with_different_sizes(what, sizes):
    if not torch.cuda.is_available():
        pytest.skip("no CUDA device")
    streams = [torch.cuda.Stream() for _ in sizes]
    calls = [_decode_call(k, s) if what == "decode" else _render_call(k, 16, what == "adjoint", s)
             for k, s in zip(sizes, streams)]
    torch.cuda.synchronize()
    failed = [None] * len(sizes)
    gate = threading.Barrier(len(sizes))

    def work(i):
        torch.cuda.set_device(0)
        fn, args, _ = calls[i]
        gate.wait()
        n = 0
        for j in range(CALLS):
            n += fn(*args) != 0
            if j % 64 == 0:
                streams[i].synchronize()
        failed[i] = n

    interval = sys.getswitchinterval()
    sys.setswitchinterval(1e-6)
    try:
        threads = [threading.Thread(target=work, args=(i,)) for i in range(len(sizes))]
        for t in threads:
            t.start()
        for t in threads:
            t.join()
    finally:
        sys.setswitchinterval(interval)
    torch.cuda.synchronize()
    assert failed == [0] * len(sizes)
