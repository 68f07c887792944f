"""Give-ups of the binning stages' look-backs (needs a GPU): a wait that runs
out raises PSI_ERR_TIMEOUT with its site and leaves nothing that the stages
queued behind it could follow out of a buffer -- no pairs, empty lists -- and
with the default limit restored the same buffers give the clean result."""
import numpy as np
import pytest

torch = pytest.importorskip("torch")

from oracle import oracle as orc
from paper_2604_10982_gb300 import scenegen as sg

from .gpu_common import opts_of

pytestmark = pytest.mark.gpu

G = 4096      # guard elements on both sides of every output
GUARD = 0x5A
TRIES = 50    # launches within which a wait of 1 ns must have run out once


@pytest.fixture()
def ctx():
    if not torch.cuda.is_available():
        pytest.skip("no CUDA device")
    from paper_2604_10982_gb300 import psi
    c = psi.Context(0)
    yield c
    psi.psi_ctx_set_wait_limit_ns(c, 0)


def _guarded(n, dtype):
    big = torch.full((n + 2 * G,), GUARD, dtype=dtype, device="cuda")
    return big, big[G:G + n]


def _intact(*bigs):
    return all(bool((b[:G] == GUARD).all()) and bool((b[-G:] == GUARD).all()) for b in bigs)


def test_intersect_giveup_leaves_no_pairs(ctx):
    """16 views of 60k surfels (938 blocks). A poll fails as soon as a block is
    ahead of one of its 32 predecessors."""
    from paper_2604_10982_gb300 import pipeline as pl, psi
    w = sg.dense_box(n=60_000, d=16)
    cams = [sg.look_camera((0.05 * i - 0.4, -6.0, 1.5), 0.02 * i - 0.15, 40 + i, 33 + i, 40.0) for i in range(16)]
    o = orc.Opts(mode=orc.EXACT, top_k=8, opacity_radius=True)
    scene = pl.DeviceScene(w.surfels, w.features)
    r = pl.make_renderer(ctx, scene, cams, opts_of(o), D=16)
    outs = lambda: [t.clone() for t in (r.rgb, r.T, r.n_last, r.F, r.topk_ids, r.topk_w)]  # noqa: E731
    r.frame(scene)
    assert ctx.status_fetch() == (0, 0)
    pairs, clean = int(r.num_pairs.item()), outs()
    assert pairs > 0 and pairs <= r.capacity
    keys_b, r.keys = _guarded(r.capacity, torch.int64)
    vals_b, r.vals = _guarded(r.capacity, torch.int32)
    ws_b, r.ws_isect = _guarded(psi.intersect_workspace_size(16 * scene.n), torch.uint8)
    assert r.ws_isect.data_ptr() % 256 == 0

    psi.psi_ctx_set_wait_limit_ns(ctx, 1)
    for _ in range(TRIES):
        r.num_pairs.fill_(-1)
        r.intersect()
        st, site = ctx.status_fetch()
        if st:
            break
        assert int(r.num_pairs.item()) == pairs
    assert (st, site) == (psi.PSI_ERR_TIMEOUT, 9)
    assert int(r.num_pairs.item()) == 0
    assert _intact(keys_b, vals_b, ws_b)
    psi.psi_ctx_set_wait_limit_ns(ctx, 0)
    # the stages behind it: an empty frame
    r.sort()
    r.render(scene)
    assert ctx.status_fetch() == (0, 0)
    assert torch.count_nonzero(r.rgb).item() == 0 and bool((r.T == 1).all()) and bool((r.topk_ids == -1).all())

    r.frame(scene)
    assert ctx.status_fetch() == (0, 0)
    assert int(r.num_pairs.item()) == pairs and _intact(keys_b, vals_b, ws_b)
    for a, b in zip(outs(), clean):
        assert torch.equal(a, b)
