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


@pytest.mark.parametrize("n,passes_bits", [(300_000, 45), (2_000_000, 61)])
def test_sort_giveup_leaves_empty_lists(ctx, n, passes_bits):
    """74 and 489 partitions, 6 and 8 passes. A poll fails as soon as a partition
    is ahead of its predecessor."""
    from paper_2604_10982_gb300 import psi
    n_tiles, capacity = 1500, n + 5
    rng = np.random.default_rng(n)
    keys = (rng.integers(0, n_tiles, n).astype(np.uint64) << np.uint64(32)) | rng.integers(0, 2**31, n).astype(np.uint64)
    pad = np.full(capacity - n, 7, np.uint64)
    k0 = torch.from_numpy(np.concatenate([keys, pad]).view(np.int64)).cuda()
    v0 = torch.arange(capacity, dtype=torch.int32, device="cuda")
    keys_b, k = _guarded(capacity, torch.int64)
    vals_b, v = _guarded(capacity, torch.int32)
    rg_b, ranges = _guarded(3 * n_tiles, torch.int32)
    ws_b, ws = _guarded(psi.sort_workspace_size(capacity), torch.uint8)
    num = torch.tensor([n], dtype=torch.int64, device="cuda")

    def sort():
        k.copy_(k0)
        v.copy_(v0)
        psi.psi_sort_keys(ctx, k, v, num, capacity, 0, passes_bits, ranges, n_tiles, ws)
        return ctx.status_fetch()

    psi.psi_ctx_set_wait_limit_ns(ctx, 1)
    for _ in range(TRIES):
        st = sort()
        if st[0]:
            break
    assert st == (psi.PSI_ERR_TIMEOUT, 8)
    assert torch.count_nonzero(ranges[:2 * n_tiles]).item() == 0
    assert torch.equal(ranges[2 * n_tiles:].sort()[0], torch.arange(n_tiles, dtype=torch.int32, device="cuda"))
    assert _intact(keys_b, vals_b, rg_b, ws_b)
    assert torch.equal(k[n:], k0[n:]) and torch.equal(v[n:], v0[n:])

    psi.psi_ctx_set_wait_limit_ns(ctx, 0)
    assert sort() == (0, 0)
    order = np.argsort(keys, kind="stable")
    assert np.array_equal(k.cpu().numpy().view(np.uint64)[:n], keys[order])
    assert np.array_equal(v.cpu().numpy()[:n], order.astype(np.int32))
    assert _intact(keys_b, vals_b, rg_b, ws_b)
