"""Tile lists at the sizes where the staging, the group lists and the Top-K
storage change over (needs a GPU): around the 32 records of a chunk, the 128
of a batch, the 256 the pixel warps stage themselves, the ring's wrap and
past it, for selections in registers (K <= 8), in shared memory (K > 8) and
dense features; the small and the general sort around their boundary.

The tolerances are the parity bars of this suite: check_values (1e-4 on colour
and T, times the largest feature on F) and 1e-3 relative L2 on gradients, plus
1e-5 between the two adjoint forms (only the order of additions differs)."""
import numpy as np
import pytest

torch = pytest.importorskip("torch")

from oracle import oracle as orc
from paper_2604_10982_gb300 import scenegen as sg

from .gpu_common import check_values, opts_of
from .test_gpu_grad import _grad_compare

pytestmark = pytest.mark.gpu


@pytest.fixture(scope="module")
def ctx():
    if not torch.cuda.is_available():
        pytest.skip("no CUDA device")
    from paper_2604_10982_gb300 import psi
    return psi.Context(0)


def _stack(n, d, seed=5):
    """n surfels stacked along the view axis of a 20x18 image (four tiles, two
    of them ragged): half of them wide enough for every tile, half a few pixels
    across, faint enough that most pixels composite their whole list."""
    u = lambda k, m: sg.uniform(seed, 100 + k, m)  # noqa: E731
    cam = sg.look_camera((0.0, -4.0, 1.0), 0.0, 20, 18, 20.0)
    z = 2.0 + np.arange(n) * (3.0 / max(n, 1))
    wide = np.arange(n) % 2 == 0
    x = np.where(wide, 0.05, 0.7) * (u(0, n) - 0.5) * z
    y = np.where(wide, 0.05, 0.7) * (u(1, n) - 0.5) * z
    c = np.stack([x, y, z], 1)
    R, t = cam.R, cam.t
    th = 0.6 * (u(2, n) - 0.5)  # tilt about the camera's x axis
    tu = np.stack([np.ones(n), np.zeros(n), np.zeros(n)], 1)
    tv = np.stack([np.zeros(n), np.cos(th), np.sin(th)], 1)
    sc = np.where(wide, 0.45, 0.06)[:, None] * z[:, None] * (0.8 + 0.4 * u(3, 2 * n).reshape(n, 2))
    f32 = lambda a: np.ascontiguousarray(a, dtype=np.float32)  # noqa: E731
    s = sg.Surfels(f32((c - t) @ R), f32(tu @ R), f32(tv @ R), f32(sc), f32(0.008 + 0.03 * u(4, n)),
                   f32(u(5, 3 * n).reshape(n, 3)))
    return sg.Workload(f"stack-{n}", s, [cam], d, 8, sg.make_features(n, d, seed))


@pytest.mark.parametrize("n", [1, 31, 33, 127, 129, 255, 257, 513, 900])
@pytest.mark.parametrize("K,D,dtype", [(8, 64, "BF16"), (5, 48, "FP8_E4M3"), (16, 128, "F32"), (32, 256, "BF16"), (0, 16, "F32")])
def test_list_lengths(ctx, n, K, D, dtype):
    from paper_2604_10982_gb300 import pipeline as pl, psi
    w = _stack(n, D)
    cam = w.cameras[0]
    o = orc.Opts(mode=orc.EXACT, top_k=K, opacity_radius=True)
    fdt = getattr(psi, dtype)
    scene = pl.DeviceScene(w.surfels, w.features, feat_dtype=fdt)
    r = pl.make_renderer(ctx, scene, [cam], opts_of(o), D=D)
    r.frame(scene)
    torch.cuda.synchronize()
    assert ctx.status_fetch() == (0, 0)
    deq = pl.dequantize(scene.q, scene.qscale, fdt)
    ref = orc.render(w.surfels, cam, o, feat=deq)
    check_values(r.rgb.cpu().numpy().astype(np.float64).T, r.T.cpu().numpy().astype(np.float64),
                 r.F.cpu().numpy().astype(np.float64), ref, cam, max_excused=0.2, fmax=np.abs(deq).max())


@pytest.mark.parametrize("n", [129, 513])
@pytest.mark.parametrize("K,D", [(8, 32), (16, 128), (20, 64), (0, 16)])
def test_list_length_gradients(ctx, n, K, D):
    w = _stack(n, D)
    _grad_compare(ctx, w, w.cameras, orc.Opts(mode=orc.EXACT, top_k=K, opacity_radius=True), D)


@pytest.mark.parametrize("capacity", [8192, 8193])
@pytest.mark.parametrize("n,end_bit", [(0, 45), (1, 45), (1023, 33), (1025, 41), (8191, 45), (8192, 64)])
def test_small_and_general_sort_agree(ctx, capacity, n, end_bit):
    """The one-CTA sort (capacity <= 8192) and the general one give the stable
    order, the ranges and a launch order of all tiles."""
    from paper_2604_10982_gb300 import psi
    n_tiles = 300
    rng = np.random.default_rng(n + end_bit)
    tile = rng.integers(0, n_tiles if end_bit > 40 else 2, n).astype(np.uint64)
    keys = (tile << np.uint64(32)) | rng.integers(0, 50, n).astype(np.uint64)  # many equal depths
    vals = np.arange(n, dtype=np.uint32)
    pad = capacity - n
    k = torch.from_numpy(np.concatenate([keys, np.full(pad, 7, np.uint64)]).view(np.int64)).cuda()
    v = torch.from_numpy(np.concatenate([vals, np.full(pad, 9, np.uint32)]).view(np.int32)).cuda()
    num = torch.tensor([n], dtype=torch.int64, device="cuda")
    ranges = torch.full((3 * n_tiles,), -1, dtype=torch.int32, device="cuda")
    ws = torch.empty(psi.sort_workspace_size(capacity), dtype=torch.uint8, device="cuda")
    psi.psi_sort_keys(ctx, k, v, num, capacity, 0, end_bit, ranges, n_tiles, ws)
    assert ctx.status_fetch() == (0, 0)
    order = np.argsort(keys, kind="stable")
    assert np.array_equal(k.cpu().numpy().view(np.uint64)[:n], keys[order])
    assert np.array_equal(v.cpu().numpy().view(np.uint32)[:n], vals[order])
    assert (k.cpu().numpy()[n:] == 7).all() and (v.cpu().numpy()[n:] == 9).all()
    rg = ranges.cpu().numpy()
    cnt = np.bincount(tile.astype(np.int64), minlength=n_tiles)
    assert np.array_equal(rg[: 2 * n_tiles].reshape(-1, 2)[:, 1] - rg[: 2 * n_tiles].reshape(-1, 2)[:, 0], cnt)
    assert np.array_equal(np.sort(rg[2 * n_tiles:]), np.arange(n_tiles))
