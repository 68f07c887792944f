"""Saved state that no frame wrote (needs a GPU) -- what an adjoint queued
behind a forward that gave up can find: ids outside the table count as empty
slots, last positions are cut to the tile's list, nothing is touched outside
the gradients."""
import pytest

torch = pytest.importorskip("torch")

from oracle import oracle as orc
from paper_2604_10982_gb300 import scenegen as sg

from .gpu_common import multi_cams, opts_of

pytestmark = pytest.mark.gpu

G = 4096
WIDTHS = dict(mu=3, tu=3, tv=3, scale=2, opacity=1, rgb=3)


@pytest.mark.parametrize("K,D", [(8, 32), (16, 128), (5, 256)])
def test_foreign_ids_are_empty_slots(K, D):
    if not torch.cuda.is_available():
        pytest.skip("no CUDA device")
    from paper_2604_10982_gb300 import pipeline as pl, psi
    ctx = psi.Context(0)
    if psi.lib().psi_debug_checks():
        pytest.skip("the debug build reports such ids")
    n = 2000
    w = sg.dense_box(n=n, d=D)
    scene = pl.DeviceScene(w.surfels, w.features)
    r = pl.make_renderer(ctx, scene, multi_cams(), opts_of(orc.Opts(mode=orc.EXACT, top_k=K, opacity_radius=True)), D=D)
    r.frame(scene)
    P = r.n_pix
    gen = torch.Generator(device="cpu").manual_seed(1)
    up = [torch.randn(*s, generator=gen).cuda() for s in ((3, P), (P, D), (P,))]
    foreign = torch.tensor([-2, -(2**31), n, n + 1, 2**31 - 1], dtype=torch.int32)
    hit = torch.rand(P, K, generator=gen) < 0.3
    bad = foreign[torch.randint(0, 5, (P, K), generator=gen)].cuda()
    ids = r.topk_ids.clone()

    def grads():
        bigs = {k: torch.full((n * c + 2 * G,), 3.0, device="cuda") for k, c in dict(WIDTHS, feat=D).items()}
        gr = {k: b[G:-G].zero_() for k, b in bigs.items()}
        r.backward(scene, *up, grads=gr)
        assert ctx.status_fetch() == (0, 0)
        assert all(bool((b[:G] == 3).all()) and bool((b[-G:] == 3).all()) for b in bigs.values())
        return {k: v.double() for k, v in gr.items()}

    r.topk_ids.copy_(torch.where(hit.cuda(), torch.full_like(ids, -1), ids))
    empty = grads()
    r.topk_ids.copy_(torch.where(hit.cuda(), bad, ids))
    for k, v in grads().items():  # the same sums in another order of float32 additions
        assert torch.linalg.norm(v - empty[k]).item() <= 1e-5 * torch.linalg.norm(empty[k]).item(), k
    # positions past every list, and before it
    r.n_last.copy_(torch.where(torch.rand(P, generator=gen) < 0.5, torch.tensor(2**31 - 1, dtype=torch.int32),
                               torch.tensor(-7, dtype=torch.int32)).cuda())
    grads()
