"""The sort's kernel count as the library reports it: the forms that the
documentation names (host only), and what the profiler sees (GPU)."""
import ctypes

import pytest

torch = pytest.importorskip("torch")

from paper_2604_10982_gb300 import _build, psi


@pytest.fixture(scope="module")
def lib():
    _build.build()
    return psi.lib()


def test_counts(lib):
    assert psi.sort_kernel_count(1000, 0, 45, 300) == 1
    assert psi.sort_kernel_count(1 << 20, 0, 45, 300) == 2 + 6 + 2    # digit counts and scan, passes, ranges and order
    assert psi.sort_kernel_count(1 << 20, 0, 45, 0) == 2 + 6
    assert psi.sort_kernel_count(1 << 20, 0, 33, 300) == 2 + 6 + 2    # 5 digits: an even number of passes
    assert psi.sort_kernel_count(1 << 20, 0, 64, 300) == 2 + 8 + 2
    # the one-CTA form: up to 8192 pairs and, with ranges, 16384 tiles
    for cap, tiles, one in ((8192, 16384, True), (8193, 16384, False), (8192, 16385, False), (8192, 0, True)):
        assert (psi.sort_kernel_count(cap, 0, 45, tiles) == 1) == one, (cap, tiles)
    k = ctypes.c_int(0)
    for bad in ((-1, 0, 45, 1), (10, -1, 45, 1), (10, 0, 65, 1), (10, 5, 5, 1), (10, 0, 45, -1)):
        assert lib.psi_sort_kernel_count(*bad, ctypes.byref(k)) == psi.PSI_ERR_INVALID_ARG
    assert lib.psi_sort_kernel_count(10, 0, 45, 1, None) == psi.PSI_ERR_INVALID_ARG


@pytest.mark.gpu
@pytest.mark.parametrize("capacity,n_tiles", [(100, 4), (8192, 300), (8193, 300), (6144, 16384), (8192, 16384), (8192, 16385),
                                              (100_000, 300)])
def test_counts_are_what_launches(capacity, n_tiles):
    if not torch.cuda.is_available():
        pytest.skip("no CUDA device")
    from torch.profiler import ProfilerActivity, profile
    ctx = psi.Context(0)
    n = 90
    keys = torch.arange(capacity, dtype=torch.int64, device="cuda") % n_tiles << 32
    vals = torch.arange(capacity, dtype=torch.int32, device="cuda")
    num = torch.tensor([n], dtype=torch.int64, device="cuda")
    ranges = torch.empty(3 * n_tiles, dtype=torch.int32, device="cuda")
    ws = torch.empty(psi.sort_workspace_size(capacity), dtype=torch.uint8, device="cuda")
    run = lambda: psi.psi_sort_keys(ctx, keys, vals, num, capacity, 0, 48, ranges, n_tiles, ws)  # noqa: E731
    run()
    torch.cuda.synchronize()
    for _ in range(5):  # a process's first profiling session can come back without device events
        with profile(activities=[ProfilerActivity.CPU, ProfilerActivity.CUDA]) as p:
            run()
            torch.cuda.synchronize()
        launched = [e.name for e in p.events() if e.device_type == torch.autograd.DeviceType.CUDA and "psi::" in e.name]
        if launched:
            break
    assert len(launched) == psi.sort_kernel_count(capacity, 0, 48, n_tiles), launched
    assert ctx.status_fetch() == (0, 0)
