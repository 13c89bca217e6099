"""The device buffers that a medium keeps from one gradient for the next: kept
within a bound, given back on request, with the medium and when the library
needs device memory, and never kept from an allocator that the caller
installed."""
import ctypes as C

import numpy as np
import pytest

from gpu_util import oracle_params, to_c

pytestmark = pytest.mark.gpu
MIB = 1 << 20


@pytest.fixture(scope="module")
def fw():
    torch = pytest.importorskip("torch")
    if not torch.cuda.is_available():
        pytest.skip("no GPU")
    import paper_2606_11103_gb300 as fw
    m, G = medium(fw, (64, 64), 4)
    m.gradient(4, G)                       # kernels and the library's static array are loaded
    m.close()
    return fw


def medium(fw, shape, n):
    prm = to_c(oracle_params(0.5, 1.1, 2, maxiter=60), fw)
    one = np.ones(shape, np.float32)
    src, rcv = np.zeros(shape, np.uint8), np.zeros(shape, np.uint8)
    src[20] = 1
    rcv[30, ::5] = 1
    m = fw.Medium.from_classes(shape, 4e-5, 1540 * one, 1000 * one, np.zeros(shape, np.uint16), [prm], cfl=0.3, pml=8)
    m.set_sources(src, np.sin(np.arange(n) * 0.4).astype(np.float32)[None] * 1e-6)
    m.set_receivers(rcv, n)
    return m, np.random.default_rng(0).standard_normal((int(rcv.sum()), n)).astype(np.float32)


def free_bytes():
    import torch
    torch.cuda.synchronize()
    return torch.cuda.mem_get_info()[0]


def test_kept_for_the_next_gradient_and_given_back(fw):
    # (images of 13 MiB: checkpoint = 24 holds 50 of them, 0.65 GiB)
    free0 = free_bytes()
    m, G = medium(fw, (512, 512), 48)
    start = m.save_state()
    out, kept = [], []
    for step in range(4):
        m.load_state(start)
        out.append(m.gradient(48, G, checkpoint=24))
        kept.append(free0 - free_bytes())
        if step == 1:
            m.release_workspace()
            assert free0 - free_bytes() < 64 * MIB
    assert all(600 * MIB < k < 900 * MIB for k in kept) and kept[0] == kept[1]
    for gc, ga in out[1:]:
        assert np.array_equal(gc, out[0][0]) and np.array_equal(ga, out[0][1])
    fw.check(fw.lib().fw_release_workspace(None))          # every medium's
    assert free0 - free_bytes() < 64 * MIB
    m.load_state(start)
    m.gradient(48, G, checkpoint=24)
    m.close()
    assert free0 - free_bytes() < 16 * MIB


def test_given_back_to_a_server_that_needs_the_memory(fw):
    m, G = medium(fw, (512, 512), 48)
    before = free_bytes()
    m.gradient(48, G, checkpoint=24)
    kept = before - free_bytes()
    assert kept > 600 * MIB
    srv = fw.Server(hbm_budget=free_bytes() + kept // 2)
    srv.close()
    m.close()


def test_bounded_over_all_media(fw):
    """With 8 GiB free for the library, four media of 0.65 GiB each: no more kept
    than a quarter of what is left, and the results are those of one alone."""
    import torch
    free0 = free_bytes()
    rest = torch.empty(free0 - (8 << 30), dtype=torch.uint8, device="cuda")
    media = [medium(fw, (512, 512), 48) for _ in range(4)]
    before = free_bytes()
    out = [m.gradient(48, G, checkpoint=24) for m, G in media]
    left = free_bytes()
    assert 600 * MIB < before - left <= left // 4
    for gc, ga in out[1:]:
        assert np.array_equal(gc, out[0][0]) and np.array_equal(ga, out[0][1])
    for m, _ in media:
        m.close()
    del rest
    torch.cuda.empty_cache()
    assert free0 - free_bytes() < 16 * MIB


def test_nothing_kept_from_an_installed_allocator(fw):
    import torch
    from paper_2606_11103_gb300 import _lib
    held = {}

    def alloc(nbytes, ctx):
        t = torch.empty(int(nbytes), dtype=torch.uint8, device="cuda")
        held[t.data_ptr()] = t
        return t.data_ptr()

    def release(ptr, ctx):
        torch.cuda.synchronize()
        held.pop(ptr)

    fa, ff = _lib.ALLOCFN(alloc), _lib.FREEFN(release)
    fw.lib().fw_set_allocator(fa, ff, None)
    try:
        m, G = medium(fw, (96, 80), 12)
        own = set(held)
        m.gradient(12, G)
        assert set(held) == own
        m.close()
        assert not held
    finally:
        fw.lib().fw_set_allocator(C.cast(None, _lib.ALLOCFN), C.cast(None, _lib.FREEFN), None)
