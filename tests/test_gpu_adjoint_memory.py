"""A gradient does not depend on what its device buffers held before: the
images of recomputed and kept steps read as zero in the padding of a row.  The
allocator hook hands out memory filled with NaN bit patterns; grids whose rows
have padding (41 and 23 columns) and a tail segment shorter than the others,
every number of checkpoint segments from one up."""
import ctypes as C

import numpy as np
import pytest

from gpu_util import oracle_params, to_c

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("shape,checkpoint", [((48, 41), 40), ((48, 41), 25), ((48, 41), 11), ((14, 16, 23), 9)])
def test_gradient_with_dirty_device_memory(shape, checkpoint):
    torch = pytest.importorskip("torch")
    if not torch.cuda.is_available():
        pytest.skip("no GPU")
    import paper_2606_11103_gb300 as fw
    from paper_2606_11103_gb300 import _lib
    held = {}

    def alloc(nbytes, ctx):
        t = torch.full(((int(nbytes) + 255) // 256 * 256,), 255, dtype=torch.uint8, device="cuda")
        torch.cuda.synchronize()
        held[t.data_ptr()] = t
        return t.data_ptr()

    def release(ptr, ctx):
        torch.cuda.synchronize()
        held.pop(ptr, None)

    fa, ff = _lib.ALLOCFN(alloc), _lib.FREEFN(release)
    rng = np.random.default_rng(3)
    dx = 1500.0 / 36e6
    c = (1500 + 30 * rng.uniform(-1, 1, shape)).astype(np.float32)
    rho = (1000 + 30 * rng.uniform(-1, 1, shape)).astype(np.float32)
    src = np.zeros(shape, np.uint8)
    src[6] = 1
    rcv = np.zeros(shape, np.uint8)
    rcv[8, ..., ::3] = 1
    n = 40
    wave = np.sin(np.arange(n) * 0.4).astype(np.float32)[None] * 1e-6
    G = rng.standard_normal((int(rcv.sum()), n)).astype(np.float32)
    prm = to_c(oracle_params(0.5, 1.1, 2, maxiter=60), fw)
    out = []
    for dirty in (False, True):
        if dirty:
            fw.lib().fw_set_allocator(fa, ff, None)
        try:
            m = fw.Medium.from_classes(shape, dx, c, rho, np.zeros(shape, np.uint16), [prm], dt=0.3 * dx / 1530, pml=4)
            m.set_sources(src, wave)
            m.set_receivers(rcv, n)
            gc, ga = m.gradient(n, G, checkpoint=checkpoint)
            out.append((gc, ga, m.receivers(), m.read_field(0), m.info()["step"], m.status()))
            m.run(5)
            out[-1] += (m.read_field(0),)
            m.close()
        finally:
            fw.lib().fw_set_allocator(C.cast(None, _lib.ALLOCFN), C.cast(None, _lib.FREEFN), None)
    assert not held
    for a, b in zip(out[0], out[1]):
        assert np.array_equal(a, b)
    assert np.isfinite(out[1][0]).all() and np.abs(out[1][0]).max() > 0


def test_workspace_is_kept_and_given_back():
    """Gradients of one medium reuse their device buffers (also after a larger
    one) and give the same result; the memory comes back with the medium."""
    torch = pytest.importorskip("torch")
    if not torch.cuda.is_available():
        pytest.skip("no GPU")
    import paper_2606_11103_gb300 as fw
    shape, n = (300, 310), 24
    prm = to_c(oracle_params(0.5, 1.1, 2, maxiter=60), fw)
    one = np.ones(shape, np.float32)
    src = np.zeros(shape, np.uint8)
    src[20] = 1
    rcv = np.zeros(shape, np.uint8)
    rcv[30, ::5] = 1
    G = np.random.default_rng(0).standard_normal((int(rcv.sum()), n)).astype(np.float32)
    wave = np.sin(np.arange(n) * 0.4).astype(np.float32)[None] * 1e-6
    torch.cuda.synchronize()
    free0 = torch.cuda.mem_get_info()[0]
    m = fw.Medium.from_classes(shape, 4e-5, 1540 * one, 1000 * one, np.zeros(shape, np.uint16), [prm], cfl=0.3, pml=8)
    m.set_sources(src, wave)
    m.set_receivers(rcv, n)
    start = m.save_state()
    out = []
    for checkpoint in (6, 24, 6, 3):
        m.load_state(start)
        out.append(m.gradient(n, G, checkpoint=checkpoint))
    for gc, ga in out[1:]:
        assert np.array_equal(gc, out[0][0]) and np.array_equal(ga, out[0][1])
    m.close()
    torch.cuda.synchronize()
    assert abs(torch.cuda.mem_get_info()[0] - free0) < 256 << 20     # the library's own code and staging array stay
