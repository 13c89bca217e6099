"""A gradient leaves its medium as a plain run of the same steps does: every
field, the receiver traces and the bytes of the saved state, whatever its
device buffers held before.  The absorbing-layer memories cover the whole grid
but steps write them inside the layer only; here they hold values the caller
wrote, also outside it.  Rows with and without padding, arrays whose size is
no multiple of the alignment in the state image (13 x 15 rows), both layers,
FP64; one, two and more checkpoint segments."""
import ctypes as C

import numpy as np
import pytest

from gpu_util import oracle_params, to_c

pytestmark = pytest.mark.gpu


@pytest.fixture(scope="module")
def fw():
    torch = pytest.importorskip("torch")
    if not torch.cuda.is_available():
        pytest.skip("no GPU")
    import paper_2606_11103_gb300 as fw
    fw.lib()
    return fw


@pytest.fixture
def dirty_memory(fw):
    """Device memory of later media and gradients comes filled with NaN."""
    import torch
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
    fw.lib().fw_set_allocator(fa, ff, None)
    yield held
    fw.lib().fw_set_allocator(C.cast(None, _lib.ALLOCFN), C.cast(None, _lib.FREEFN), None)


def states_after_run_and_gradient(fw, shape, pml, transition, storage, checkpoint, n_mech=2):
    rng = np.random.default_rng(11)
    dx = 1500.0 / 36e6
    c = (1500 + 30 * rng.uniform(-1, 1, shape)).astype(np.float32)
    rho = (1000 + 30 * rng.uniform(-1, 1, shape)).astype(np.float32)
    src = np.zeros(shape, np.uint8)
    src[6] = 1
    rcv = np.zeros(shape, np.uint8)
    rcv[7, ..., ::3] = 1
    n = 24
    wave = np.sin(np.arange(n) * 0.4).astype(np.float32)[None] * 1e-6
    G = rng.standard_normal((int(rcv.sum()), n)).astype(np.float32)
    prm = [to_c(oracle_params(a, y, n_mech, maxiter=60), fw) for a, y in ((0.5, 1.1), (0.9, 1.5))]
    m = fw.Medium.from_classes(shape, dx, c, rho, rng.integers(0, 2, shape).astype(np.uint16), prm,
                               dt=0.3 * dx / 1530, pml=pml, transition=transition, storage=storage)
    m.set_sources(src, wave)
    m.set_receivers(rcv, n)
    nd = len(shape)
    names = [(fw.FW_FIELD_P, 0)] + [(fw.FW_FIELD_V, k) for k in range(nd)]
    names += [(fw.FW_FIELD_PSI1, k) for k in range(n_mech * nd)] + [(fw.FW_FIELD_PSI2, k) for k in range(n_mech)]
    layer = [(w, k) for w in (fw.FW_FIELD_PSI1P, fw.FW_FIELD_PSI2P) for k in range(nd)] if pml else []
    m.write_field(fw.FW_FIELD_P, 0, (1e3 * rng.standard_normal(shape)).astype(np.float32))
    for w, k in layer:
        m.write_field(w, k, rng.standard_normal(shape).astype(np.float32))
    start = m.save_state()
    out = []
    for gradient in (False, True):
        m.load_state(start)
        if gradient:
            m.gradient(n, G, checkpoint=checkpoint)
        else:
            m.run(n)
        f64 = storage == "f64"
        out.append([m.read_field(w, k, f64=f64) for w, k in names + layer] + [m.receivers(f64=f64), m.save_state()])
    m.close()
    return zip(names + layer + ["traces", "state"], *out)


@pytest.mark.parametrize("shape,pml,transition,storage,checkpoint", [
    ((48, 64), 4, 0, "f32", 24), ((48, 64), 4, 3, "f32", 13), ((48, 64), 4, 3, "f64", 5), ((48, 41), 4, 2, "f32", 7),
    ((14, 16, 32), 3, 0, "f32", 24), ((14, 16, 32), 3, 2, "f32", 12), ((13, 15, 32), 3, 0, "f32", 7),
    ((13, 15, 32), 3, 1, "f64", 9), ((14, 16, 23), 3, 0, "f32", 5), ((64, 96), 0, 0, "f32", 7)])
def test_state_after_a_gradient_is_that_of_a_run(fw, dirty_memory, shape, pml, transition, storage, checkpoint):
    for label, a, b in states_after_run_and_gradient(fw, shape, pml, transition, storage, checkpoint):
        assert np.array_equal(a, b), label
    assert not dirty_memory


@pytest.mark.parametrize("shape,pml,transition,checkpoint,n_mech", [
    ((1024, 1056), 9, 0, 7, 3), ((1024, 1056), 9, 4, 24, 4), ((1029, 1021), 7, 5, 9, 2), ((2049, 515), 0, 0, 7, 1),
    ((1030, 1024), 11, 0, 24, 4), ((40, 72, 130), 6, 3, 7, 1), ((40, 72, 130), 6, 0, 7, 2), ((40, 72, 130), 5, 0, 24, 3),
    ((40, 72, 130), 7, 0, 9, 4)])
def test_state_after_a_gradient_of_staged_sweeps(fw, shape, pml, transition, checkpoint, n_mech):
    """Planes from 2048 tiles on and volumes: a run takes the sweeps staged by
    TMA, the gradient's last two segments the image steps."""
    for label, a, b in states_after_run_and_gradient(fw, shape, pml, transition, "f32", checkpoint, n_mech):
        assert np.array_equal(a, b), label


def test_sides_of_the_attenuation_gradient_add_up_in_fp64(fw):
    """Each cell's terms of a step, one of the pressure and one of the velocity
    update, are FP32 sums that are added up in FP64: after one step their sum
    has more than FP32's 24 bits except where the terms' last bits happen to
    allow it (random bits: well below 9 cells of 10)."""
    shape = (12, 14, 40)
    rng = np.random.default_rng(7)
    dx = 1500.0 / 36e6
    one = np.ones(shape, np.float32)
    m = fw.Medium.from_classes(shape, dx, 1500 * one, 1000 * one, np.zeros(shape, np.uint16),
                               [to_c(oracle_params(0.5, 1.1, 2, maxiter=60), fw)], dt=0.3 * dx / 1530)
    rcv = np.ones(shape, np.uint8)
    m.set_receivers(rcv, 1)
    for w, count in ((fw.FW_FIELD_P, 1), (fw.FW_FIELD_V, 3), (fw.FW_FIELD_PSI1, 6), (fw.FW_FIELD_PSI2, 2)):
        for k in range(count):
            m.write_field(w, k, rng.standard_normal(shape).astype(np.float32))
    _, ga = m.gradient(1, rng.standard_normal((int(rcv.sum()), 1)), checkpoint=1, f64=True)
    m.close()
    assert np.isfinite(ga).all() and np.all(ga != 0)
    assert np.mean(ga != ga.astype(np.float32).astype(np.float64)) > 0.1
