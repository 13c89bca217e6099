"""Reading a field into device memory: the kernel writes a destination of this
device directly, also at odd offsets inside an allocation; one that is too
small for the field is refused, nothing written."""
import ctypes as C

import numpy as np
import pytest

from gpu_util import oracle_params, to_c

pytestmark = pytest.mark.gpu
SHAPE = (64, 60)


@pytest.fixture
def medium():
    torch = pytest.importorskip("torch")
    if not torch.cuda.is_available():
        pytest.skip("no GPU")
    import paper_2606_11103_gb300 as fw
    one = np.ones(SHAPE, np.float32)
    m = fw.Medium.from_classes(SHAPE, 4e-5, 1540 * one, 1000 * one, np.zeros(SHAPE, np.uint16),
                               [to_c(oracle_params(0.5, 1.1, 2, maxiter=60), fw)], cfl=0.3)
    p = np.random.default_rng(0).standard_normal(SHAPE).astype(np.float32)
    m.write_field(fw.FW_FIELD_P, 0, p)
    yield fw, m, p
    m.close()


@pytest.mark.parametrize("f64", [False, True])
@pytest.mark.parametrize("offset", [0, 1, 8, 12])          # bytes into the allocation: aligned for the type or not
def test_device_destination(medium, f64, offset):
    import torch
    fw, m, p = medium
    eb = 8 if f64 else 4
    buf = torch.full((p.size * eb + 64,), 255, dtype=torch.uint8, device="cuda")
    fw.check(fw.lib().fw_read_field(m.h, fw.FW_FIELD_P, 0, C.c_void_p(buf.data_ptr() + offset), int(f64), None))
    h = buf.cpu().numpy()
    assert np.array_equal(h[offset:offset + p.size * eb].view(np.float64 if f64 else np.float32).reshape(SHAPE), p)
    assert (h[:offset] == 255).all() and (h[offset + p.size * eb:] == 255).all()


def test_destination_too_small_is_refused(medium):
    """Blocks of 4 KiB from one page of 2 MiB: the one asked for lies among
    others, so that no byte outside this process's memory is at stake."""
    import torch
    fw, m, p = medium
    rt = C.CDLL("libcudart.so.13")
    rt.cudaFree.argtypes = [C.c_void_p]
    blocks = [C.c_void_p() for _ in range(64)]
    for b in blocks:
        assert rt.cudaMalloc(C.byref(b), C.c_size_t(4096)) == 0
    at = sorted(b.value for b in blocks)
    dst = next((a for a, e in zip(at, at[16:]) if e - a < 1 << 20 and a >> 21 == e >> 21), None)
    try:
        if dst is None:
            pytest.skip("the blocks do not lie together")
        assert fw.lib().fw_read_field(m.h, fw.FW_FIELD_P, 0, C.c_void_p(dst), 0, None) == fw._lib.FW_ERR_CUDA
    finally:
        rt.cudaGetLastError()
        for b in blocks:
            rt.cudaFree(b)
    torch.cuda.synchronize()
    assert np.array_equal(m.read_field(fw.FW_FIELD_P, 0), p)
