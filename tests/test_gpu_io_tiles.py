"""Sources and receivers scattered over every tile of the pressure sweep (tile
edges and corners, cells that hold both, several waveforms, traces of every
third step), and sets replaced between runs, against the FP64 oracle.
Tolerances: the repository's for a run of this kind, 1e-5 (FP32) and 1e-11
(FP64), on p and the traces."""
import numpy as np
import pytest

from gpu_util import Pair, oracle_params, rel_l2

pytestmark = pytest.mark.gpu


@pytest.fixture(scope="module")
def fw():
    torch = pytest.importorskip("torch")
    if not torch.cuda.is_available():
        pytest.skip("no GPU")
    import paper_2606_11103_gb300 as fw
    fw.lib()
    return fw


@pytest.mark.parametrize("shape,storage", [((70, 261), "f32"), ((70, 261), "f64"), ((19, 23, 133), "f32"),
                                           ((19, 23, 133), "f64"), ((33, 8, 64), "f32")])
def test_scattered_sources_and_receivers(fw, shape, storage):
    rng = np.random.default_rng(11)
    one = np.ones(shape, np.float32)
    dx = 1540.0 / 36e6
    dt = 0.3 * dx / 1540.0
    pr = Pair(fw, shape, dx, dt, 1540 * one, 1000 * one, np.zeros(shape, np.uint16), [oracle_params(0.5, 1.1, 2)],
              storage=storage)
    tol = 1e-5 if storage == "f32" else 1e-11
    n = 40
    for density in (0.2, 0.03):
        src = (rng.random(shape) < density).astype(np.uint8)
        rcv = (rng.random(shape) < density).astype(np.uint8)
        src.reshape(-1)[[0, -1]] = 1
        rcv.reshape(-1)[[0, -1]] = 1
        waves = (1e3 * dx ** (len(shape) - 1) / 1.54e6 * rng.standard_normal((5, 2 * n))).astype(np.float32)
        wave_of = rng.integers(0, 5, int(src.sum())).astype(np.int32)
        pr.sources(src, waves, wave_of)
        pr.receivers(rcv, 2 * n, 3)
        pr.run(n)
        f64 = storage == "f64"
        assert rel_l2(pr.gpu.receivers(f64=f64), pr.orc.traces) <= tol
        assert rel_l2(pr.gpu.read_field(0, 0, f64=f64), pr.orc.p) <= tol
    # no receivers, then no sources: the other set stays in place
    pr.gpu.set_receivers(np.zeros(shape, np.uint8), n)
    pr.run(5)
    assert rel_l2(pr.gpu.read_field(0, 0, f64=storage == "f64"), pr.orc.p) <= tol
