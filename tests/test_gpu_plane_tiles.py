"""2D sweeps staged by TMA (grids from 2048 tiles of 128 x 4 points on) against
the unstaged 2D sweeps on the same medium: odd sides, partial tiles at both
edges, every storage, both time schemes, with and without the absorbing layer
and the nonlinear factor.

Both forms do the same FP32 operations per cell in the same order; only the
compiler's contraction of a product and a sum may differ, an ulp (6e-8) per
operation.  Tolerance on the relative L2 difference after 40 steps: 1e-5, the
repository's FP32 target (bfloat16 and binary16 memory variables: times the
share of the stretched derivative they carry, about 1e-2, over their roundoff
2^-8 and 2^-11 at most once per step: 1e-3)."""
import numpy as np
import pytest

from gpu_util import oracle_params, rel_l2, to_c

pytestmark = pytest.mark.gpu


@pytest.fixture(scope="module")
def fw():
    torch = pytest.importorskip("torch")
    if not torch.cuda.is_available():
        pytest.skip("no GPU")
    import paper_2606_11103_gb300 as fw
    fw.lib()
    return fw


@pytest.mark.parametrize("shape,storage,order,pml,lt,nl,nmech", [
    ((1029, 1021), "f32", 2, 11, 0, False, 4),
    ((1029, 1021), "f32", 4, 11, 5, True, 3),
    ((4097, 257), "f32", 2, 7, 4, True, 2),
    ((205, 5121), "f32", 4, 0, 0, False, 1),
    ((1025, 1027), "bf16", 2, 9, 0, False, 4),
    ((1031, 1150), "f16", 4, 9, 3, False, 2),
    ((16385, 513), "f32", 2, 13, 0, False, 1),     # 20485 tiles: runs of four
])
def test_staged_sweeps_equal_unstaged(fw, monkeypatch, shape, storage, order, pml, lt, nl, nmech):
    rng = np.random.default_rng(5)
    params = [oracle_params(a, y, nmech, maxiter=60) for a, y in ((0.5, 1.1), (0.9, 1.6), (0.0, 1.0))]
    cls = rng.integers(0, 3, ((shape[0] + 36) // 37, (shape[1] + 28) // 29))
    cls = np.kron(cls, np.ones((37, 29), np.int64))[:shape[0], :shape[1]].astype(np.uint16)
    c = (1500 + 60 * rng.uniform(-1, 1, shape)).astype(np.float32)
    rho = (1000 + 60 * rng.uniform(-1, 1, shape)).astype(np.float32)
    beta = (3 + rng.uniform(0, 2, shape)).astype(np.float32) if nl else None
    dx = 1500.0 / (3e6 * 12)
    dt = 0.3 * dx / 1560.0
    p0 = (1e3 * rng.standard_normal(shape)).astype(np.float32)
    src = np.zeros(shape, np.uint8)
    src[shape[0] // 2, ::7] = 1
    rcv = np.zeros(shape, np.uint8)
    rcv[shape[0] // 3, ::11] = 1
    wave = (1e3 * dx / 1.5e6 * np.sin(np.arange(40) * 0.5)).astype(np.float32)[None]
    out = []
    for staged in (True, False):
        if staged:
            monkeypatch.delenv("FWGB_NO_TMA", raising=False)
        else:
            monkeypatch.setenv("FWGB_NO_TMA", "1")
        m = fw.Medium.from_classes(shape, dx, c, rho, cls, [to_c(p, fw) for p in params], dt=dt, beta=beta, pml=pml,
                                   transition=lt, storage=storage, time_order=order)
        m.set_sources(src, wave)
        m.set_receivers(rcv, 40)
        m.write_field(fw.FW_FIELD_P, 0, p0)
        m.run(40)
        rc, top = m.status()
        fields = [m.read_field(0), m.read_field(1, 0), m.read_field(1, 1)]
        fields += [m.read_field(fw.FW_FIELD_PSI1, k) for k in range(2 * nmech)]
        fields += [m.read_field(fw.FW_FIELD_PSI2, k) for k in range(nmech)]
        if pml:
            fields += [m.read_field(w, k) for w in (fw.FW_FIELD_PSI1P, fw.FW_FIELD_PSI2P) for k in range(2)]
        out.append((rc, top, fields + [m.receivers()]))
        m.close()
    assert out[0][0] == out[1][0] == 0
    tol = 1e-5 if storage == "f32" else 1e-3
    assert abs(out[0][1] - out[1][1]) <= tol * out[1][1]
    errs = [rel_l2(a, b) if np.any(b) else float(np.abs(a).max()) for a, b in zip(out[0][2], out[1][2])]
    print("largest difference %.2e" % max(errs))
    assert max(errs) <= tol
