"""A request's admission footprint covers what building it takes from the
arena, also when nearly every cell holds a source: the lists of the sources and
of their cells are then as large as the fields, and the receivers, on cells of
their own, make the latter grow (old and new list at once)."""
import time

import numpy as np
import pytest

from gpu_util import oracle_params, to_c

pytestmark = pytest.mark.gpu


def test_arena_of_a_footprint_holds_a_request_of_many_sources():
    torch = pytest.importorskip("torch")
    if not torch.cuda.is_available():
        pytest.skip("no GPU")
    import paper_2606_11103_gb300 as fw
    shape, n = (2048, 2048), 400
    one = np.ones(shape, np.float32)
    src, rcv = np.ones(shape, np.uint8), np.zeros(shape, np.uint8)
    src[8], rcv[8, ::64] = 0, 1
    dx = 1500.0 / 36e6
    q = dict(shape=shape, dx=dx, dt=0.3 * dx / 1530, c=1500 * one, rho=1000 * one,
             class_idx=np.zeros(shape, np.uint16), classes=[to_c(oracle_params(0.5, 1.1, 2, maxiter=60), fw)],
             n_steps=n, src_mask=src, waves=np.full((1, n), 1e-9, np.float32), rcv_mask=rcv)
    srv = fw.Server(hbm_budget=4 << 30)
    srv.submit(**q)
    footprint, done = 0, []
    while not done:
        footprint = max(footprint, srv.stats()["bytes_reserved"])
        done = srv.poll(timeout=0.001)
    srv.close()
    assert done[0]["status"] == 0 and footprint > 0
    srv = fw.Server(hbm_budget=footprint)
    srv.submit(**q)
    t_end, alone = time.time() + 60, []
    while not alone and time.time() < t_end:
        alone = srv.poll(timeout=0.5)
    srv.close()
    assert alone and alone[0]["status"] == 0
    assert np.array_equal(alone[0]["traces"], done[0]["traces"])
