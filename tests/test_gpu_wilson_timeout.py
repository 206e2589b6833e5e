"""The copy waits of the tiled fine operator are bounded and a warp leaves as a
whole: launches made to wait for bytes that never come (their own time runs
out, no fault of the GPU) end, report the error, and the next apply on the same
context is correct, for one vector and several, on whole and partial blocks."""
import time

import pytest
import torch

import synthetic as syn
from oracle import lattice as lat
from gpu_helpers import make_ctx, oracle_fine, rel_l2, to_dev, to_np

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("policy", [12, 14])
@pytest.mark.parametrize("nrhs", [1, 3])
def test_stalled_tile_times_out_and_context_stays_usable(gpu_lib, policy, nrhs):
    gb = gpu_lib
    dims = (10, 4, 6, 4)
    vol = lat.volume(dims)
    mg, U = make_ctx(gb, dims, [(2, 2, 2, 2)], [4], prec_fine=1, prec_coarse=1)
    x = syn.gaussian_field((nrhs, vol, 12), 71)
    xd = to_dev(x, torch.complex64)
    y = torch.zeros_like(xd)
    key = f"wilson/v{vol}/n{nrhs}/c1"

    def apply():
        if nrhs == 1:
            gb.mg_wilson_clover_apply(mg.ctx, y[0], xd[0])
        else:
            gb.mg_wilson_clover_apply_multi(mg.ctx, y, xd, nrhs)

    gb.mg_tune_set(key, policy)
    gb.mg_inject_fault(mg.ctx, "wilson_tile_wait", 1)
    t0 = time.monotonic()
    apply()
    with pytest.raises(gb.MGError) as e:
        gb.mg_device_status(mg.ctx)
    assert e.value.status == gb.MG_ERR_TIMEOUT
    assert 0.9 < time.monotonic() - t0 < 30.0  # one second, and a second one per tile in flight
    gb.mg_device_status(mg.ctx)  # the record was cleared
    apply()
    gb.mg_device_status(mg.ctx)
    op = oracle_fine(U, dims)
    for v in range(nrhs):
        assert rel_l2(to_np(y[v]), op.apply(x[v])) < 1e-5  # the FP32 tier
    gb.mg_tune_set(key, -1)
    mg.close()
