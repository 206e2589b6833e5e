"""The waits of the tensor-core Galerkin build are bounded and its roles leave
together: the thread that issues the MMAs is made to wait on a barrier that
nothing arrives at (its own time runs out, no fault of the GPU), the producing
and draining warps, which wait for it, must follow at once, the error is
reported, and the next build on the same context is correct."""
import time

import pytest
import torch

import synthetic as syn
from oracle import lattice as lat, multigrid as mgo
from gpu_helpers import make_ctx, oracle_fine, rel_l2, to_dev, to_np

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("nv", [16, 24])
def test_stalled_build_times_out_and_context_stays_usable(gpu_lib, nv):
    gb = gpu_lib
    dims, block = (4, 4, 4, 8), (2, 2, 2, 4)
    mg, U = make_ctx(gb, dims, [block], [nv], prec_fine=1, prec_coarse=1, eps=0.5)
    v = syn.gaussian_field((nv, lat.volume(dims), 12), 31)
    gb.mg_set_nullvecs(mg.ctx, 0, to_dev(v))
    out = torch.empty((mg.levels[1]["volume"], 9, 2 * nv, 2 * nv), dtype=torch.complex128,
                      device="cuda")
    gb.mg_build_coarse(mg.ctx, 0)
    gb.mg_device_status(mg.ctx)
    gb.mg_inject_fault(mg.ctx, "galerkin_mma_wait", 1)
    t0 = time.monotonic()
    gb.mg_build_coarse(mg.ctx, 0)
    with pytest.raises(gb.MGError) as e:
        gb.mg_device_status(mg.ctx)
    waited = time.monotonic() - t0
    assert e.value.status == gb.MG_ERR_TIMEOUT
    assert 0.9 < waited < 10.0, waited  # the budget is one second
    gb.mg_device_status(mg.ctx)  # the record was cleared
    gb.mg_build_coarse(mg.ctx, 0)
    gb.mg_get_coarse_links(mg.ctx, 1, out)
    gb.mg_device_status(mg.ctx)
    want = mgo.galerkin(oracle_fine(U, dims), mgo.block_orthonormalise(v, dims, block), block).blocks
    assert rel_l2(to_np(out), want) < 1e-5
    mg.close()
