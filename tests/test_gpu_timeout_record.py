"""A wait that gave up stays on record until mg_device_status reads it: the rank
test at the end of a null-vector setup, which uses a status word of its own,
must not wipe the time-out of the sweeps before it."""
import pytest
import torch

import synthetic as syn
from oracle import lattice as lat
from gpu_helpers import make_ctx, to_dev

pytestmark = pytest.mark.gpu


def test_timeout_in_a_setup_is_reported_after_it(gpu_lib):
    gb = gpu_lib
    dims, nv = (8, 4, 4, 4), 4
    mg, _ = make_ctx(gb, dims, [(4, 2, 2, 2)], [nv], prec_fine=1, prec_coarse=1, sweeps=2)
    init = to_dev(syn.gaussian_field((nv, lat.volume(dims), 12), 73))
    key = f"wilson/v{lat.volume(dims)}/n{nv}/c1"
    gb.mg_tune_set(key, 14)
    gb.mg_setup_nullvecs(mg.ctx, 0, init)
    gb.mg_device_status(mg.ctx)
    gb.mg_inject_fault(mg.ctx, "wilson_tile_wait", 1)
    try:
        gb.mg_setup_nullvecs(mg.ctx, 0, init)
    except gb.MGError:
        pass  # vectors swept with an operator that was not applied may be anything
    with pytest.raises(gb.MGError) as e:
        gb.mg_device_status(mg.ctx)
    assert e.value.status == gb.MG_ERR_TIMEOUT
    gb.mg_device_status(mg.ctx)  # the record was cleared
    gb.mg_setup_nullvecs(mg.ctx, 0, init)
    gb.mg_device_status(mg.ctx)
    out = torch.empty((nv, lat.volume(dims), 12), dtype=torch.complex128, device="cuda")
    gb.mg_get_nullvecs(mg.ctx, 0, out)
    assert bool(torch.isfinite(torch.view_as_real(out)).all())
    gb.mg_tune_set(key, -1)
    mg.close()
