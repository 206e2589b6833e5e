"""Where the fine operator's plain launch and a tiled one are about as fast, the MR
steps take the tiled one (it forms their inner products): fewer launches per
setup sweep, the same vectors.  A pinned policy is taken as it is."""
import pytest
import torch

import synthetic as syn
from oracle import lattice as lat, multigrid as mgo
from gpu_helpers import make_ctx, oracle_fine, rel_l2, to_dev, to_np

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("pin", [None, 0])
def test_policy_of_the_sweeps(gpu_lib, pin):
    gb = gpu_lib
    dims, nv, sweeps = (8, 4, 4, 4), 2, 3
    vol = lat.volume(dims)
    key = f"wilson/v{vol}/n{nv}/c1"
    x0 = syn.gaussian_field((nv, vol, 12), 83)
    gb.mg_tune_set(key, -1 if pin is None else pin)
    mg, U = make_ctx(gb, dims, [(2, 2, 2, 2)], [nv], sweeps=sweeps, prec_fine=1, prec_coarse=1)
    for _ in range(2):  # (the first one tunes)
        before = gb.mg_launch_count(mg.ctx)
        gb.mg_setup_nullvecs(mg.ctx, 0, to_dev(x0))
        launches = gb.mg_launch_count(mg.ctx) - before
    raw = torch.empty((nv, vol, 12), dtype=torch.complex128, device="cuda")
    gb.mg_get_nullvecs(mg.ctx, 0, raw, kind=0)
    assert rel_l2(to_np(raw), mgo.null_vectors(oracle_fine(U, dims), x0, sweeps)) < 1e-5
    if pin is None:
        tiled = min((ms for c, ms in gb.mg_tune_report(key) if c >= 12), default=1e9)
        best = min(ms for _, ms in gb.mg_tune_report(key))
        fused = tiled <= best + 3e-3
    else:
        assert gb.mg_tune_get(key) == pin
        fused = False
    gb.mg_tune_set(key, 0)
    before = gb.mg_launch_count(mg.ctx)
    gb.mg_setup_nullvecs(mg.ctx, 0, to_dev(x0))
    separate = gb.mg_launch_count(mg.ctx) - before
    assert launches == separate - (sweeps if fused else 0)
    gb.mg_tune_set(key, -1)
    mg.close()
