"""The inner products that the tiled fine operator forms for the minimal-residual
steps, through whole setups against the oracle: every block shape, partial blocks
(whose surplus threads must add nothing), and, for one vector, more blocks than
the resident CTAs walk at once."""
import pytest
import torch

import synthetic as syn
from oracle import dirac, lattice as lat, multigrid as mgo
from gpu_helpers import make_ctx, rel_l2, to_dev, to_np

pytestmark = pytest.mark.gpu


def _setup(gb, dims, block, x0, sweeps, policy, U):
    nv, vol = x0.shape[0], lat.volume(dims)
    key = f"wilson/v{vol}/n{nv}/c1"
    gb.mg_tune_set(key, policy)
    mg, _ = make_ctx(gb, dims, [block], [nv], sweeps=sweeps, prec_fine=1, prec_coarse=1, U=U)
    gb.mg_setup_nullvecs(mg.ctx, 0, to_dev(x0))
    raw = torch.empty((nv, vol, 12), dtype=torch.complex128, device="cuda")
    gb.mg_get_nullvecs(mg.ctx, 0, raw, kind=0)
    gb.mg_device_status(mg.ctx)
    assert gb.mg_tune_get(key) == policy
    gb.mg_tune_set(key, -1)
    mg.close()
    return to_np(raw)


@pytest.mark.parametrize("dims,block", [((10, 6, 6, 6), (2, 2, 2, 2)), ((8, 4, 4, 2), (2, 2, 2, 1))])
@pytest.mark.parametrize("nv", [1, 3])
@pytest.mark.parametrize("policy", [12, 13, 14, 15])
def test_setup_on_partial_blocks(gpu_lib, policy, nv, dims, block):
    """Three sweeps in FP32 against FP64: the FP32 tier 1e-5."""
    U = syn.gauge_field(dims, 0.3, 1)
    x0 = syn.gaussian_field((nv, lat.volume(dims), 12), 81)
    raw = _setup(gpu_lib, dims, block, x0, 3, policy, U)
    op = dirac.wilson_clover_op(U, dims, -0.2, 1.0, True)
    assert rel_l2(raw, mgo.null_vectors(op, x0, 3)) < 1e-5


@pytest.fixture(scope="module")
def large():
    dims = (18, 16, 16, 32)
    U = syn.gauge_field(dims, 0.3, 1)
    x0 = syn.gaussian_field((1, lat.volume(dims), 12), 82)
    return dims, U, x0, mgo.null_vectors(dirac.wilson_clover_op(U, dims, -0.2, 1.0, True), x0, 1)


@pytest.mark.parametrize("policy", [12, 13, 14, 15])
def test_one_vector_on_more_blocks_than_resident_ctas(gpu_lib, large, policy):
    """1152 to 3072 blocks, against at most 152 x 7 resident CTAs of 64 threads and
    152 x 3 of 128; partial blocks in x.  One sweep, the FP32 tier."""
    dims, U, x0, want = large
    raw = _setup(gpu_lib, dims, (2, 2, 2, 2), x0, 1, policy, U)
    assert rel_l2(raw, want) < 1e-5
