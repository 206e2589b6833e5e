"""Tensor-core Galerkin build with as many coarse sites as make the CTAs' shares of
diagonal blocks uneven (the face blocks are then dealt out to even them): every
output block against the FP64 build of the same operator and vectors."""
import pytest
import torch

import synthetic as syn
from oracle import lattice as lat
from gpu_helpers import make_ctx, to_dev

pytestmark = pytest.mark.gpu


def _build(gb, dims, block, nv, U, v, prec):
    mg, _ = make_ctx(gb, dims, [block], [nv], prec_fine=prec, prec_coarse=prec, eps=0.5, U=U)
    gb.mg_set_nullvecs(mg.ctx, 0, v)
    cvol = mg.levels[1]["volume"]
    # (stale links of an earlier build would hide a block that is not written)
    gb.mg_set_coarse_links(mg.ctx, 1, torch.full((cvol, 9, 2 * nv, 2 * nv), 7.0,
                                                 dtype=torch.complex128, device="cuda"))
    gb.mg_build_coarse(mg.ctx, 0)
    out = torch.empty((cvol, 9, 2 * nv, 2 * nv), dtype=torch.complex128, device="cuda")
    gb.mg_get_coarse_links(mg.ctx, 1, out)
    gb.mg_device_status(mg.ctx)
    mg.close()
    return out


@pytest.mark.parametrize("dims,block", [
    ((4, 8, 8, 32), (4, 4, 4, 4)),       # 32 coarse sites: fewer blocks than two rounds
    ((12, 12, 12, 16), (4, 4, 4, 4)),    # 108: some CTAs without a diagonal block
    ((12, 12, 12, 28), (4, 4, 4, 4)),    # 189: some with two
    ((8, 8, 16, 38), (4, 4, 4, 2)),      # 304: two full rounds on 152 SMs
])
@pytest.mark.parametrize("nv", [16, 24])
def test_every_block_is_built(gpu_lib, dims, block, nv):
    """1e-5 of the block's own norm, the FP32 tier (FP64 against FP64-rounded-to-FP32
    arithmetic, Gaussian vectors)."""
    gb = gpu_lib
    U = syn.gauge_field(dims, 0.5, 1)
    v = to_dev(syn.gaussian_field((nv, lat.volume(dims), 12), 39))
    got = _build(gb, dims, block, nv, U, v, 1)
    want = _build(gb, dims, block, nv, U, v, 0)
    err = torch.linalg.vector_norm(got - want, dim=(2, 3))
    assert bool((err < 1e-5 * torch.linalg.vector_norm(want, dim=(2, 3))).all())
