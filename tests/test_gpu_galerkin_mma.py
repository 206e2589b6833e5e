"""Galerkin product of the FP32 Wilson-clover level with the contractions on
the tensor cores (16 and 24 null vectors) against the FP64 oracle: every
block of Eq. (3), aggregates whose site and face counts are not multiples of
the chunk of eight sites, coarse extents of one (the hop wraps onto the
aggregate's own lattice edge), more output blocks than SMs.  The FP32 tier
1e-5 relative L2; each output block separately within 1e-5 of the largest."""
import numpy as np
import pytest
import torch

import synthetic as syn
from oracle import lattice as lat, multigrid as mgo
from gpu_helpers import make_ctx, oracle_fine, rel_l2, to_dev, to_np

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("dims,block,nv", [
    ((4, 4, 4, 4), (2, 2, 2, 2), 16),
    ((4, 4, 4, 8), (4, 2, 2, 2), 24),
    ((6, 4, 4, 4), (3, 2, 2, 4), 24),     # 48 sites, faces of 16, 24 and 12
    ((6, 2, 4, 6), (3, 1, 2, 3), 16),     # 18 sites, faces of 6, 9 and 18
    ((4, 4, 4, 4), (4, 4, 4, 4), 24),     # one aggregate: every hop wraps
    ((8, 8, 4, 4), (2, 2, 2, 2), 24),     # 288 output blocks
])
@pytest.mark.parametrize("antiperiodic", [1, 0])
def test_galerkin_tensor_cores(gpu_lib, dims, block, nv, antiperiodic):
    gb = gpu_lib
    mg, U = make_ctx(gb, dims, [block], [nv], prec_fine=1, prec_coarse=1, eps=0.5,
                     antiperiodic=antiperiodic)
    v = syn.gaussian_field((nv, lat.volume(dims), 12), 31)
    gb.mg_set_nullvecs(mg.ctx, 0, to_dev(v))
    gb.mg_build_coarse(mg.ctx, 0)
    n, cvol = 2 * nv, mg.levels[1]["volume"]
    out = torch.full((cvol, 9, n, n), float("nan"), dtype=torch.complex128, device="cuda")
    gb.mg_get_coarse_links(mg.ctx, 1, out)
    gb.mg_device_status(mg.ctx)
    op = oracle_fine(U, dims, antiperiodic=bool(antiperiodic))
    want = mgo.galerkin(op, mgo.block_orthonormalise(v, dims, block), block).blocks
    got = to_np(out)
    assert rel_l2(got, want) < 1e-5, rel_l2(got, want)
    big = max(np.linalg.norm(want[:, s]) for s in range(9))
    for s in range(9):
        assert np.linalg.norm(got[:, s] - want[:, s]) < 1e-5 * big, s
    mg.close()


@pytest.mark.parametrize("dims,block", [
    ((4, 4, 4, 4), (2, 2, 2, 2)),     # 16 sites: two units of a chunk
    ((4, 4, 4, 8), (2, 2, 2, 4)),     # 32 sites: four units of a chunk
    ((4, 4, 4, 8), (2, 4, 2, 4)),     # 64 sites: four units of two chunks
    ((4, 4, 4, 8), (4, 4, 4, 4)),     # 256 sites: 16 units of two chunks
])
def test_galerkin_tensor_cores_accuracy(gpu_lib, dims, block):
    """FP32 accuracy whatever the aggregate: P rounded to FP32 (2^-24 at most),
    T a chain of about 20 FP32 operations (rms sqrt(20) 2^-24 / sqrt 3, 2.6
    x 2^-24), the split operands (2^-23 at most each, dropped term included)
    and at most six truncating accumulations in a unit (mean half a unit in
    the last place, 3 x 2^-24): together under 6 x 2^-24 relative L2.  Units
    of four chunks give 11 x 2^-24."""
    gb = gpu_lib
    nv = 24
    mg, U = make_ctx(gb, dims, [block], [nv], prec_fine=1, prec_coarse=1, eps=0.5)
    v = syn.gaussian_field((nv, lat.volume(dims), 12), 31)
    gb.mg_set_nullvecs(mg.ctx, 0, to_dev(v))
    gb.mg_build_coarse(mg.ctx, 0)
    out = torch.empty((mg.levels[1]["volume"], 9, 2 * nv, 2 * nv), dtype=torch.complex128,
                      device="cuda")
    gb.mg_get_coarse_links(mg.ctx, 1, out)
    gb.mg_device_status(mg.ctx)
    want = mgo.galerkin(oracle_fine(U, dims), mgo.block_orthonormalise(v, dims, block), block).blocks
    assert rel_l2(to_np(out), want) < 6 * 2.0 ** -24
    mg.close()
