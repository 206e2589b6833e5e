"""Tensor-core Galerkin build with null vectors that are small where a face block
gets its entries: every output block must be as accurate relative to itself as
FP32 arithmetic makes it, whatever the size of the vectors there."""
import numpy as np
import pytest
import torch

import synthetic as syn
from oracle import lattice as lat, multigrid as mgo
from gpu_helpers import make_ctx, oracle_fine, to_dev, to_np

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("nv", [16, 24])
@pytest.mark.parametrize("mass", [-0.2, 1e5])
@pytest.mark.parametrize("size", [1e-3, 1e-6, 1e-9])
def test_blocks_of_small_entries(gpu_lib, nv, mass, size):
    """4^4 aggregates, sites at their faces `size` of the inner ones.  A face block
    sums products of two small numbers: P rounded to FP32 (2^-24 at most, twice),
    a chain of about 10 FP32 operations per entry of T (rms sqrt(10) 2^-24 /
    sqrt 3, 1.9 x 2^-24), at most six truncating accumulations in a unit (mean half
    a unit in the last place, 3 x 2^-24): under 6 x 2^-24 of the block's own norm;
    the diagonal block, whose chains are twice as long, likewise (its sums, of
    one sign, are judged on Gaussian vectors elsewhere)."""
    gb = gpu_lib
    dims, block = (8, 4, 4, 8), (4, 4, 4, 4)
    vol = lat.volume(dims)
    mg, U = make_ctx(gb, dims, [block], [nv], prec_fine=1, prec_coarse=1, mass=mass, eps=0.5)
    s = np.arange(vol)
    local = [s % 8 % 4, s // 8 % 4, s // 32 % 4, s // 128 % 4]
    inner = np.all([(c > 0) & (c < 3) for c in local], axis=0)
    v = syn.gaussian_field((nv, vol, 12), 37) * np.where(inner, 1.0, size)[None, :, None]
    gb.mg_set_nullvecs(mg.ctx, 0, to_dev(v))
    gb.mg_build_coarse(mg.ctx, 0)
    out = torch.empty((mg.levels[1]["volume"], 9, 2 * nv, 2 * nv), dtype=torch.complex128,
                      device="cuda")
    gb.mg_get_coarse_links(mg.ctx, 1, out)
    gb.mg_device_status(mg.ctx)
    want = mgo.galerkin(oracle_fine(U, dims, mass=mass), mgo.block_orthonormalise(v, dims, block),
                        block).blocks
    err = np.linalg.norm(to_np(out) - want, axis=(2, 3)) / np.linalg.norm(want, axis=(2, 3))
    assert err.max() < 6 * 2.0 ** -24, (err.max(axis=0) * 2.0 ** 24).round(2)
    mg.close()
