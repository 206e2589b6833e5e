"""FP32 multi-RHS coarse apply with even counts: the launch of two rows per thread
is among the tuner's candidates wherever the block is small (n <= 48), and every
candidate gives the oracle's result, interleaved and back to back."""
import numpy as np
import pytest

import torch

import synthetic as syn
from oracle import dirac, lattice as lat
from gpu_helpers import make_ctx, rel_l2, to_dev, to_np

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("nrhs", [2, 4, 6, 8, 12, 24])
@pytest.mark.parametrize("nv", [8, 16, 24])
def test_two_row_launches(gpu_lib, nv, nrhs):
    """Rows of 9 n products summed in FP32: 1e-5 relative L2, the FP32 tier."""
    gb = gpu_lib
    cdims, n = (3, 2, 2, 4), 2 * nv
    vol = lat.volume(cdims)
    mg, _ = make_ctx(gb, cdims, [(1, 1, 1, 1)], [nv], prec_fine=1, prec_coarse=1)
    links = syn.gaussian_field((vol, 9, n, n), 67) / np.sqrt(n)
    gb.mg_set_coarse_links(mg.ctx, 1, to_dev(links))
    x = syn.gaussian_field((vol, n, nrhs), 68)
    cop = dirac.StencilOp(cdims, links)
    want = np.stack([cop.apply(x[:, :, k]) for k in range(nrhs)], axis=-1)
    xd = to_dev(x, torch.complex64)
    y = torch.empty_like(xd)
    key = f"stream_mr/p1/n{n}/v{vol}/r{nrhs}/b0"
    gb.mg_tune_set(key, -1)
    gb.mg_coarse_apply(mg.ctx, 1, y, xd, nrhs=nrhs)
    choices = [c for c, _ in gb.mg_tune_report(key)]
    assert (20 in choices) == (n <= 32 or nrhs % 8 != 0)
    for choice in choices:
        gb.mg_tune_set(key, choice)
        y.fill_(float("nan"))
        gb.mg_coarse_apply(mg.ctx, 1, y, xd, nrhs=nrhs)
        assert rel_l2(to_np(y), want) < 1e-5, choice
    gb.mg_tune_set(key, -1)
    mg.close()
