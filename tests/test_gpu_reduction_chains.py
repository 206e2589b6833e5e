"""FP32 partial sums of the batched reductions stay short however many vectors
share the grid: the squared norms of a setup's vectors, which the normalisation
divides by."""
import pytest
import torch

import synthetic as syn
from oracle import lattice as lat
from gpu_helpers import make_ctx

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("nv", [8, 48])
def test_batched_norms_do_not_lose_small_terms(gpu_lib, nv):
    """The first 2^14 entries of every vector are +-1, all others +-s (1 + i) with
    s^2 = 0.9 x 2^-24, under half a unit in the last place of 1: an FP32 sum that
    began with a 1 never sees another entry.  Sums of at most four rounds lose
    three entries, 3 x 2 s^2 = 5.4 x 2^-24 of the squared norm; the rounded
    inverse norm adds 2 x 2^-24 (products with 1 are exact).  Sums as long as a
    thread's share of the vector lose 128 entries' worth with 48 vectors."""
    gb = gpu_lib
    dims = (16, 16, 16, 32)
    vol = lat.volume(dims)
    gen = torch.Generator(device="cuda").manual_seed(11)

    def sign(*shape):
        return 2.0 * torch.randint(0, 2, shape, generator=gen, device="cuda",
                                   dtype=torch.float64) - 1.0

    s = (0.9 * 2.0 ** -24) ** 0.5
    v = torch.complex(s * sign(nv, vol * 12), s * sign(nv, vol * 12))
    v[:, :1 << 14] = sign(nv, 1 << 14).to(torch.complex128)
    mg, _ = make_ctx(gb, dims, [(4, 4, 4, 4)], [nv], prec_fine=1, prec_coarse=1, sweeps=0,
                     U=syn.gauge_field(dims, 0.3, 1))
    gb.mg_setup_nullvecs(mg.ctx, 0, v.view(nv, vol, 12))
    raw = torch.empty((nv, vol, 12), dtype=torch.complex128, device="cuda")
    gb.mg_get_nullvecs(mg.ctx, 0, raw, 0)
    norms = (raw.real ** 2 + raw.imag ** 2).sum((1, 2))
    assert float((norms - 1).abs().max()) < 8 * 2.0 ** -24
    mg.close()
