"""FP32 multi-RHS coarse applies on more sites than one grid dimension of 65535
holds (a 32^4 lattice in 2^4 aggregates has 16^4), odd and even counts."""
import pytest
import torch

from gpu_helpers import make_ctx

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("nrhs", [3, 2, 8])
def test_coarse_apply_beyond_65535_sites(gpu_lib, nrhs):
    """Rows of 9 n products of FP32 numbers summed in FP32: 1e-5 relative L2, the
    FP32 tier of the other applies."""
    gb = gpu_lib
    dims, n = (16, 16, 16, 17), 16
    vol = 16 * 16 * 16 * 17
    mg, _ = make_ctx(gb, dims, [(1, 1, 1, 1)], [n // 2], prec_fine=1, prec_coarse=1)
    gen = torch.Generator(device="cuda").manual_seed(5)
    links = torch.view_as_complex(torch.randn(vol, 9, n, n, 2, generator=gen, device="cuda",
                                              dtype=torch.float64)) / n ** 0.5
    gb.mg_set_coarse_links(mg.ctx, 1, links)
    x = torch.view_as_complex(torch.randn(vol, n, nrhs, 2, generator=gen, device="cuda",
                                          dtype=torch.float32))
    y = torch.full_like(x, float("nan"))
    gb.mg_coarse_apply(mg.ctx, 1, y, x, nrhs=nrhs)
    x64 = x.to(torch.complex128)
    idx = torch.arange(vol, device="cuda").view(dims[::-1])
    want = links[:, 0] @ x64
    for mu in range(4):
        want += links[:, 1 + 2 * mu] @ x64[torch.roll(idx, -1, 3 - mu).reshape(-1)]
        want += links[:, 2 + 2 * mu] @ x64[torch.roll(idx, 1, 3 - mu).reshape(-1)]
    err = torch.linalg.vector_norm(y - want) / torch.linalg.vector_norm(want)
    assert float(err) < 1e-5
    mg.close()
