"""The rank test of the block orthonormalisation compares the norm a column keeps
with 1e-12 of the block's Frobenius norm, which is summed as accurately as the
columns' own norms."""
import numpy as np
import pytest

from oracle import lattice as lat
from gpu_helpers import make_ctx, to_dev

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("rows_per_thread", [1, 2])
@pytest.mark.parametrize("share,deficient", [(1 - 1e-6, True), (1 + 1e-6, False)])
def test_rank_threshold(gpu_lib, rows_per_thread, share, deficient):
    """Column 0 is all ones, columns 1..46 have entries +-s (1 + i) with
    s^2 = 0.9 x 2^-24, so FP32 sums that begin with a 1 lose all of them:
    46 x 2 s^2 = 4.9e-6 of the squared norm, 2.5e-6 of the norm.  The last column
    is orthogonal to the others with 1e-12 (1 -+ 1e-6) of the norm."""
    gb = gpu_lib
    dims, nv = (4, 4, 2, 2 * rows_per_thread), 48
    block = (4, 4, 2, rows_per_thread)
    half, vol = 32 * rows_per_thread * 6, lat.volume(dims)
    rng = np.random.default_rng(3)
    s = np.sqrt(0.9 * 2.0 ** -24)
    sign = lambda *shape: 2.0 * rng.integers(0, 2, shape) - 1.0  # noqa: E731
    v = np.zeros((nv, vol, 12), dtype=np.complex128)
    site = np.arange(vol)
    for agg in range(2):
        mine = site[(site // 32) // rows_per_thread == agg]
        for chi in (0, 1):
            m = s * (sign(half, nv) + 1j * sign(half, nv))
            m[:, 0] = 1.0
            q, _ = np.linalg.qr(m[:, :-1])
            last = m[:, -1]
            for _ in range(3):
                last = last - q @ (q.conj().T @ last)
            norm = np.linalg.norm(m[:, :-1])
            m[:, -1] = last * (1e-12 * share * norm / np.linalg.norm(last))
            v[:, mine, 6 * chi:6 * chi + 6] = m.T.reshape(nv, half // 6, 6)
    mg, _ = make_ctx(gb, dims, [block], [nv], prec_fine=1, prec_coarse=1)
    if deficient:
        with pytest.raises(gb.MGError) as e:
            gb.mg_set_nullvecs(mg.ctx, 0, to_dev(v))
        assert e.value.status == gb.MG_ERR_RANK
    else:
        gb.mg_set_nullvecs(mg.ctx, 0, to_dev(v))
    mg.close()
