"""The one-launch A^T B of Rayleigh-Ritz over grids of more than two 32-column
tiles a side (bases of 65 to 150 columns, up to 512 rows), and of the
column-Gram route over up to 128 columns, as order-2 decompositions against
the float64 oracle."""
import numpy as np
import pytest
import torch

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("m,n,r,p,q", [(300, 9000, 5, 8, 4), (511, 9000, 10, 15, 4), (512, 9000, 10, 20, 4),
                                       (200, 9000, 10, 20, 4), (512, 96, 20, 20, 2), (300, 128, 24, 20, 2)])
def test_wide_small_products_match_oracle(m, n, r, p, q):
    import oracle
    import paper_2308_01480_gb300 as tt
    rng = np.random.default_rng(m + n)
    A = (rng.standard_normal((m, r)) * np.linspace(2.0, 1.0, r)) @ rng.standard_normal((r, n))
    A = (A + 0.02 * rng.standard_normal((m, n))).astype(np.float32)
    cores, _ = tt.decompose(torch.from_numpy(A).cuda(), [r], p, q, omega_seed=3)
    ref = oracle.tt_rbki(A, [r], p, q, seed=3)
    # the repository's FP32 criterion
    assert oracle.tt_distance([c.cpu().double().numpy() for c in cores], ref) <= 1e-4
