"""The small A^T B of Rayleigh-Ritz and of the column-Gram route at the edges
of its launch rule (chunks of 32 rows, groups of 256 rows, the 512-row limit
of the one-launch form; 32-column tiles), as order-2 decompositions against
the float64 oracle."""
import numpy as np
import pytest
import torch

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("m", [31, 32, 33, 255, 257, 512, 513, 1024])
@pytest.mark.parametrize("n,r,p,q", [(150, 5, 6, 2),      # basis of 33 columns
                                     (12, 4, 5, 1)])      # column-Gram route (n < m)
def test_small_products_match_oracle(m, n, r, p, q):
    import oracle
    import paper_2308_01480_gb300 as tt
    rng = np.random.default_rng(m + n)
    A = (rng.standard_normal((m, r)) * np.linspace(2.0, 1.0, r)) @ rng.standard_normal((r, n))
    A = (A + 0.02 * rng.standard_normal((m, n))).astype(np.float32)
    cores, _ = tt.decompose(torch.from_numpy(A).cuda(), [r], p, q, omega_seed=3)
    ref = oracle.tt_rbki(A, [r], p, q, seed=3)
    # the repository's FP32 criterion
    assert oracle.tt_distance([c.cpu().double().numpy() for c in cores], ref) <= 1e-4
