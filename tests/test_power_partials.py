"""The workspace holds the fused CUDA-core power's partials at every width a
power runs at: a capped last block, and the r columns of the literal form, are
narrower than r + p and may have twice the CTAs."""
import pytest

import paper_2308_01480_gb300 as tt

# m, r, p, q, literal, columns of the narrower power, which is the one that
# needs most: 304 CTAs (two an SM) where r + p columns leave room for 152
CASES = [(135, 2, 34, 3, False, 27), (129, 2, 31, 3, False, 30), (133, 2, 34, 3, False, 25), (137, 28, 20, 1, True, 28),
         (120, 32, 16, 2, True, 32)]


@pytest.mark.parametrize("m,r,p,q,literal,c", CASES)
def test_workspace_holds_the_partials_of_narrower_powers(m, r, p, q, literal, c):
    n = 304 * (64 if m > 128 else 128)              # one column tile a CTA
    total = tt.workspace_size((m, n), (r,), p, q, tt.options(paper_literal=literal))
    # two remainders, the sketch matrix, the partials
    assert total >= 4 * (2 * r * n + (r + p) * n + 304 * m * c)
