"""Powers narrower than r + p columns (a capped last block, the literal form)
on the fused CUDA-core path, whose CTAs and so partials may then be twice as
many, in a workspace of exactly the queried size with guard bytes behind it,
against the float64 oracle."""
import numpy as np
import pytest
import torch

pytestmark = pytest.mark.gpu

GUARD = 8 << 20


@pytest.mark.parametrize("m,r,p,q,literal", [(135, 20, 16, 3, False), (129, 10, 23, 3, False), (137, 28, 20, 1, True),
                                             (120, 32, 16, 2, True)])
def test_narrow_powers_stay_in_their_partials(m, r, p, q, literal):
    import oracle
    import paper_2308_01480_gb300 as tt
    n = 40000 + m
    rng = np.random.default_rng(m)
    A = (rng.standard_normal((m, r)) / np.sqrt(m) * np.linspace(2.0, 1.0, r)) @ rng.standard_normal((r, n))
    A = (A / A.std() + 0.02 * rng.standard_normal((m, n))).astype(np.float32)
    opts = tt.options(paper_literal=literal)
    size = tt.workspace_size((m, n), (r,), p, q, opts)
    buf = torch.full((size + GUARD,), 0xA5, dtype=torch.uint8, device="cuda")
    cores, _ = tt.decompose(torch.from_numpy(A).cuda(), [r], p, q, omega_seed=3, opts=opts, workspace=buf[:size])
    torch.cuda.synchronize()
    assert bool((buf[size:] == 0xA5).all())
    assert tt.device_status(buf[:size]) == 0
    ref = (oracle.tt_rbki_literal if literal else oracle.tt_rbki)(A, [r], p, q, seed=3)
    # the repository's FP32 criterion
    assert oracle.tt_distance([c.cpu().double().numpy() for c in cores], ref) <= 1e-4
