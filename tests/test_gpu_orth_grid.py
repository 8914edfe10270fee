"""The grid form of the block orthonormalisation at the edges of its launch
rules, in a workspace of exactly the queried size with guard bytes behind it,
against the float64 oracle."""
import numpy as np
import pytest
import torch

pytestmark = pytest.mark.gpu

GUARD = 8 << 20


def _check(dims, r, p, q):
    import oracle
    import paper_2308_01480_gb300 as tt
    rng = np.random.default_rng(sum(dims))
    F = [rng.standard_normal((n, r)) / np.sqrt(n) for n in dims]
    rest = F[-1].T
    for f in reversed(F[1:-1]):
        rest = (f.T[:, :, None] * rest[:, None, :]).reshape(r, -1)
    A = ((F[0] * np.linspace(2.0, 1.0, r)) @ rest).reshape(dims)
    A = (A / A.std() + 0.02 * rng.standard_normal(dims)).astype(np.float32)
    ranks = [r] * (len(dims) - 1)
    opts = tt.options()
    size = tt.workspace_size(dims, ranks, p, q, opts)
    buf = torch.full((size + GUARD,), 0xA5, dtype=torch.uint8, device="cuda")
    cores, _ = tt.decompose(torch.from_numpy(A).cuda(), ranks, p, q, omega_seed=3, opts=opts, workspace=buf[:size])
    torch.cuda.synchronize()
    assert bool((buf[size:] == 0xA5).all())
    assert tt.device_status(buf[:size]) == 0
    ref = oracle.tt_rbki(A, ranks, p, q, seed=3)
    # the repository's FP32 criterion
    assert oracle.tt_distance([c.cpu().double().numpy() for c in cores], ref) <= 1e-4


@pytest.mark.parametrize("dims,r,p,q", [((250, 250, 250), 45, 10, 2), ((9000, 300), 40, 10, 3), ((9000, 300), 56, 8, 1)])
def test_mixed_routes_stay_in_the_workspace(dims, r, p, q):
    """The first blocks take the grid form, the last does not."""
    _check(dims, r, p, q)


@pytest.mark.parametrize("m,r,p,q", [(22800, 20, 10, 4),    # 219,552 bytes of dynamic shared memory in the last block
                                     (44000, 10, 10, 4),    # 219,792
                                     (12000, 40, 10, 2),    # 220,784
                                     (43200, 9, 8, 5),      # 221,920
                                     (10300, 38, 10, 3)])   # 222,912: more than a CTA has beside the static arrays
def test_blocks_near_the_shared_memory_limit(m, r, p, q):
    """Layouts just inside and just outside what a CTA can have: either the
    grid form runs or another route does, none is refused at its launch."""
    _check((m, (r + p) * (q + 1) + 10), r, p, q)


@pytest.mark.parametrize("m,r,p,q", [(44394, 10, 8, 5), (40417, 11, 10, 4), (45946, 16, 10, 2)])
def test_blocks_in_the_tight_layout(m, r, p, q):
    """Layouts that leave no room to split Q^T Z over groups of threads."""
    _check((m, (r + p) * (q + 1) + 10), r, p, q)
