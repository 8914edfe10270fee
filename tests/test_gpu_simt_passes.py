"""The CUDA-core streaming passes (FP32, and BF16 rows TMA cannot read) at the
edges of their launch rules: row tiles of 16/32/48/64, the 128- and 256-row
limits of the fused power, column tiles, widths b at each register-tile
boundary, rows split over the grid, and aligned against unaligned rows, all
against a float64 recomputation."""
import pytest
import torch

pytestmark = pytest.mark.gpu

SHAPES = [(m, n, b) for m, n in [(16, 600), (17, 601), (32, 515), (33, 1024), (48, 1023), (49, 300), (64, 4097),
                                 (65, 640), (128, 1300), (129, 2052), (256, 1301), (257, 700), (1100, 130),
                                 (2048, 61), (5000, 300)]
          for b in (4, 5, 13, 20, 21, 33)]
SHAPES += [(60, 5000, b) for b in (1, 6, 7, 8, 9, 12, 16, 17, 24, 25, 32, 40, 41, 48, 49, 64)]


def _check(got, ref, bound):
    # FP32 sums of up to 5,000 terms: the repository's 1e-5 of the largest
    # absolute-value bound
    assert float((got.double() - ref).abs().max()) <= 1e-5 * float(bound.max())


@pytest.mark.parametrize("m,n,b", SHAPES)
@pytest.mark.parametrize("dtype", ["float32", "bfloat16"])
def test_simt_passes(m, n, b, dtype):
    import paper_2308_01480_gb300 as tt
    if dtype == "bfloat16" and n % 8 == 0:
        n += 1
    g = torch.Generator(device="cuda")
    g.manual_seed(m * 7 + n + b)
    C = torch.randn(m, n, generator=g, device="cuda").to(getattr(torch, dtype))
    W = torch.randn(n, b, generator=g, device="cuda")
    X = torch.randn(m, b, generator=g, device="cuda")
    Cd, Wd, Xd = C.double(), W.double(), X.double()
    _check(tt.tt_pass(tt.TT_PASS_SKETCH, C, x=W), Cd @ Wd, Cd.abs() @ Wd.abs())
    P = tt.tt_pass(tt.TT_PASS_PROJECT, C, x=X)
    _check(P, Xd.T @ Cd, Xd.abs().T @ Cd.abs())
    assert torch.equal(tt.tt_pass(tt.TT_PASS_PROJECT, C, x=X, y_dtype=torch.bfloat16), P.bfloat16())
    Y = tt.tt_pass(tt.TT_PASS_GRAMAPPLY, C, x=X)
    _check(Y, Cd @ (Cd.T @ Xd), Cd.abs() @ (Cd.abs().T @ Xd.abs()))
    assert torch.equal(Y, tt.tt_pass(tt.TT_PASS_GRAMAPPLY, C, x=X))
    if b == 5 and m <= 2048:
        G = tt.tt_pass(tt.TT_PASS_GRAM, C)
        _check(G, Cd @ Cd.T, Cd.abs() @ Cd.abs().T)
        assert torch.equal(G, G.T)
