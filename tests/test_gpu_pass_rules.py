"""The CUDA-core passes on both sides of their launch rules: the projection's
64-column form (rows 16 to 256, 19,456 columns, widths 12/13, 20/21, 24/25,
48/49; 160 rows), its row groups and 24-column tiles of unaligned rows, the
fused power's short tiles (2,048 columns; 128 rows, 9,728 columns and 12
widths), the Gram's tile edge and splits; against a float64 recomputation."""
import pytest
import torch

pytestmark = pytest.mark.gpu

PROJ = [(m, n, b) for m in (1, 17, 64, 65, 160, 161, 256) for n in (1, 63, 65, 1001, 2052) for b in (12, 13, 21, 25, 49)]
PROJ += [(60, n, b) for n in (19455, 19456, 19457) for b in (5, 13, 20, 21, 24, 25, 48, 49, 64)]
PROJ += [(m, 4001, b) for m in (48, 49, 300) for b in (10, 41, 45, 48, 60)] + [(257, 900, 60), (50, 40003, 45), (90, 30000, 30)]
POWER = [(m, n, b) for m in (1, 20, 33, 64, 65, 128, 129, 256) for n in (1, 31, 33, 2048, 2049) for b in (4, 7, 12, 13, 33)]
POWER += [(m, n, b) for m in (129, 200) for n in (9727, 9728, 9729) for b in (12, 13, 48)]
GRAM = [(m, n) for m in (1, 16, 17, 32, 33, 64, 100, 240, 400) for n in (1, 64, 65, 700, 2001)] + [(800, 1601), (1000, 300), (39, 20011)]


def _case(m, n, b, dtype):
    g = torch.Generator(device="cuda")
    g.manual_seed(m * 7 + n + b)
    C = torch.randn(m, n, generator=g, device="cuda").to(getattr(torch, dtype))
    return C, torch.randn(m, b, generator=g, device="cuda")


def _check(got, ref, bound):
    # FP32 sums: the repository's 1e-5 of the largest absolute-value bound
    assert float((got.double() - ref).abs().max()) <= 1e-5 * float(bound.max())


@pytest.mark.parametrize("dtype", ["float32", "bfloat16"])
def test_projection_rules(dtype):
    import paper_2308_01480_gb300 as tt
    for m, n, b in PROJ:
        n += 1 if dtype == "bfloat16" and n % 8 == 0 else 0
        C, X = _case(m, n, b, dtype)
        P = tt.tt_pass(tt.TT_PASS_PROJECT, C, x=X)
        _check(P, X.double().T @ C.double(), X.double().abs().T @ C.double().abs())
        assert torch.equal(tt.tt_pass(tt.TT_PASS_PROJECT, C, x=X, y_dtype=torch.bfloat16), P.bfloat16())


@pytest.mark.parametrize("dtype", ["float32", "bfloat16"])
def test_power_rules(dtype):
    import paper_2308_01480_gb300 as tt
    for m, n, b in POWER:
        n += 1 if dtype == "bfloat16" and n % 8 == 0 else 0
        C, X = _case(m, n, b, dtype)
        Cd, Xd = C.double(), X.double()
        _check(tt.tt_pass(tt.TT_PASS_GRAMAPPLY, C, x=X), Cd @ (Cd.T @ Xd), Cd.abs() @ (Cd.abs().T @ Xd.abs()))


@pytest.mark.parametrize("dtype", ["float32", "bfloat16"])
def test_gram_rules(dtype):
    import paper_2308_01480_gb300 as tt
    for m, n in GRAM:
        n += 1 if dtype == "bfloat16" and n % 8 == 0 else 0
        C, _ = _case(m, n, 1, dtype)
        G = tt.tt_pass(tt.TT_PASS_GRAM, C)
        _check(G, C.double() @ C.double().T, C.double().abs() @ C.double().abs().T)
        assert torch.equal(G, G.T)
