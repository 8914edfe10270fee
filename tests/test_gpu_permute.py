"""tt_permute_convert over its kernels (rows, tiles, generic): tile edges,
short and odd modes, strided, broadcast and misaligned sources, against
torch's permute bit for bit."""
import pytest

pytestmark = pytest.mark.gpu

CASES = [
    # dims, perm, source slicing: None dense, "pad" strided rows, "off" base one element in, "bc" a broadcast mode
    ((64, 33), (1, 0), None), ((31, 65), (1, 0), None), ((8, 8), (1, 0), None), ((7, 300), (1, 0), None),
    ((32, 64, 5), (1, 0, 2), None), ((3, 129, 66), (2, 0, 1), None), ((17, 9, 11, 13), (3, 1, 0, 2), None),
    ((256, 32, 64, 32), (3, 1, 0, 2), None), ((5, 1, 40, 1, 36), (4, 2, 0, 1, 3), None),
    ((40, 40, 40), (0, 1, 2), None), ((40, 41), (0, 1), "pad"), ((40, 44), (0, 1), "pad"), ((64, 70), (1, 0), "pad"),
    ((63, 4, 16), (1, 0, 2), None), ((63, 4, 18), (1, 0, 2), None), ((50, 34), (1, 0), "off"), ((50, 36), (0, 1), "off"),
    ((12, 33, 20), (2, 0, 1), "bc"), ((33, 20), (0, 1), "bc"), ((1,), (0,), None), ((1030,), (0,), None),
    ((2, 3, 2, 3, 2, 3, 2, 5), (7, 0, 6, 1, 5, 2, 4, 3), None), ((1000, 1100), (1, 0), None),
]


@pytest.mark.parametrize("dims,perm,how", CASES)
@pytest.mark.parametrize("src,dst", [("float32", "bfloat16"), ("bfloat16", "float32"), ("float32", "float32"),
                                     ("bfloat16", "bfloat16")])
def test_permute_routes_bit_exact(dims, perm, how, src, dst):
    import torch
    import paper_2308_01480_gb300 as tt
    ts, td = getattr(torch, src), getattr(torch, dst)
    torch.manual_seed(3)
    if how == "pad":
        x = torch.randn(*dims[:-1], dims[-1] + 3, device="cuda").to(ts)[..., :dims[-1]]
    elif how == "off":
        n = 1
        for d in dims:
            n *= d
        x = torch.randn(n + 1, device="cuda").to(ts)[1:].view(*dims)
    elif how == "bc":
        x = torch.randn(dims[0], *([1] * (len(dims) - 1)), device="cuda").to(ts).expand(*dims)
    else:
        x = torch.randn(*dims, device="cuda").to(ts)
    out = tt.permute_convert(x, list(perm), td)
    ref = x.permute(*perm).contiguous().to(td)
    assert torch.equal(out, ref)
