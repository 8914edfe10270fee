"""tt_permute_convert of sources whose fastest mode is not dense (every second
or third entry, in place and transposed), against torch's permute bit for
bit."""
import pytest
import torch

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("dims,step,perm", [((40, 66), 2, (0, 1)), ((40, 66), 2, (1, 0)), ((65, 130), 3, (1, 0)),
                                            ((7, 9, 64), 2, (2, 0, 1)), ((33, 5, 40), 2, (0, 2, 1)), ((3, 2000), 2, (1, 0)),
                                            ((300, 4), 2, (1, 0))])
@pytest.mark.parametrize("src", ["float32", "bfloat16"])
@pytest.mark.parametrize("dst", ["float32", "bfloat16"])
def test_strided_fastest_mode(dims, step, perm, src, dst):
    import paper_2308_01480_gb300 as tt
    g = torch.Generator(device="cuda")
    g.manual_seed(sum(dims))
    x = torch.randn(*dims, generator=g, device="cuda").to(getattr(torch, src))[..., ::step]
    out = tt.permute_convert(x, list(perm), getattr(torch, dst))
    assert torch.equal(out, x.permute(*perm).contiguous().to(getattr(torch, dst)))
