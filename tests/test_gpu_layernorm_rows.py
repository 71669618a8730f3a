"""Layer norm forward on both sides of the lines between its three ways through the rows (multiples of the rows that 148 SMs hold), with
row lengths that do not fill the last 32-chunk group and row counts that leave some warps a row less."""
import pytest
import torch

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("hidden,rows", [(8, 1), (264, 7945), (264, 7944), (1024, 2048), (1024, 2049), (1024, 9001), (1280, 1639),
                                         (1280, 13337), (2048, 1025), (2048, 5003), (512, 20011),
                                         (8, 3553), (200, 9473), (512, 2369), (640, 3552), (640, 3553), (768, 9473), (1024, 2369), (1024, 3553),
                                         (1000, 9473), (1280, 2369), (1536, 20011), (2048, 1185), (1800, 2369), (2048, 9473)])
def test_layernorm_rows(hidden, rows):
    from paper_2607_03229_b200 import binding as B

    gen = torch.Generator(device="cuda").manual_seed(hidden + rows)
    ld = hidden + 8   # rows apart in both matrices: what lies between them stays as it is
    x = (torch.randn(rows, ld, device="cuda", generator=gen) * 2 + 0.5).bfloat16()
    gamma = (1 + 0.1 * torch.randn(hidden, device="cuda", generator=gen)).bfloat16()
    beta = torch.randn(hidden, device="cuda", generator=gen).bfloat16()
    y = torch.full((rows, ld), -7.0, device="cuda", dtype=torch.bfloat16)
    B.layernorm_fwd(x[:, :hidden], gamma, beta, y[:, :hidden], 1e-6)
    ref = torch.nn.functional.layer_norm(x[:, :hidden].float(), (hidden,), gamma.float(), beta.float(), 1e-6)
    # one rounding to bf16 (2^-8 of the result at most, half of it to nearest) and fp32 sums of up to 2048 terms beside it
    assert ((y[:, :hidden].float() - ref).abs() <= ref.abs() * 2 ** -8 + 1e-4).all()
    assert (y[:, hidden:] == -7).all()
