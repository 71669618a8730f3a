"""What an image's tokens come out as does not depend on what they are packed with: a row of a projection or of its input gradient has
the same bits in a small and in a large matrix (whatever tile widths the two take), and an image through a layer stack the same bits
alone and in a microbatch."""
import numpy as np
import pytest
import torch

from paper_2607_03229_b200 import binding as B, dist as D, workloads as W
from _util import status_buf, to_dev

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("N,K", [(1024, 4096), (520, 2048), (192, 1024), (1288, 136)])
def test_rows_of_a_projection(N, K):
    big = 6000
    a, w = to_dev(W.normal_bf16(81, 0, (big, K))), to_dev(W.scaled_normal_bf16(81, 1, (N, K), std=K ** -0.5))
    b, u = to_dev(W.normal_bf16(81, 2, (N,))), to_dev(W.normal_bf16(81, 3, (big, N)))
    wt = w.t().contiguous()
    st = status_buf()
    for run in (lambda m, c: B.linear_fwd(a[:m], w, c, bias=b, residual=u[:m], status_buf=st),
                lambda m, c: B.linear_fwd(a[:m], w, c, bias=b, gelu=True, status_buf=st),
                lambda m, c: B.linear_dgrad(a[:m], wt, c, status_buf=st),
                lambda m, c: B.linear_dgrad(a[:m], wt, c, gelu_input=u[:m], status_buf=st)):
        ref = torch.empty((big, N), dtype=torch.bfloat16, device="cuda")
        run(big, ref)
        for m in (1, 86, 300, 777, 1024, 2100):
            c = torch.empty((m, N), dtype=torch.bfloat16, device="cuda")
            run(m, c)
            assert torch.equal(c, ref[:m]), m
    assert st.cpu().tolist()[0] == 0


@pytest.mark.parametrize("H,Dh,rope", [(16, 64, False), (4, 80, True)])
@pytest.mark.parametrize("mode", [B.FROZEN, B.TRAINED])
def test_an_image_alone_and_packed(H, Dh, rope, mode):
    hidden, n_layers = H * Dh, 2
    ffn = 4 * hidden
    counts = [777, 40, 300, 1500, 1, 900]
    shapes = {n: s(hidden, ffn) for n, s in D.LAYER_PARAM_SHAPES}
    layers = [B.LayerWeights.from_tensors(**{n: to_dev(W.scaled_normal_bf16(82, 20 * l + i, s, std=s[-1] ** -0.5 if len(s) > 1 else 0.1,
                                                                           mean=1.0 if n.endswith("gamma") else 0.0))
                                             for i, (n, s) in enumerate(shapes.items())}) for l in range(n_layers)]
    x = to_dev(W.normal_bf16(83, 0, (sum(counts), hidden)))

    def run(rows, cts):
        T = sum(cts)
        y, st = torch.empty((T, hidden), dtype=torch.bfloat16, device="cuda"), status_buf()
        ws = torch.empty(B.encoder_workspace_bytes(n_layers, T, hidden, ffn, mode), dtype=torch.uint8, device="cuda")
        lse = torch.empty((n_layers, H, T), device="cuda") if mode == B.TRAINED else None
        tabs = tuple(torch.from_numpy(t).cuda() for t in W.rope2d_tables(cts, Dh)) if rope else None
        B.encoder_fwd(rows, y, layers, H, ffn, B.seg_plan(cts, mode).to_device(), float(np.float32(Dh ** -0.5)), 1e-6, ws, lse, st, rope=tabs)
        torch.cuda.synchronize()
        assert st.cpu().tolist()[0] == 0
        return y

    packed, at = run(x, counts), 0
    for n in counts:
        assert torch.equal(run(x[at:at + n].contiguous(), [n]), packed[at:at + n]), n
        at += n
