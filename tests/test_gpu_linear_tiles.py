"""The projection kernel at the sizes where its tile width and its ragged edges change, against the fp64 oracle: every width (64, 128,
192, 256), rows on both sides of a 256-row tile, and the epilogues that carry two operands at once."""
import numpy as np
import pytest
import torch

from oracle import layer as OL
from paper_2607_03229_b200 import binding as B, workloads as W
from _util import to_dev, to_f64, status_buf

pytestmark = pytest.mark.gpu

# One bf16 rounding of an fp32-accumulated result: 2^-9 relative, doubled; the absolute part covers the fp32 accumulation of
# K <= 4096 products of O(1) / sqrt(K) weights and the 1.5e-7 of the GELU's erf.
REL, ABS = 2.0 ** -8, 2e-3


def _close(got, ref):
    err = np.abs(got - ref)
    assert (err <= ABS + REL * np.abs(ref)).all(), float((err - REL * np.abs(ref)).max())


@pytest.mark.parametrize("M,N,K", [(86, 960, 320),      # width 64
                                   (255, 1032, 72), (257, 1032, 72),   # one 256-row tile and two
                                   (777, 3072, 1024),   # width 192
                                   (777, 4096, 1024),   # width 256
                                   (300, 520, 2048),    # two tiles of rows, ragged last chunk
                                   (777, 1024, 4096),   # four row tiles, a long contraction
                                   (90, 320, 192), (90, 320, 200),   # two blocks of the contraction per stage, an odd number of them; whole atoms or not
                                   (4000, 1288, 136)])  # several tiles per pair
def test_linear_and_dgrad_tile_choices(M, N, K):
    a, w = W.normal_bf16(51, 0, (M, K)), W.scaled_normal_bf16(51, 1, (N, K), std=K ** -0.5)
    b, r, u = W.scaled_normal_bf16(51, 2, (N,), std=0.5), W.normal_bf16(51, 3, (M, N)), W.normal_bf16(51, 4, (M, N))
    wt = np.ascontiguousarray(w.T)                       # the same product through the input-gradient entry point
    ad, wd, bd, rd, ud, wtd = (to_dev(x) for x in (a, w, b, r, u, wt))
    lin = OL.linear(OL.widen(a), OL.widen(w), None)
    lin_b = lin + OL.widen(b)
    st = status_buf()
    out = torch.full((M + 1, N + 8), 7.0, dtype=torch.bfloat16, device="cuda")
    for kw, ref in (({}, lin), ({"bias": bd, "gelu": True}, OL.gelu(lin_b)),
                    ({"bias": bd, "residual": rd, "gelu": True}, OL.gelu(lin_b) + OL.widen(r))):
        B.linear_fwd(ad, wd, out[:M, :N], status_buf=st, **kw)
        _close(to_f64(out[:M, :N]), ref)
    for kw, ref in (({}, lin), ({"gelu_input": ud, "residual": rd}, lin * OL.gelu_grad(OL.widen(u)) + OL.widen(r))):
        B.linear_dgrad(ad, wtd, out[:M, :N], status_buf=st, **kw)
        _close(to_f64(out[:M, :N]), ref)
    assert (out[M:] == 7.0).all() and (out[:, N:] == 7.0).all() and st.cpu().tolist()[0] == 0


@pytest.mark.parametrize("T,N,K", [(64, 264, 72),       # one block of tokens: nothing to split
                                   (300, 1536, 512),    # width 128, split in two
                                   (700, 1288, 1032),   # ragged tiles of both widths
                                   (3489, 1024, 1024),  # split token range
                                   (2000, 520, 2560)])
def test_wgrad_tile_choices(T, N, K):
    dy, x = W.normal_bf16(52, 0, (T, N)), W.normal_bf16(52, 1, (T, K))
    dw = torch.full((N + 1, K + 4), 0.5, dtype=torch.float32, device="cuda")
    st = status_buf()
    B.linear_wgrad(to_dev(dy), to_dev(x), dw[:N, :K], st)
    ref, _ = OL.linear_wgrad(OL.widen(dy), OL.widen(x))
    got = dw.cpu().double().numpy()
    # fp32 accumulation of T exact bf16 products per element
    assert np.abs(got[:N, :K] - 0.5 - ref).max() <= 1e-5 * max(1.0, np.abs(ref).max()) + 4e-7 * T ** 0.5 * 16
    assert (got[N:] == 0.5).all() and (got[:, K:] == 0.5).all() and st.cpu().tolist()[0] == 0
