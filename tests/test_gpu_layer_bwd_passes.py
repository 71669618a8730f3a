"""The passes of the layer backward at the sizes where they branch: LayerNorm backward for every number of 16-byte chunks per lane
and for fewer rows than warps, and the bias gradients that the weight-gradient kernel adds up on its way (ragged tokens, output
columns that do not fill a tile, a token range shorter than one block)."""
import numpy as np
import pytest
import torch

from oracle import layer as OL
from paper_2607_03229_b200 import binding as B, workloads as W
from _util import rel_l2, status_buf, to_dev, to_f64

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("T,hidden", [(3, 264), (1300, 520), (5, 768), (700, 1032), (1200, 1288), (600, 1536), (601, 1800)])
def test_layernorm_bwd_chunk_counts(T, hidden):
    x = W.scaled_normal_bf16(61, 0, (T, hidden), std=2.0, mean=0.7)
    dy, g, r = W.normal_bf16(61, 1, (T, hidden)), W.scaled_normal_bf16(61, 2, (hidden,), std=0.1, mean=1.0), W.normal_bf16(61, 3, (T, hidden))
    pad = 8
    dx = torch.full((T, hidden + pad), 7.0, dtype=torch.bfloat16, device="cuda")
    dg, db = torch.full((hidden,), 0.25, device="cuda"), torch.full((hidden,), -0.5, device="cuda")
    B.layernorm_bwd(to_dev(x), to_dev(dy), to_dev(g), dx[:, :hidden], dg, db, 1e-6, to_dev(r))
    dx_ref, dg_ref, db_ref = OL.layernorm_bwd(OL.widen(x), OL.widen(dy), OL.widen(g), 1e-6)
    dx_ref = dx_ref + OL.widen(r)
    # one bf16 rounding of the result (2^-9, doubled) and fp32 row sums; fp32 column sums of T terms
    assert (np.abs(to_f64(dx[:, :hidden]) - dx_ref) <= 2e-4 + 2.0 ** -8 * np.abs(dx_ref)).all() and (dx[:, hidden:] == 7.0).all()
    tol = 1e-5 * max(1.0, np.abs(dg_ref).max()) + 2e-6 * T ** 0.5 * 8
    assert np.abs(dg.cpu().double().numpy() - 0.25 - dg_ref).max() <= tol
    assert np.abs(db.cpu().double().numpy() + 0.5 - db_ref).max() <= tol


@pytest.mark.parametrize("counts,H,D,ffn,rope", [([20], 1, 64, 72, False), ([70, 3], 3, 80, 264, True), ([600, 900], 5, 64, 1288, True)])
def test_layer_bwd_bias_gradients(counts, H, D, ffn, rope):
    hidden, T = H * D, sum(counts)
    pb = W.layer_params_bf16(62, hidden, ffn)
    x, dy = to_dev(W.normal_bf16(62, 0, (T, hidden))), to_dev(W.normal_bf16(62, 1, (T, hidden)))
    plan = B.seg_plan(counts, B.TRAINED).to_device()
    weights = B.LayerWeights.from_tensors(**{k: to_dev(v) for k, v in pb.items()})
    grads = {k: torch.full(v.shape, 0.5, device="cuda") for k, v in pb.items()}
    y, dx = torch.empty_like(x), torch.empty_like(x)
    lse = torch.empty((H, T), device="cuda")
    ws_f = torch.zeros(B.encoder_layer_workspace_bytes(T, hidden, ffn), dtype=torch.uint8, device="cuda")
    ws_b = torch.empty(B.encoder_layer_bwd_workspace_bytes(T, hidden, H, ffn), dtype=torch.uint8, device="cuda")
    st = status_buf()
    scale = float(np.float32(D ** -0.5))
    tabs = W.rope2d_tables(counts, D) if rope else None
    dev_tabs = None if tabs is None else tuple(torch.from_numpy(t).cuda() for t in tabs)
    B.encoder_layer_fwd(x, y, weights, H, ffn, plan, scale, 1e-6, ws_f, lse, st, rope=dev_tabs)
    kept = ws_f.clone()
    B.encoder_layer_bwd(dy, x, dx, weights, B.LayerGrads.from_tensors(**grads), H, ffn, plan, scale, 1e-6, lse, ws_f, ws_b, st, rope=dev_tabs)
    torch.cuda.synchronize()
    assert st.cpu().tolist()[0] == 0 and torch.equal(kept, ws_f)       # what the forward left is only read
    ow = OL.LayerWeights(g1=OL.widen(pb["ln1_gamma"]), b1=OL.widen(pb["ln1_beta"]), wqkv=OL.widen(pb["w_qkv"]), bqkv=OL.widen(pb["b_qkv"]),
                         wo=OL.widen(pb["w_o"]), bo=OL.widen(pb["b_o"]), g2=OL.widen(pb["ln2_gamma"]), b2=OL.widen(pb["ln2_beta"]),
                         w1=OL.widen(pb["w_fc1"]), bb1=OL.widen(pb["b_fc1"]), w2=OL.widen(pb["w_fc2"]), bb2=OL.widen(pb["b_fc2"]))
    cu = np.concatenate([[0], np.cumsum(counts)]).astype(np.int32)
    dx_ref, ref = OL.encoder_layer_bwd(W.normal_bf16(62, 0, (T, hidden)), ow, cu, H, scale, 1e-6, W.normal_bf16(62, 1, (T, hidden)),
                                       None if tabs is None else tuple(t.astype(np.float64) for t in tabs))
    # about ten bf16-rounded stages of 2^-9 each in a row, as for the whole layer
    assert rel_l2(to_f64(dx), dx_ref) <= 1.5e-2
    for name in grads:
        got = grads[name].cpu().double().numpy() - 0.5
        assert rel_l2(got, ref[name].reshape(got.shape)) <= 1.5e-2, name
    # the bias gradient of the last projection is the plain column sum of dy
    b2 = to_f64(dy).sum(axis=0)
    assert np.abs(grads["b_fc2"].cpu().double().numpy() - 0.5 - b2).max() <= 1e-5 * np.abs(b2).max() + 1e-5
