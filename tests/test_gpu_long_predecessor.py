"""A projection inside a layer loads its first weights while the attention before it still runs: however long that takes (here more
than the second after which a wait inside a kernel gives up), the layer ends with its result and without a time-out."""
import numpy as np
import pytest
import torch

from paper_2607_03229_b200 import binding as B, dist as D
from _util import status_buf

pytestmark = pytest.mark.gpu


def test_attention_of_more_than_a_second():
    T, hidden = 2_000_000, 64          # one segment, one head: 1.0e15 FLOPs
    ffn = 512
    gen = torch.Generator(device="cuda").manual_seed(95)
    p = {}
    for name, shape in D.LAYER_PARAM_SHAPES:
        s = shape(hidden, ffn)
        std, mean = (s[-1] ** -0.5, 0.0) if len(s) > 1 else (0.1, 1.0 if name.endswith("gamma") else 0.0)
        p[name] = (torch.randn(s, device="cuda", generator=gen) * std + mean).bfloat16()
    x = torch.randn((T, hidden), device="cuda", generator=gen).bfloat16()
    y, st = torch.empty_like(x), status_buf()
    ws = torch.empty(B.encoder_layer_workspace_bytes(T, hidden, ffn), dtype=torch.uint8, device="cuda")
    plan = B.seg_plan([T], B.FROZEN).to_device()
    ev = [torch.cuda.Event(enable_timing=True) for _ in range(2)]
    ev[0].record()
    B.encoder_layer_fwd(x, y, B.LayerWeights.from_tensors(**p), 1, ffn, plan, float(np.float32(hidden ** -0.5)), 1e-6, ws, None, st)
    ev[1].record()
    torch.cuda.synchronize()
    assert st.cpu().tolist()[0] == 0
    assert ev[0].elapsed_time(ev[1]) > 1100        # or the sizes have to grow with the machine
    w = {k: v.double() for k, v in p.items()}
    ln = lambda t, which: torch.nn.functional.layer_norm(t, (hidden,), w[which + "_gamma"], w[which + "_beta"], 1e-6)
    rows = torch.tensor([0, 777_777, T - 1], device="cuda")
    kv = [ln(x[i:i + 250_000].double(), "ln1") @ w["w_qkv"].t() + w["b_qkv"] for i in range(0, T, 250_000)]
    k, v = (torch.cat([c[:, i * hidden:(i + 1) * hidden] for c in kv]) for i in (1, 2))
    xr = x[rows].double()
    q = (ln(xr, "ln1") @ w["w_qkv"].t() + w["b_qkv"])[:, :hidden]
    x1 = xr + torch.softmax(q @ k.t() * hidden ** -0.5, -1) @ v @ w["w_o"].t() + w["b_o"]
    ref = x1 + torch.nn.functional.gelu(ln(x1, "ln2") @ w["w_fc1"].t() + w["b_fc1"]) @ w["w_fc2"].t() + w["b_fc2"]
    # one layer: the bf16-rounded intermediates of the other layer tests
    assert float((y[rows].double() - ref).norm() / ref.norm()) <= 1e-2
