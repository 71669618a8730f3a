"""Attention backward of lists of short segments at head_dim 80, whose tiles share a pool of buffers, against the same segments in a
list that does not qualify for it (one segment of more than 384 rows, or fewer units than SMs) and against the oracle: unit lengths of
one, two and three steps in turn, around the edges of a tile."""
import numpy as np
import pytest
import torch

import oracle
from paper_2607_03229_b200 import binding as B, workloads as W
from _util import GRAD_REL_L2, rel_l2, status_buf, to_dev, to_f64

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("D", [64, 80])
@pytest.mark.parametrize("counts", [[5], [128], [129, 127], [256, 1, 257], [384, 100, 300, 64, 385 - 1, 31]])
def test_short_lists_give_the_gradients_of_others(counts, D):
    H, T = 2, sum(counts)
    q, k, v, do = (W.normal_bf16(91, i, (T, H, D)) for i in range(4))
    scale = float(np.float32(D ** -0.5))
    cu = np.concatenate([[0], np.cumsum(counts)]).astype(np.int32)

    def run(copies, tail):   # the segments `copies` times over, then `tail` rows of one more
        more = [tail] if tail else []
        plan = B.seg_plan(counts * copies + more, B.TRAINED).to_device()
        n = T * copies + tail
        dev = []
        for x in (q, k, v, do):
            y = torch.zeros((n, H, D), dtype=torch.bfloat16, device="cuda")
            y[:T * copies] = to_dev(x).repeat(copies, 1, 1)
            dev.append(y)
        o, lse, st = torch.empty_like(dev[0]), torch.empty((H, n), device="cuda"), status_buf()
        out = [torch.full_like(dev[0], 7.0) for _ in range(3)]
        ws = torch.empty(B.attn_workspace_bytes(n, H, D, B.TRAINED), dtype=torch.uint8, device="cuda")
        B.varlen_attn_fwd(dev[0], dev[1], dev[2], o, lse, plan, scale, st)
        B.varlen_attn_bwd(dev[3], dev[0], dev[1], dev[2], o, lse, *out, plan, scale, ws, st)
        torch.cuda.synchronize()
        assert st.cpu().tolist()[0] == 0
        return out

    sms = torch.cuda.get_device_properties(0).multi_processor_count
    many = sms // (int(B.seg_plan(counts, B.TRAINED).bwd_items.size) * H) + 1
    few = run(1, 0)
    short, long = run(3 * many, 0), run(3 * many, 385)
    for i in (1, 2):   # dK and dV: the same products in the same order, whatever the schedule
        assert torch.equal(short[i], long[i][:3 * many * T])
        for c in range(3 * many):
            assert torch.equal(short[i][c * T:(c + 1) * T], few[i])
    # dQ: the key tiles' contributions (three at most) are added in any order; fp32 sums, one rounding to bf16
    assert rel_l2(to_f64(short[0]), to_f64(long[0][:3 * many * T])) <= 1e-3
    grads = oracle.attn_bwd(do, q, k, v, cu, scale)
    for i in range(3):   # the bound of the other lists: bf16 P, dS, O and result
        assert rel_l2(to_f64(few[i]), grads[i]) <= GRAD_REL_L2
        for c in (0, 3 * many - 1):
            assert rel_l2(to_f64(short[i][c * T:(c + 1) * T]), grads[i]) <= GRAD_REL_L2
