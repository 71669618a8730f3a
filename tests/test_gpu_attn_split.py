"""Attention forward with one query tile per unit (few units) and with two (many), around the edges of both tile heights: the same
rows from either, and both against the oracle."""
import numpy as np
import pytest
import torch

import oracle
from paper_2607_03229_b200 import binding as B, workloads as W
from _util import status_buf, to_dev, to_f64

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("D", [64, 80])
@pytest.mark.parametrize("counts", [[1], [127, 1], [128], [129], [256, 257], [300, 128, 385, 5]])
def test_few_units_give_the_rows_of_many(counts, D):
    H, T = 2, sum(counts)
    q, k, v = (W.normal_bf16(71, i, (T, H, D)) for i in range(3))
    scale = float(np.float32(D ** -0.5))

    def run(copies):   # the same images `copies` times over: many units take two query tiles each
        plan = B.seg_plan(counts * copies, B.TRAINED).to_device()
        dq, dk, dv = (to_dev(x).repeat(copies, 1, 1) for x in (q, k, v))
        o, lse, st = torch.full_like(dq, 7.0), torch.zeros((H, T * copies), device="cuda"), status_buf()
        B.varlen_attn_fwd(dq, dk, dv, o, lse, plan, scale, st)
        torch.cuda.synchronize()
        assert st.cpu().tolist()[0] == 0
        return o, lse

    sms = torch.cuda.get_device_properties(0).multi_processor_count
    items = int(B.seg_plan(counts, B.TRAINED).fwd_items.size)
    many = sms // (2 * items * H) + 1
    o1, l1 = run(1)
    o2, l2 = run(many)
    assert torch.equal(o1, o2[:T]) and torch.equal(o1, o2[-T:]) and torch.equal(l1, l2[:, :T])
    cu = np.concatenate([[0], np.cumsum(counts)]).astype(np.int32)
    O_ref, L_ref = oracle.attn_fwd(q, k, v, cu, scale)
    # bf16 probabilities and output: 2^-8 of values of O(1) and of their fp32 sums
    assert np.abs(to_f64(o1) - O_ref).max() <= 1e-2 and np.abs(l1.cpu().double().numpy() - L_ref).max() <= 1e-3
