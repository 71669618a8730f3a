"""Attention forward of lists of one, a few and many waves of units, which ask for their next unit at different times: the same rows from
all, for units of one key tile and of several in turn, on both sides of where the wait for a tile's scores changes."""
import numpy as np
import pytest
import torch

from paper_2607_03229_b200 import binding as B, workloads as W
from _util import status_buf, to_dev

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("D", [64, 80])
@pytest.mark.parametrize("counts", [[35, 154, 128, 129], [256, 1, 257], [384, 385, 100, 512], [300, 1100, 40]])
def test_waves_give_the_same_rows(counts, D):
    H, T = 2, sum(counts)
    q, k, v = (to_dev(W.normal_bf16(97, i, (T, H, D))) for i in range(3))
    sms = torch.cuda.get_device_properties(0).multi_processor_count
    units = int(B.seg_plan(counts, B.TRAINED).fwd_items.size) * H

    def run(copies):
        plan = B.seg_plan(counts * copies, B.TRAINED).to_device()
        dev = [x.repeat(copies, 1, 1) for x in (q, k, v)]
        o, lse, st = torch.full_like(dev[0], 7.0), torch.zeros((H, T * copies), device="cuda"), status_buf()
        B.varlen_attn_fwd(*dev, o, lse, plan, float(np.float32(D ** -0.5)), st)
        torch.cuda.synchronize()
        assert st.cpu().tolist()[0] == 0
        return o, lse

    o1, l1 = run(1)
    for copies in (sms // units + 1, 3 * sms // units, 8 * sms // units, 8 * sms // units + 1):
        o, lse = run(copies)
        assert torch.equal(o, o1.repeat(copies, 1, 1)) and torch.equal(lse, l1.repeat(1, copies)), copies
