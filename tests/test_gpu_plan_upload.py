"""The plan's upload on both sides of every size its carriers change at (256, 1024, 3072 and 8128 words as kernel arguments, pinned
memory beyond): what arrives is what the planner wrote, on whichever stream is current."""
import numpy as np
import pytest
import torch

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("segments", [0, 1, 19, 20, 78, 79, 236, 237, 624, 626, 3000])
@pytest.mark.parametrize("side", [False, True])
def test_plan_arrives(segments, side):
    from paper_2607_03229_b200 import binding as B

    counts = [1 + (7 * i) % 128 for i in range(segments)]   # one work item of either kind each: 13 words a segment
    stream = torch.cuda.Stream() if side else torch.cuda.current_stream()
    with torch.cuda.stream(stream):
        plans = [B.seg_plan(counts, B.TRAINED).to_device() for _ in range(3)]
        for p in plans:
            for host, dev in ((p.cu_seqlens, p.cu_seqlens_dev), (p.fwd_items, p.fwd_items_dev), (p.bwd_items, p.bwd_items_dev)):
                assert np.array_equal(dev.cpu().numpy().reshape(-1), np.ascontiguousarray(host).view(np.int32).reshape(-1))
