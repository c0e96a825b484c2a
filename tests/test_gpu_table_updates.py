"""The block table may be written by the kernel right before a run: a streaming launch looks at it early, for
a hint only, and has to compute with what it holds by then."""
import math

import numpy as np
import pytest
import torch

from paper_2412_18106_b200 import binding as xb
from paper_2412_18106_b200 import workloads as W
from tests import helpers as H

pytestmark = pytest.mark.gpu
SCALE = 1.0 / math.sqrt(128.0)


@pytest.mark.parametrize("page,hq,hkv,lens", [(128, 8, 2, [1, 127, 128, 300]), (16, 8, 2, [15, 16, 2000]),
                                              (64, 7, 1, [5000]), (128, 32, 8, [700] * 40)])
@pytest.mark.parametrize("before", [-1, 1 << 30, 0])
def test_table_written_right_before(page, hq, hkv, lens, before):
    import oracle
    b = W.custom("late_table", hq, hkv, page, [(1, n, 0, None) for n in lens], seed=5)
    t = W.make_tensors(b)
    ctx = xb.XYAttn(hq, hkv, page, device=0)
    info = ctx.plan_batch(b)
    assert info.num_dense_tasks == 0
    q, k, v = t.q.cuda(), t.k_pool.cuda(), t.v_pool.cuda()
    good = torch.from_numpy(np.where(b.block_table < 0, 0, b.block_table).astype(np.int32)).cuda()
    table = torch.full_like(good, before)
    qkv = torch.zeros((b.total_q, hq + 2 * hkv, 128), dtype=torch.bfloat16, device="cuda")
    other = torch.zeros_like(k), torch.zeros_like(v)
    outs = []
    for _ in range(3):
        table.fill_(before)
        torch.cuda._sleep(200000)
        table.copy_(good)
        ctx.append_kv(qkv, *other, table)  # into another pool: a launch that lets the run start early
        outs.append(xb.attention(ctx, b, q, k, v, table, SCALE))
    torch.cuda.synchronize()
    assert ctx.device_status() == 0
    O_ref, L_ref = oracle.attention(b, t, SCALE)
    for o, lse in outs:
        H.check_against_oracle(o.double().cpu().numpy(), lse.double().cpu().numpy(), O_ref, L_ref, "late table")
    ctx.close()
