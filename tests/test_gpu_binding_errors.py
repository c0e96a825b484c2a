"""Arguments that cannot be served raise an ordinary exception, whichever form of the call looks at them."""
import pytest
import torch

from paper_2412_18106_b200 import gemm as xg
from paper_2412_18106_b200 import workloads as W
from tests import helpers as H

pytestmark = pytest.mark.gpu


def test_sparse_tensors_raise():
    b = W.config1_tiny()
    d = H.DeviceBatch(b, W.make_tensors(b))
    ctx = H.make_ctx(b)
    ctx.plan_batch(b)
    good = [d.q, d.k_pool, d.v_pool, d.block_table, H.SCALE, d.o, d.lse]
    for i in (0, 1, 2, 3, 5, 6):
        args = list(good)
        args[i] = args[i].nan_to_num(0.0).to_sparse() if args[i].is_floating_point() else args[i].to_sparse()
        with pytest.raises(Exception):
            ctx.run(*args)
    with pytest.raises(Exception):
        ctx.run(*good, tree_mask=torch.zeros((4, 4), device="cuda").to_sparse())
    qkv = torch.zeros((b.total_q, b.num_q_heads + 2 * b.num_kv_heads, 128), dtype=torch.bfloat16, device="cuda")
    with pytest.raises(Exception):
        ctx.append_kv(qkv.to_sparse(), d.k_pool, d.v_pool, d.block_table)
    a, w, c = (torch.zeros((64, 64), dtype=torch.bfloat16, device="cuda") for _ in range(3))
    for args in ((a.to_sparse(), w, c), (a, w.to_sparse(), c), (a, w, c.to_sparse())):
        with pytest.raises(Exception):
            xg.xy_gemm_run(*args)
    with pytest.raises(Exception):
        xg.xy_gemm_run(a, w, c, workspace=torch.zeros(64, dtype=torch.uint8, device="cuda").to_sparse())
    ctx.run(*good)  # and the context is as before
    assert ctx.device_status() == 0
    ctx.close()


def test_wrong_types_and_strides_raise():
    b = W.config1_tiny()
    d = H.DeviceBatch(b, W.make_tensors(b))
    ctx = H.make_ctx(b)
    ctx.plan_batch(b)
    good = [d.q, d.k_pool, d.v_pool, d.block_table, H.SCALE, d.o, d.lse]
    bad = [(0, d.q.float()), (0, d.q.cpu()), (0, d.q.transpose(1, 2)), (3, d.block_table.long()), (4, float("nan")), (4, "1"),
           (5, d.o.half()), (6, d.lse.double()), (6, d.lse.t()), (1, d.k_pool.transpose(1, 2))]
    for i, x in bad:
        args = list(good)
        args[i] = x
        with pytest.raises(Exception):
            ctx.run(*args)
    ctx.close()
