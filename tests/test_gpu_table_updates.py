"""What a run is given may be written by the kernel right before it: the block table, the scales of an fp8 cache, a
mask of the caller's.  A streaming launch looks at the table early, for a hint only, while that kernel is still
running; every run has to compute with what they hold by then.

The kernel before is an append of one token with many heads, which lets its successor in before its stores: its V
rows, written last, are the table, the scales and the mask of the run behind it."""
import numpy as np
import pytest
import torch

import oracle
from paper_2412_18106_b200 import binding as xb
from paper_2412_18106_b200 import workloads as W
from tests import helpers as H

pytestmark = pytest.mark.gpu
HEADS = 1024  # K, then V heads of 256 bytes each, 4 KB in flight at a time: tens of microseconds


class LateWriter:
    """Lays int32 / float32 / int64 arrays out at the end of the V rows of one token and writes them there by append_kv."""

    def __init__(self, arrays):
        self.ctx = xb.XYAttn(HEADS, HEADS, 8, max_requests=1, max_q_tokens=1, max_pages_per_req=1, workspace_bytes=1 << 20)
        self.ctx.plan([1], [0], [0], [-1], None)
        # [page, token, head, D]: the heads of a token are neighbours
        pools = [torch.zeros((1, 8, HEADS, 128), dtype=torch.bfloat16, device="cuda") for _ in range(2)]
        self.k, self.v = (p.permute(0, 2, 1, 3) for p in pools)
        self.row = pools[1].view(-1)[: HEADS * 128].view(torch.uint8)
        self.table = torch.zeros((1, 1), dtype=torch.int32, device="cuda")
        self.qkv = torch.zeros((1, 3 * HEADS, 128), dtype=torch.bfloat16, device="cuda")
        src = self.qkv.view(-1)[2 * HEADS * 128:].view(torch.uint8)
        self.views, self.good, end = [], [], self.row.numel()
        for a in arrays:
            n = a.numel() * a.element_size()
            end = (end - n) & ~255
            assert end > self.row.numel() // 2  # in the last quarter of what the append writes
            src[end:end + n] = a.contiguous().cuda().view(-1).view(torch.uint8)
            self.views.append(self.row[end:end + n].view(a.dtype).view(a.shape))
            self.good.append(a)

    def write(self, before):
        """Fills the arrays with `before` and queues the append that completes them."""
        for v, b in zip(self.views, before):
            v.copy_(b) if torch.is_tensor(b) else v.fill_(b)
        torch.cuda._sleep(400000)  # what follows is queued before it begins
        self.ctx.append_kv(self.qkv, self.k, self.v, self.table)

    def check(self):
        assert all(torch.equal(v.cpu().view(torch.uint8), g.view(torch.uint8)) for v, g in zip(self.views, self.good))


TREE = np.array([-1, 0, 0], dtype=np.int32)
DECODE = [
    (128, 8, 2, [(1, n, 0, None) for n in (1, 127, 128, 300)]),
    (16, 8, 2, [(1, n, 0, None) for n in (15, 16, 2000)]),
    (64, 7, 1, [(1, 5000, 0, None)]),
    (128, 32, 8, [(1, 700, 0, None)] * 40),
    (32, 8, 2, [(3, 200, 1, TREE), (1, 900, 0, None), (3, 126, 1, TREE)]),
]
MIXED = (32, 8, 2, [(90, 200, 0, None), (40, 300, 1, W.random_tree(np.random.default_rng(3), 40, 6)), (1, 1000, 0, None),
                    (3, 130, 1, TREE)])


@pytest.mark.parametrize("page,hq,hkv,reqs", DECODE + [MIXED], ids=["p128", "p16", "long", "many", "trees", "mixed"])
@pytest.mark.parametrize("before", ["negative", "huge", "zero", "others"])
@pytest.mark.parametrize("fp8", [False, True], ids=["bf16", "fp8"])
def test_tables_written_right_before(page, hq, hkv, reqs, before, fp8):
    b = W.custom("late_table", hq, hkv, page, reqs, seed=5)
    t = W.make_tensors(b)
    t = W.to_fp8_kv(t) if fp8 else t
    ctx = xb.XYAttn(hq, hkv, page, device=0, kv_dtype=xb.XY_KV_FP8_E4M3 if fp8 else xb.XY_KV_BF16)
    info = ctx.plan_batch(b)
    assert (info.num_dense_tasks == 0) == (reqs is not MIXED[3])
    q, k, v = t.q.cuda(), t.k_pool.cuda(), t.v_pool.cuda()
    table = torch.from_numpy(np.where(b.block_table < 0, 0, b.block_table).astype(np.int32))
    mask = torch.from_numpy(ctx.get_tree_mask().view(np.int64).copy())
    late = [table] + ([t.k_scale, t.v_scale] if fp8 else []) + ([mask] if mask.numel() else [])
    w = LateWriter(late)
    # the pages of other requests, in range but wrong; scales and masks that would show
    stale = [{"negative": -1, "huge": 1 << 30, "zero": 0, "others": table.roll(1, 0).flip(1)}[before]]
    stale += ([float("nan")] * 2 if fp8 else []) + ([0] if mask.numel() else [])
    outs = []
    for _ in range(3):
        o = torch.full((b.total_q, hq, 128), float("nan"), dtype=torch.bfloat16, device="cuda")
        lse = torch.full((b.total_q, hq), float("nan"), dtype=torch.float32, device="cuda")
        w.write(stale)
        dev = list(w.views)
        bt, scales = dev.pop(0), [dev.pop(0), dev.pop(0)] if fp8 else []
        (ctx.run_fp8kv if fp8 else ctx.run)(q, k, v, *scales, bt, H.SCALE, o, lse, tree_mask=dev[0] if dev else None)
        outs.append((o, lse))
    torch.cuda.synchronize()
    assert ctx.device_status() == 0
    w.check()
    ref = oracle.attention_fp8(b, t, H.SCALE) if fp8 else oracle.attention(b, t, H.SCALE)
    for o, lse in outs:
        H.check_against_oracle(o.double().cpu().numpy(), lse.double().cpu().numpy(), *ref, "late table")
    ctx.close()
    w.ctx.close()
