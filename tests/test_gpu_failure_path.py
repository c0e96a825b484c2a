"""The device-side failure path and the validation aid, exercised without faulting the GPU.

A bounded wait is made to run out: the producer of the only worker leaves out one stage fill
(nothing reads unwritten memory, the readers simply never see the stage filled) while the wait
limit is short.  The kernel must return, the status must show the timeout, and the next ordinary
run on the same context must be correct."""
import os

import numpy as np
import pytest
import torch

import oracle
from paper_2412_18106_b200 import binding as xb
from paper_2412_18106_b200 import workloads as W
from tests import helpers as H

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("kernel", [xb.XY_KERNEL_AUTO, xb.XY_KERNEL_MMA], ids=["auto", "mma"])
@pytest.mark.parametrize("skip", [0, 3, 9])
def test_a_wait_that_runs_out_is_reported_and_the_context_recovers(kernel, skip):
    b = W.config1_tiny()
    t = W.make_tensors(b)
    ctx = H.make_ctx(b, kernel=kernel, num_workers=1)
    ctx.plan_batch(b)
    d = H.DeviceBatch(b, t)
    O_ref, LSE_ref = oracle.attention(b, t, H.SCALE)
    ctx.debug_inject(wait_limit_polls=20000, skip_fill=skip)
    ctx.run(d.q, d.k_pool, d.v_pool, d.block_table, H.SCALE, d.o, d.lse)
    torch.cuda.synchronize()                       # the kernel returned
    assert ctx.device_status() == xb.XY_ERR_DEVICE_TIMEOUT
    assert ctx.device_status() == 0                # reported once, then cleared
    # an ordinary run without reading the status in between also recovers
    ctx.run(d.q, d.k_pool, d.v_pool, d.block_table, H.SCALE, d.o, d.lse)
    ctx.debug_inject(0, -1)
    for _ in range(2):
        o = torch.full_like(d.o, float("nan"))
        lse = torch.full_like(d.lse, float("nan"))
        ctx.run(d.q, d.k_pool, d.v_pool, d.block_table, H.SCALE, o, lse)
        torch.cuda.synchronize()
        H.check_against_oracle(o.float().cpu().numpy().astype(np.float64), lse.cpu().numpy().astype(np.float64),
                               O_ref, LSE_ref, "run after a timeout")
    assert ctx.device_status() == xb.XY_ERR_DEVICE_TIMEOUT   # the second failing run is on record too
    assert ctx.device_status() == 0
    ctx.close()
    # tensor memory was freed: a fresh context (which allocates all 512 columns again) works
    H.parity(b, kernel=kernel, num_workers=1)


def test_debug_context_rejects_a_bad_block_table_before_launching():
    os.environ["XY_ATTN_DEBUG"] = "1"
    try:
        b = W.config1_tiny()
        ctx = H.make_ctx(b)
    finally:
        del os.environ["XY_ATTN_DEBUG"]
    ctx.plan_batch(b)
    t = W.make_tensors(b)
    d = H.DeviceBatch(b, t)
    good = d.block_table.clone()
    d.block_table[3, 2] = b.num_pages + 7
    with pytest.raises(xb.XYAttnError) as e:
        ctx.run(d.q, d.k_pool, d.v_pool, d.block_table, H.SCALE, d.o, d.lse)
    assert e.value.code == xb.XY_ERR_INVALID_ARG and "request 3" in str(e.value)
    torch.cuda.synchronize()
    assert ctx.last_launches() == 0 and torch.isnan(d.lse).all()
    ctx.run(d.q, d.k_pool, d.v_pool, good, H.SCALE, d.o, d.lse)
    torch.cuda.synchronize()
    assert ctx.device_status() == 0
    O_ref, LSE_ref = oracle.attention(b, t, H.SCALE)
    H.check_against_oracle(d.o.float().cpu().numpy().astype(np.float64), d.lse.cpu().numpy().astype(np.float64),
                           O_ref, LSE_ref, "debug context")
    ctx.close()


@pytest.mark.parametrize("workers,decode", [(3, True), (40, True), (0, True), (5, False), (0, False)],
                         ids=["stream-3", "stream-40", "stream-all", "meta-5", "meta-all"])
def test_many_ctas_that_give_up_leave_a_clean_context(workers, decode):
    """Every CTA gives up after a fill that never comes, with split units half counted and the queue half
    dealt: the next ordinary run, with and without reading the status in between, is right, and bitwise
    what the runs before the failure gave."""
    b = W.config2_decode(num_requests=9, kv_lo=300, kv_hi=3000) if decode else W.config1_tiny()
    t = W.make_tensors(b)
    ctx = H.make_ctx(b, num_workers=workers)
    ctx.plan_batch(b)
    d = H.DeviceBatch(b, t)

    def run():
        o, lse = torch.full_like(d.o, float("nan")), torch.full_like(d.lse, float("nan"))
        ctx.run(d.q, d.k_pool, d.v_pool, d.block_table, H.SCALE, o, lse)
        return o, lse

    good = [run() for _ in range(3)]
    for read in (True, False):
        ctx.debug_inject(wait_limit_polls=20000, skip_fill=1)
        run()
        ctx.debug_inject(0, -1)
        if read:
            assert ctx.device_status() == xb.XY_ERR_DEVICE_TIMEOUT
        good += [run() for _ in range(2)]
    assert ctx.device_status() == xb.XY_ERR_DEVICE_TIMEOUT and ctx.device_status() == 0
    O_ref, LSE_ref = oracle.attention(b, t, H.SCALE)
    for o, lse in good:
        assert torch.equal(lse, good[0][1])
    o, lse = good[-1]
    H.check_against_oracle(o.float().cpu().numpy().astype(np.float64), lse.cpu().numpy().astype(np.float64), O_ref, LSE_ref,
                           "run after a timeout")


@pytest.mark.parametrize("workers,skip,decode", [(3, 20, True), (3, 45, True), (20, 1, True), (2, 2, False), (7, 20, False),
                                                 (100, 1, False)])
def test_status_read_clears_what_a_cleaner_that_gave_up_has_left(workers, skip, decode):
    """With a wait limit of one poll the CTA that cleans up after a failure does not wait for the others (as if they
    could not get an SM).  Queue head and counters then stay as they are; reading the status clears them, so that
    the runs behind it are ordinary ones."""
    b = (W.config2_decode(num_requests=9, kv_lo=300, kv_hi=3000) if decode else
         W.config3_splitfuse(chunk=300, prefix=300, num_decode=9, kv_lo=200, kv_hi=1500))
    t = W.make_tensors(b)
    O_ref, LSE_ref = oracle.attention(b, t, H.SCALE)
    ctx = H.make_ctx(b, num_workers=workers)
    ctx.plan_batch(b)
    d = H.DeviceBatch(b, t)
    for _ in range(3):
        ctx.debug_inject(wait_limit_polls=1, skip_fill=skip)
        ctx.run(d.q, d.k_pool, d.v_pool, d.block_table, H.SCALE, d.o, d.lse)
        ctx.debug_inject(0, -1)
        assert ctx.device_status() == xb.XY_ERR_DEVICE_TIMEOUT
        for _ in range(2):
            o, lse = torch.full_like(d.o, float("nan")), torch.full_like(d.lse, float("nan"))
            ctx.run(d.q, d.k_pool, d.v_pool, d.block_table, H.SCALE, o, lse)
            assert ctx.device_status() == 0
            H.check_against_oracle(o.float().cpu().numpy().astype(np.float64), lse.cpu().numpy().astype(np.float64), O_ref,
                                   LSE_ref, "run after a status read")
    ctx.close()


@pytest.mark.parametrize("workers", [0, 7])
@pytest.mark.parametrize("skip", [0, 1, 6])
def test_two_launches_side_by_side_give_up_and_leave_a_clean_context(skip, workers):
    """The dense and the streaming launch of a shared-prefix plan share the status word and the unit counters,
    side by side as one after the other (7 workers): after a wait that ran out in either, the next ordinary runs
    are bitwise what they were before."""
    b, groups = W.shared_prefix_decode(seed=7, num_groups=5, members=42, prefix=512, suffix_hi=400, hq=16, hkv=4)
    t = W.make_tensors(b)
    ctx = H.make_ctx(b, num_workers=workers, max_requests=512)
    ctx.plan_batch(b, groups=groups)
    d = H.DeviceBatch(b, t)

    def run():
        o, lse = torch.full_like(d.o, float("nan")), torch.full_like(d.lse, float("nan"))
        ctx.run(d.q, d.k_pool, d.v_pool, d.block_table, H.SCALE, o, lse)
        assert ctx.last_launches() == 3
        return o, lse

    good = run()
    H.check_against_oracle(good[0].float().cpu().numpy().astype(np.float64), good[1].cpu().numpy().astype(np.float64),
                           *oracle.attention(b, t, H.SCALE), "two launches")
    for read in (True, False):
        ctx.debug_inject(wait_limit_polls=20000, skip_fill=skip)
        run()
        ctx.debug_inject(0, -1)
        if read:
            assert ctx.device_status() == xb.XY_ERR_DEVICE_TIMEOUT
        for _ in range(2):
            o, lse = run()
            assert torch.equal(o, good[0]) and torch.equal(lse, good[1])
    assert ctx.device_status() == xb.XY_ERR_DEVICE_TIMEOUT and ctx.device_status() == 0
    ctx.close()


# (The tiny batch has 32 fills: with two workers one of them comes to its twelfth however the tasks fall; with five
# that would depend on their pace.)
@pytest.mark.parametrize("decode,workers", [(True, 3), (True, 0), (False, 2)], ids=["stream-3", "stream-all", "meta-2"])
@pytest.mark.parametrize("skip", [1, 11])
def test_fp8_run_gives_up_and_the_context_recovers(decode, workers, skip):
    b = W.config2_decode(num_requests=9, kv_lo=300, kv_hi=3000) if decode else W.config1_tiny()
    t8 = W.to_fp8_kv(W.make_tensors(b))
    ctx = H.make_ctx(b, num_workers=workers, kv_dtype=xb.XY_KV_FP8_E4M3)
    ctx.plan_batch(b)
    q, k, v, ks, vs = (x.cuda() for x in (t8.q, t8.k_pool, t8.v_pool, t8.k_scale, t8.v_scale))
    bt = torch.from_numpy(np.where(b.block_table < 0, 0, b.block_table).astype(np.int32)).cuda()

    def run():
        o = torch.full((b.total_q, b.num_q_heads, 128), float("nan"), dtype=torch.bfloat16, device="cuda")
        lse = torch.full((b.total_q, b.num_q_heads), float("nan"), dtype=torch.float32, device="cuda")
        ctx.run_fp8kv(q, k, v, ks, vs, bt, H.SCALE, o, lse)
        return o, lse

    good = run()
    H.check_against_oracle(good[0].float().cpu().numpy().astype(np.float64), good[1].cpu().numpy().astype(np.float64),
                           *oracle.attention_fp8(b, t8, H.SCALE), "fp8")
    for read in (True, False):
        ctx.debug_inject(wait_limit_polls=20000, skip_fill=skip)
        run()
        ctx.debug_inject(0, -1)
        if read:
            assert ctx.device_status() == xb.XY_ERR_DEVICE_TIMEOUT
        for _ in range(2):
            o, lse = run()
            assert torch.equal(o, good[0]) and torch.equal(lse, good[1])
    ctx.close()


# Batches for one worker, which comes to every fill: a long streaming task beside a chunk, a long dense task beside a
# short one, and many tasks of one to four tiles.
AHEAD = {
    "stream": [(500, 0, 0, None), (1, 6000, 0, None)],
    "dense": [(64, 5000, 0, None), (1, 90, 0, None)],
    "short": [(500, 0, 0, None)] + [(1, 20 + 2 * i, 0, None) for i in range(14)],
}


@pytest.mark.parametrize("fp8,kernel", [(False, xb.XY_KERNEL_AUTO), (False, xb.XY_KERNEL_MMA), (True, xb.XY_KERNEL_AUTO)],
                         ids=["auto", "mma", "fp8"])
@pytest.mark.parametrize("batch", sorted(AHEAD))
@pytest.mark.parametrize("skip", [24, 25, 38, 39])
def test_one_tile_missing_while_the_producers_are_ahead(batch, skip, fp8, kernel):
    """A K tile (even) or a V tile (odd) is left out deep in a run: the other kind's stages are full, their producer
    waits for its readers or has tasks in hand that nobody has read, and copies are in flight.  The run ends, every
    role and warp of it, and the runs behind it are bitwise those before it."""
    b = W.custom("ahead_" + batch, 8, 2, 64, AHEAD[batch], seed=21)
    kw = dict(num_workers=1, kernel=kernel)
    if fp8:
        kw["kv_dtype"] = xb.XY_KV_FP8_E4M3
    ctx = H.make_ctx(b, **kw)
    info = ctx.plan_batch(b)
    tasks = ctx.get_tasks()
    assert info.num_dense_tasks > 0 and 2 * int((tasks["kt_hi"] - tasks["kt_lo"]).sum()) > skip
    t = W.make_tensors(b)
    t = W.to_fp8_kv(t) if fp8 else t
    q, k, v = t.q.cuda(), t.k_pool.cuda(), t.v_pool.cuda()
    scales = (t.k_scale.cuda(), t.v_scale.cuda()) if fp8 else ()
    bt = torch.from_numpy(np.where(b.block_table < 0, 0, b.block_table).astype(np.int32)).cuda()

    def run():
        o = torch.full((b.total_q, b.num_q_heads, 128), float("nan"), dtype=torch.bfloat16, device="cuda")
        lse = torch.full((b.total_q, b.num_q_heads), float("nan"), dtype=torch.float32, device="cuda")
        (ctx.run_fp8kv if fp8 else ctx.run)(q, k, v, *scales, bt, H.SCALE, o, lse)
        return o, lse

    good = run()
    assert ctx.last_launches() == 1  # both kinds of task by the meta-kernel
    ref = oracle.attention_fp8(b, t, H.SCALE) if fp8 else oracle.attention(b, t, H.SCALE)
    H.check_against_oracle(good[0].float().cpu().numpy().astype(np.float64), good[1].cpu().numpy().astype(np.float64),
                           *ref, batch)
    for limit in (20000, 1):
        ctx.debug_inject(wait_limit_polls=limit, skip_fill=skip)
        run()
        ctx.debug_inject(0, -1)
        assert ctx.device_status() == xb.XY_ERR_DEVICE_TIMEOUT and ctx.device_status() == 0
        o, lse = run()
        assert ctx.device_status() == 0 and torch.equal(o, good[0]) and torch.equal(lse, good[1])
    ctx.close()
