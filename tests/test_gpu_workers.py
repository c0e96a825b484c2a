"""A context with fewer workers than the device has SMs leaves the others alone."""
import numpy as np
import pytest
import torch

import oracle
from paper_2412_18106_b200 import workloads as W
from tests import helpers as H

pytestmark = pytest.mark.gpu


def batches():
    shared, groups = W.shared_prefix_decode(seed=3, num_groups=5, members=42, prefix=512, suffix_hi=400, hq=16, hkv=4)
    return {"decode": (W.config2_decode(num_requests=30, kv_lo=100, kv_hi=1500), None),
            "mix": (W.config3_splitfuse(chunk=300, prefix=300, num_decode=9, kv_lo=200, kv_hi=1500), None),
            "shared": (shared, groups)}


@pytest.mark.parametrize("name", ["decode", "mix", "shared"])
@pytest.mark.parametrize("workers", [1, 7, 100])
def test_no_more_ctas_than_workers(name, workers):
    b, groups = batches()[name]
    t = W.make_tensors(b)
    ctx = H.make_ctx(b, num_workers=workers, max_requests=512)
    ctx.plan_batch(b, groups=groups)
    O, LSE = H.run_gpu(b, t, ctx=ctx)
    assert 1 <= ctx.last_ctas() <= workers
    H.check_against_oracle(O, LSE, *oracle.attention(b, t, H.SCALE), name)
    w = ctx.worker_times().astype(np.int64)
    assert w.shape == (workers, 4) and w[:, 3].sum() > 0
    assert (w[:, 2].sum() > 0) == (name != "decode")
    ctx.close()


def test_whole_device_runs_two_streaming_ctas_per_worker():
    sms = torch.cuda.get_device_properties(0).multi_processor_count
    b = W.config2_decode(num_requests=100, kv_lo=500, kv_hi=3000)
    ctx = H.make_ctx(b)
    ctx.plan_batch(b)
    H.run_gpu(b, W.make_tensors(b), ctx=ctx)
    assert ctx.last_ctas() == min(len(ctx.get_tasks()), 2 * sms)
    ctx.close()
