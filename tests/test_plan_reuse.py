"""Plans made and destroyed while earlier steps still run: device memory handed from one plan to the next."""
import numpy as np
import pytest

from paper_2503_18989_b200 import workloads as W

from common import assert_parity, oracle_replay

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("steps,streams", [(3, 1), (150, 1), (150, 2)])     # below and beyond what waits in the list
def test_destroyed_plans_hand_their_memory_on(cuda_device, steps, streams):
    """Three batches in turn, a new plan per step, destroyed right after its call was enqueued."""
    import torch
    from paper_2503_18989_b200 import binding as B, runner
    scs = [W.spec_verify(num_requests=n, min_prefix=40, max_prefix=3000, H=8, seed=500 + n) for n in (3, 9, 17)]
    caches = [runner.DeviceCache(sc.cache, sc.k_pool, sc.v_pool, cuda_device) for sc in scs]
    held = [runner.DeviceStep(c, sc.steps[0]) for c, sc in zip(caches, scs)]
    ss = [torch.cuda.Stream(cuda_device) for _ in range(streams)]
    torch.cuda.synchronize()
    for i in range(steps):
        c, sc, ds = caches[i % 3], scs[i % 3], held[i % 3]
        st, stream = sc.steps[0], ss[(i % 3) % streams]
        plan = B.hat_plan_create(c.desc, 8, st.cu_chunk, st.prefix_len, st.chunk_len, st.block_table)
        if i % 5 == 4:                                       # a call that the plan's own event does not cover
            B.hat_kv_append(c.desc, plan, ds.k_new, ds.v_new, stream.cuda_stream)
        else:
            B.hat_chunk_attention(c.desc, plan, ds.q, ds.k_new, ds.v_new, ds.out, ds.lse, 0.0, ds.workspace,
                                  ds.workspace_bytes, stream.cuda_stream)
        plan.close()
    for sc, c, ds in zip(scs, caches, held):
        out, lse = ds.results()
        kp, vp, want = oracle_replay(sc)
        assert_parity(out, want[0][0], "out")
        assert_parity(lse, want[0][1], "lse")
        gk, gv = c.pools_to_host()
        assert np.array_equal(gk, kp) and np.array_equal(gv, vp)
        assert ds.canaries_intact()
        ds.close()
    B.hat_release_cached()
