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


def test_a_loop_of_plans_allocates_nothing_once_warm(cuda_device):
    """Plans of a few KB (one draft-verification request) and of more than the smallest block, made, used and destroyed in
    turn; and plans of one size after the list is full of another's."""
    import torch
    from paper_2503_18989_b200 import binding as B, runner
    small = W.spec_verify(num_requests=1, min_prefix=700, max_prefix=700, H=8, seed=521)
    large = W.spec_verify(num_requests=24, min_prefix=9000, max_prefix=12000, H=8, seed=522)
    held = []
    for sc in (small, large):
        cache = runner.DeviceCache(sc.cache, sc.k_pool, sc.v_pool, cuda_device)
        held.append((cache, runner.DeviceStep(cache, sc.steps[0]), sc.steps[0]))

    def make(cache, st):
        return B.hat_plan_create(cache.desc, 8, st.cu_chunk, st.prefix_len, st.chunk_len, st.block_table)

    def loop(which, n):
        cache, ds, st = held[which]
        for _ in range(n):
            plan = make(cache, st)
            B.hat_chunk_attention(cache.desc, plan, ds.q, ds.k_new, ds.v_new, ds.out, ds.lse, 0.0, ds.workspace, ds.workspace_bytes)
            torch.cuda.synchronize()
            plan.close()

    for which in (0, 1):
        loop(which, 1)
        warm = B.hat_device_alloc_count()
        loop(which, 80)
        assert B.hat_device_alloc_count() == warm
    plans = [make(held[0][0], held[0][2]) for _ in range(70)]         # more than wait in the list
    B.hat_release_cached()
    for plan in plans:
        plan.close()
    loop(1, 1)
    warm = B.hat_device_alloc_count()
    loop(1, 5)
    assert B.hat_device_alloc_count() == warm
    for _, ds, _ in held:
        ds.close()
    B.hat_release_cached()
