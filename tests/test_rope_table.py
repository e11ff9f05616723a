"""The plan's table of cosines and sines: shared by rotation calls and the projection, one base at a time."""
import numpy as np
import pytest

from paper_2503_18989_b200 import workloads as W

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("interleaved", [False, True])
def test_calls_with_two_bases_on_one_plan(cuda_device, interleaved):
    """A plan whose table holds one base computes another base's angles in the kernel: the same bits as a plan of its
    own, in any order and in place; 6 heads, so that the last thread of a row has fewer."""
    import torch
    from paper_2503_18989_b200 import binding as B, runner
    rng = np.random.Generator(np.random.PCG64(7))
    prefix, chunk = [0, 37, 4090, 8000], [5, 16, 130, 1]
    table, num_pages = W._place_pages(rng, np.asarray(prefix) + np.asarray(chunk), slack_pages=4)
    st = W._make_step(300, "bf16", 6, 128, prefix, chunk, table)
    sc = W._scenario("rope", "bf16", 6, 128, "paged", num_pages, [st], 300)

    def rotate(plan_of, theta):
        q = torch.empty_like(plan_of.q)
        B.hat_rope_q(plan_of.plan, plan_of.q, q, theta, interleaved)
        B.hat_kv_append_rope(plan_of.cache.desc, plan_of.plan, plan_of.k_new, plan_of.v_new, theta, interleaved)
        torch.cuda.synchronize()
        k, v = plan_of.cache.pools_to_host()
        return q.cpu().numpy(), k, v

    def fresh():
        return runner.DeviceStep(runner.DeviceCache(sc.cache, sc.k_pool, sc.v_pool, cuda_device), st)

    one, two = fresh(), fresh()
    a = rotate(one, 10000.0)
    b = rotate(two, 500000.0)
    assert not np.array_equal(a[0], b[0])
    for theta, want in ((500000.0, b), (10000.0, a), (500000.0, b)):
        for got, ref in zip(rotate(one, theta), want):
            assert np.array_equal(got, ref)
    B.hat_rope_q(two.plan, two.q, two.q, 500000.0, interleaved)
    torch.cuda.synchronize()
    assert np.array_equal(two.q.cpu().numpy(), b[0])
