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


@pytest.mark.parametrize("captured", ["rope", "projection"])
@pytest.mark.parametrize("direct", ["rope", "projection"])
def test_a_replayed_graph_with_another_base(cuda_device, captured, direct):
    """A graph holds a call with one base, direct calls of the same plan use another, before and after a replay: each
    gives the bits it gives on a plan of its own."""
    import torch
    from paper_2503_18989_b200 import binding as B, runner
    rng = np.random.Generator(np.random.PCG64(8))
    H, d, hidden = 2, 128, 192
    prefix, chunk = [0, 37, 4090], [5, 16, 130]
    table, num_pages = W._place_pages(rng, np.asarray(prefix) + np.asarray(chunk), slack_pages=4)
    st = W._make_step(310, "bf16", H, d, prefix, chunk, table)
    sc = W._scenario("rope", "bf16", H, d, "paged", num_pages, [st], 310)
    xb, wb = W.projection_inputs(311, "bf16", st.total_rows, hidden, 3 * H * d)
    x, w = runner._dev_u16(xb, cuda_device), runner._dev_u16(wb, cuda_device)

    def fresh():
        return runner.DeviceStep(runner.DeviceCache(sc.cache, sc.k_pool, sc.v_pool, cuda_device), st)

    def call(kind, ds, theta, q, stream):
        if kind == "rope":
            B.hat_rope_q(ds.plan, ds.q, q, theta, False, stream)
        else:
            B.hat_qkv_rope_append(ds.cache.desc, ds.plan, x, hidden, w, q, theta, False, stream)

    s = torch.cuda.Stream(cuda_device)
    want = {}
    for kind, theta in ((captured, 500000.0), (direct, 10000.0)):
        ds = fresh()
        q = torch.empty_like(ds.q)
        torch.cuda.synchronize()
        call(kind, ds, theta, q, s.cuda_stream)
        torch.cuda.synchronize()
        want[kind, theta] = q.cpu().numpy()
        ds.close()

    ds = fresh()
    q_graph, q = torch.empty_like(ds.q), torch.empty_like(ds.q)
    torch.cuda.synchronize()
    graph = torch.cuda.CUDAGraph()
    with torch.cuda.graph(graph, stream=s):
        call(captured, ds, 500000.0, q_graph, s.cuda_stream)
    for _ in range(3):
        q.fill_(-1)
        q_graph.fill_(-1)
        torch.cuda.synchronize()
        call(direct, ds, 10000.0, q, s.cuda_stream)
        torch.cuda.synchronize()
        assert np.array_equal(q.cpu().numpy(), want[direct, 10000.0])
        with torch.cuda.stream(s):
            graph.replay()
        torch.cuda.synchronize()
        assert np.array_equal(q_graph.cpu().numpy(), want[captured, 500000.0])
    ds.close()
