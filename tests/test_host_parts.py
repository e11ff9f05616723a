"""Calls with host buffers that are large enough to be split into parts (copies overlap the kernels)."""
import numpy as np
import pytest

from paper_2503_18989_b200 import workloads as W

from common import assert_parity, oracle_replay
from test_stream_kernel import _batch

pytestmark = pytest.mark.gpu

# heads odd in number, so that the parts' lse rows are not 16-byte aligned; an empty chunk; requests of every class
_PREFIX = [300, 0, 77, 1000, 16, 640, 5, 129, 900, 33]
_CHUNK = [400, 3, 512, 16, 129, 0, 300, 7, 256, 200]


@pytest.mark.parametrize("dtype,group,tree,pinned", [("fp16", 1, False, True), ("bf16", 2, True, True), ("fp16", 1, False, False)])
def test_parts_of_a_host_call(cuda_device, dtype, group, tree, pinned):
    import torch
    from paper_2503_18989_b200 import binding as B, runner
    H, d = 5, 128
    sc = _batch(dtype, H, d, _PREFIX, _CHUNK, 301, group)
    st = sc.steps[0]
    if tree:
        st.tree_mask = W.random_tree_masks(5, _CHUNK)
    cache = runner.DeviceCache(sc.cache, sc.k_pool, sc.v_pool, cuda_device)
    ds = runner.DeviceStep(cache, st)
    T, Hq = st.total_rows, H * group
    host = lambda a: torch.from_numpy(a.view(np.int16)).pin_memory() if pinned else torch.from_numpy(a.view(np.int16).copy())
    q, k, v = host(st.q), host(st.k_new), host(st.v_new)
    nbytes = B.hat_plan_staging_bytes(ds.plan)
    streams = [torch.cuda.Stream(cuda_device) for _ in range(2)]
    sets = []
    for _ in streams:
        o, l = torch.full((T, Hq, d), float("nan")), torch.full((T, Hq), float("nan"))
        sets.append((o.pin_memory() if pinned else o, l.pin_memory() if pinned else l,
                     torch.empty(nbytes, dtype=torch.uint8, device=cuda_device)))
    torch.cuda.synchronize()
    before = B.hat_launch_count()
    for i in range(6):                                       # alternate streams, two calls in flight
        o, l, stg = sets[i % 2]
        B.hat_chunk_attention_host(cache.desc, ds.plan, q, k, v, o, l, 0.0, stg, nbytes, ds.workspace, ds.workspace_bytes,
                                   streams[i % 2].cuda_stream)
    assert B.hat_launch_count() - before >= 6 * 4             # several parts, a streaming and a tile kernel in most
    torch.cuda.synchronize()
    assert B.hat_last_device_status(ds.plan) == B.HAT_OK
    kp, vp, want = oracle_replay(sc)
    for o, l, _ in sets:
        assert_parity(o.numpy(), want[0][0], "out")
        assert_parity(l.numpy(), want[0][1], "lse")
    gk, gv = cache.pools_to_host()
    assert np.array_equal(gk, kp) and np.array_equal(gv, vp) and ds.canaries_intact()
    ds.close()


def test_drafts_are_announced_in_the_last_part_that_has_some(cuda_device):
    """The verify event of a call in parts: the drafts' rows are final in staging memory when it has occurred; the parts
    behind it hold prompt chunks only."""
    import torch
    from paper_2503_18989_b200 import binding as B, runner
    H, d = 5, 128
    sc = _batch("fp16", H, d, [700, 33] + _PREFIX[:1] + [900, 640, 1000], [4, 16] + _CHUNK[:1] + [512, 500, 512], 303)
    st = sc.steps[0]
    cache = runner.DeviceCache(sc.cache, sc.k_pool, sc.v_pool, cuda_device)
    ds = runner.DeviceStep(cache, st)
    T = st.total_rows
    q, k, v = (torch.from_numpy(a.view(np.int16)).pin_memory() for a in (st.q, st.k_new, st.v_new))
    nbytes = B.hat_plan_staging_bytes(ds.plan)
    o, l = torch.empty((T, H, d)).pin_memory(), torch.empty((T, H)).pin_memory()
    staging = torch.full((nbytes,), 0xFF, dtype=torch.uint8, device=cuda_device)
    s, side = torch.cuda.Stream(cuda_device), torch.cuda.Stream(cuda_device)
    torch.cuda.synchronize()
    before = B.hat_launch_count()
    B.hat_chunk_attention_host(cache.desc, ds.plan, q, k, v, o, l, 0.0, staging, nbytes, ds.workspace, ds.workspace_bytes, s.cuda_stream)
    assert B.hat_launch_count() - before >= 4                         # several parts
    B.hat_plan_wait_verify(ds.plan)
    pad = lambda n: (n + 255) // 256 * 256
    at = 3 * pad(T * H * d * 2)                                       # q, k_new, v_new of as many heads
    with torch.cuda.stream(side):
        rows = staging[at:at + 20 * H * d * 4].cpu().view(torch.float32).view(20, H, d).numpy()
    torch.cuda.synchronize()
    kp, vp, want = oracle_replay(sc)
    assert_parity(rows, want[0][0][:20], "drafts in staging")
    assert_parity(o.numpy(), want[0][0], "out")
    ds.close()


@pytest.mark.parametrize("first,second", [("host", "device"), ("device", "host"), ("host", "host")])
def test_a_call_in_parts_and_the_plans_other_calls_are_ordered(cuda_device, first, second, monkeypatch):
    """Two calls of one plan on two streams: the second one's kernels wait for the first, whichever of them copies from host
    buffers in parts.  The first call is held back by a kernel in front of it; some requests are cut, so that both calls use
    the plan's workspace."""
    import torch
    from paper_2503_18989_b200 import binding as B, runner
    monkeypatch.setenv("HAT_VERIFY_CLUSTER", "0")                     # drafts too in pieces that meet in the workspace
    H, d = 5, 128
    sc = _batch("fp16", H, d, _PREFIX + [30000], _CHUNK + [4], 302)
    st = sc.steps[0]
    cache = runner.DeviceCache(sc.cache, sc.k_pool, sc.v_pool, cuda_device)
    ds = runner.DeviceStep(cache, st)
    assert ds.info["max_splits"] > 1 and ds.workspace_bytes > 0 and ds.info["stream_kernel"] == 1
    T = st.total_rows
    q, k, v = (torch.from_numpy(a.view(np.int16)).pin_memory() for a in (st.q, st.k_new, st.v_new))
    nbytes = B.hat_plan_staging_bytes(ds.plan)
    bufs = [(torch.full((T, H, d), float("nan")).pin_memory(), torch.full((T, H), float("nan")).pin_memory(),
             torch.empty(nbytes, dtype=torch.uint8, device=cuda_device)) for _ in range(2)]
    streams = [torch.cuda.Stream(cuda_device) for _ in range(2)]

    def call(kind, i):
        if kind == "device":
            ds.attend(stream=streams[i].cuda_stream)
        else:
            o, l, stg = bufs[i]
            B.hat_chunk_attention_host(cache.desc, ds.plan, q, k, v, o, l, 0.0, stg, nbytes, ds.workspace, ds.workspace_bytes,
                                       streams[i].cuda_stream)

    before = B.hat_launch_count()
    call("host", 0)                                                   # the parts are planned, everything is loaded
    assert B.hat_launch_count() - before >= 4
    torch.cuda.synchronize()
    for t in (ds.out, ds.lse, *(x for o, l, _ in bufs for x in (o, l))):
        t.fill_(float("nan"))
    torch.cuda.synchronize()
    held, done = torch.cuda.Event(), torch.cuda.Event()
    with torch.cuda.stream(streams[0]):
        torch.cuda._sleep(1_000_000_000)                              # about half a second
        held.record()
    call(first, 0)
    call(second, 1)
    done.record(streams[1])
    while not held.query():
        assert not done.query() or held.query(), "the second call did not wait for the first"
    torch.cuda.synchronize()
    assert B.hat_last_device_status(ds.plan) == B.HAT_OK
    kp, vp, want = oracle_replay(sc)
    got = [(bufs[i][0].numpy(), bufs[i][1].numpy()) if kind == "host" else ds.results() for i, kind in enumerate((first, second))]
    for o, l in got:
        assert_parity(o, want[0][0], "out")
        assert_parity(l, want[0][1], "lse")
    gk, gv = cache.pools_to_host()
    assert np.array_equal(gk, kp) and np.array_equal(gv, vp) and ds.canaries_intact()
    ds.close()
