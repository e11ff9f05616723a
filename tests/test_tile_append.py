"""The append inside the tile kernels: pages shared by prefix and chunk, pages the chunk does not fill, row blocks and key
ranges that share pages, grouped heads, both kernels in one call, and streaming-class chunks in the same call."""
import numpy as np
import pytest

from paper_2503_18989_b200 import workloads as W

from test_stream_kernel import _batch, _check

pytestmark = pytest.mark.gpu

# prefix mod 16 of 0 and not, chunks that end inside and at the end of a page, one and several row blocks, empty prefixes
_PREFIX = [0, 1, 15, 16, 128, 250, 127, 129, 0, 1000, 33]
_CHUNK = [17, 31, 64, 48, 128, 129, 256, 257, 512, 300, 7]


@pytest.mark.parametrize("dtype,d,group,layout", [("fp16", 128, 1, "paged"), ("bf16", 128, 1, "paged"), ("bf16", 128, 4, "contiguous"),
                                                  ("fp16", 64, 2, "contiguous"), ("bf16", 64, 1, "paged")])
def test_append_on_the_way(cuda_device, dtype, d, group, layout):
    _check(_batch(dtype, 2, d, _PREFIX, _CHUNK, 61 + group, group, layout), cuda_device, repeat=2)


@pytest.mark.parametrize("kernel", ["pair", "tc5"])
@pytest.mark.parametrize("dtype", ["fp16", "bf16"])
@pytest.mark.parametrize("split", ["0", "256"])        # key ranges that end inside the chunk
def test_append_in_each_tile_kernel(cuda_device, kernel, dtype, split, monkeypatch):
    monkeypatch.setenv("HAT_PREFILL_KERNEL", kernel)
    monkeypatch.setenv("HAT_PREFILL_SPLIT_LEN", split)
    _check(_batch(dtype, 3, 128, _PREFIX, _CHUNK, 71), cuda_device)


@pytest.mark.parametrize("kernel", ["pair", "tc5"])
def test_pool_strides_that_fold_neither_way(cuda_device, kernel, monkeypatch):
    """Pages with a gap behind the tokens of a head and one behind the heads: two boxes per page instead of one."""
    import torch
    from paper_2503_18989_b200 import binding as B, runner
    from common import assert_parity, oracle_replay
    monkeypatch.setenv("HAT_PREFILL_KERNEL", kernel)
    H, d = 2, 128
    sc = _batch("bf16", H, d, _PREFIX, _CHUNK, 91)
    st, n = sc.steps[0], sc.cache.num_pages
    s_head, s_page = 16 * d + 64, H * (16 * d + 64) + 128
    pools = []
    for src in (sc.k_pool, sc.v_pool):
        wide = np.full((n, s_page), 0x7FC0, np.uint16)                       # NaN in the gaps
        for h in range(H):
            wide[:, h * s_head:h * s_head + 16 * d] = src.reshape(n, H, 16 * d)[:, h]
        pools.append(wide)
    dev = [torch.from_numpy(p.view(np.int16)).to(cuda_device) for p in pools]
    desc = B.make_cache_desc("bf16", n, H, d, s_page, d, s_head, dev[0], dev[1])
    plan = B.hat_plan_create(desc, H, st.cu_chunk, st.prefix_len, st.chunk_len, st.block_table)
    q, k, v = (runner._dev_u16(x, cuda_device) for x in (st.q, st.k_new, st.v_new))
    out = torch.zeros((st.total_rows, H, d), device=cuda_device)
    lse = torch.zeros((st.total_rows, H), device=cuda_device)
    nb = B.hat_plan_workspace_bytes(plan)
    ws = torch.empty(max(nb, 256), dtype=torch.uint8, device=cuda_device)
    B.hat_chunk_attention(desc, plan, q, k, v, out, lse, 0.0, ws, nb)
    torch.cuda.synchronize()
    assert B.hat_last_device_status(plan) == B.HAT_OK
    kp, vp, want = oracle_replay(sc)
    assert_parity(out.cpu().numpy(), want[0][0], "out")
    assert_parity(lse.cpu().numpy(), want[0][1], "lse")
    for got, before, ref in zip(dev, pools, (kp, vp)):
        got = got.cpu().numpy().view(np.uint16)
        for h in range(H):
            cols = slice(h * s_head, h * s_head + 16 * d)
            assert np.array_equal(got[:, cols], ref.reshape(n, H, 16 * d)[:, h])
            before[:, cols] = got[:, cols]
        assert np.array_equal(got, before)                                   # the gaps are untouched


def test_wide_and_narrow_units_together_back_to_back(cuda_device):
    """bf16 batches with both kinds of units run both kernels, the second one in the tail of the first; calls follow
    without a wait."""
    rng = np.random.default_rng(5)
    chunk = rng.choice([17, 64, 100, 128, 200, 256, 300, 512], size=9).tolist()
    prefix = rng.integers(0, 1500, size=9).tolist()
    _check(_batch("bf16", 8, 128, prefix, chunk, 81), cuda_device, repeat=20)


@pytest.mark.parametrize("d,drafts", [(128, False), (128, True), (64, False)])
@pytest.mark.parametrize("requests,apart", [(37, False), (38, True)])     # 8 heads: two units a CTA at most, and just above
def test_append_in_front_of_many_short_units(cuda_device, d, drafts, requests, apart):
    """Above two units a CTA of the one-CTA kernel, short ones, a kernel in front appends; the launches tell which way it went."""
    from paper_2503_18989_b200 import binding as B, runner
    rng = np.random.default_rng(requests)
    prefix = rng.integers(0, 400, size=requests).tolist() + ([700, 33] if drafts else [])
    chunk = rng.integers(17, 128, size=requests).tolist() + ([4, 16] if drafts else [])
    sc = _batch("fp16", 8, d, prefix, chunk, 95)
    cache = runner.DeviceCache(sc.cache, sc.k_pool, sc.v_pool, cuda_device)
    ds = runner.DeviceStep(cache, sc.steps[0])
    assert ds.info["prefill_kernel"] == 1 and ds.info["prefill_split_len"] == 0      # (cut drafts are merged without a launch)
    before = B.hat_launch_count()
    ds.attend()
    assert B.hat_launch_count() - before == 1 + drafts + apart
    ds.close()
    _check(sc, cuda_device, repeat=2)
