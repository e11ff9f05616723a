"""Which units of a batch the CTA pairs take, and both tile kernels behind one another."""
import numpy as np
import pytest

from paper_2503_18989_b200 import binding as B, workloads as W

from test_stream_kernel import _batch, _check


def _pair_units(prefix, chunk, H, dtype="bf16"):
    rng = np.random.Generator(np.random.PCG64(3))
    table, pages = W._place_pages(rng, np.asarray(prefix) + np.asarray(chunk), slack_pages=2)
    c = B.make_cache_desc(dtype, pages, H, 128, H * 16 * 128, 128, 16 * 128)
    cu = np.concatenate([[0], np.cumsum(chunk)]).astype(np.int32)
    p = B.hat_plan_create(c, H, cu, np.asarray(prefix, np.int32), np.asarray(chunk, np.int32), table, B.HAT_PLAN_HOST_ONLY)
    return B.hat_plan_get_info(p).as_dict()["num_pair_units"]


def test_pairs_take_long_wide_units_of_batches_that_fill_them(hat_lib):
    assert _pair_units([4000] * 4, [512] * 4, 32) == 8 * 32
    assert _pair_units([4000] * 4 + [50, 700], [512] * 4 + [100, 4], 32) == 8 * 32       # narrow units and drafts stay out
    assert _pair_units([4000] * 4, [512] * 4, 8) == 0                                    # few units
    assert _pair_units([500] * 8, [512] * 8, 40) == 0                                    # short ones
    assert _pair_units([4000] * 8, [512] * 8, 40, "fp16") == 0                           # fp16 stays on single CTAs


@pytest.mark.gpu
@pytest.mark.parametrize("kernel", ["mixed", ""])           # wide units on pairs whatever their length; as the plan picks them (none, 8 heads)
def test_wide_and_narrow_units_of_one_batch(cuda_device, kernel, monkeypatch):
    if kernel:
        monkeypatch.setenv("HAT_PREFILL_KERNEL", kernel)
    prefix = [0, 300, 1000, 37, 2000, 640, 90, 1500]
    chunk = [512, 384, 128, 64, 300, 17, 4, 256]
    _check(_batch("bf16", 8, 128, prefix, chunk, 83), cuda_device, repeat=10)


@pytest.mark.gpu
@pytest.mark.parametrize("chunk,prefix", [([256], [1000]), ([129], [0]), ([200, 512], [700, 33])])     # halves merged by clusters; one unit a CTA
def test_small_bf16_batches_on_single_ctas(cuda_device, chunk, prefix):
    _check(_batch("bf16", 8, 128, prefix, chunk, 84), cuda_device, repeat=3)


@pytest.mark.gpu
@pytest.mark.parametrize("dtype", ["fp16", "bf16"])
@pytest.mark.parametrize("heads,chunk,prefix,split", [(25, 256, 200, 256), (25, 129, 300, 384), (40, 77, 700, 640), (37, 128, 383, 256)])
def test_halves_of_64_columns(cuda_device, dtype, heads, chunk, prefix, split, monkeypatch):
    """From half a round of CTAs on, clusters merge rows of 64 columns too; calls follow without a wait, and out16 is out rounded once."""
    import torch
    from paper_2503_18989_b200 import runner
    monkeypatch.setenv("HAT_PREFILL_KERNEL", "tc5")
    monkeypatch.setenv("HAT_PREFILL_TILE_ROWS", "128")
    monkeypatch.setenv("HAT_PREFILL_SPLIT_LEN", str(split))
    sc = _batch(dtype, heads, 64, [prefix], [chunk], 19)
    ds = runner.DeviceStep(runner.DeviceCache(sc.cache, sc.k_pool, sc.v_pool, cuda_device), sc.steps[0])
    assert ds.info["max_splits"] == 2 and ds.workspace_bytes == 0           # the clusters need none
    ds.attend(fused_append=True)
    ds.attend16(fused_append=True)
    torch.cuda.synchronize()
    kind = torch.float16 if dtype == "fp16" else torch.bfloat16
    assert torch.equal(ds.out16.view(kind), ds.out.to(kind))
    ds.close()
    _check(sc, cuda_device, repeat=5)


@pytest.mark.gpu
@pytest.mark.parametrize("dtype,d,heads,split", [("fp16", 128, 25, None), ("bf16", 64, 40, None), ("bf16", 128, 32, None), ("bf16", 128, 40, None),      # as planned
                                                 ("fp16", 128, 25, 384), ("fp16", 64, 16, 384)])       # pieces behind a merge launch
def test_uneven_units_longest_first(cuda_device, dtype, d, heads, split, monkeypatch):
    """One to four rounds of units of very different length, in batches whose units the plan puts in an order of its own (3 to 14 % sooner by
    its model), with heads that come in fours (the order is found on a quarter of them) and not."""
    from paper_2503_18989_b200 import runner
    monkeypatch.setenv("HAT_PREFILL_KERNEL", "tc5")
    if split:
        monkeypatch.setenv("HAT_PREFILL_SPLIT_LEN", str(split))
    sc = _batch(dtype, heads, d, [0, 1200, 40, 700, 5, 300, 2000], [300, 17, 513, 129, 64, 3, 40], 23)
    ds = runner.DeviceStep(runner.DeviceCache(sc.cache, sc.k_pool, sc.v_pool, cuda_device), sc.steps[0])
    assert 148 < ds.info["num_prefill_items"] * heads <= 4 * 148 and ds.info["prefill_kernel"] == 1
    ds.close()
    _check(sc, cuda_device, repeat=4)
