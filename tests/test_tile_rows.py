"""Small prefill batches on the one-CTA tile kernel: units of 128 or 256 rows, as many CTAs as units (whose output rows lanes store
in pairs, and whose two chains store half of the columns each), chunks with an odd last row, ranges of one key tile."""
import pytest

from test_stream_kernel import _batch, _check

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("rows", ["0", "128", "256"])
@pytest.mark.parametrize("dtype", ["fp16", "bf16"])
@pytest.mark.parametrize("prefix,chunk", [(0, 17), (0, 128), (0, 129), (111, 255), (640, 256), (1500, 257), (2000, 33), (900, 385)])
def test_one_request(cuda_device, dtype, prefix, chunk, rows, monkeypatch):
    monkeypatch.setenv("HAT_PREFILL_KERNEL", "tc5")
    monkeypatch.setenv("HAT_PREFILL_TILE_ROWS", rows)
    _check(_batch(dtype, 3, 128, [prefix], [chunk], 11), cuda_device)


@pytest.mark.parametrize("dtype", ["fp16", "bf16"])
@pytest.mark.parametrize("split", ["128", "256", "896"])     # both halves in a cluster, ragged halves, more pieces than two
@pytest.mark.parametrize("prefix,chunk", [(0, 129), (0, 256), (255, 100), (383, 128), (700, 256), (1000, 17), (1663, 300)])
def test_tiles_cut_in_two(cuda_device, dtype, prefix, chunk, split, monkeypatch):
    """Calls follow without a wait, so that a cluster's shared memory is in use when the next one starts."""
    monkeypatch.setenv("HAT_PREFILL_KERNEL", "tc5")
    monkeypatch.setenv("HAT_PREFILL_TILE_ROWS", "128")
    monkeypatch.setenv("HAT_PREFILL_SPLIT_LEN", split)
    _check(_batch(dtype, 5, 128, [prefix], [chunk], 17), cuda_device, repeat=5)


@pytest.mark.parametrize("chunk", [129, 256, 301])
def test_output_in_the_cache_type(cuda_device, chunk):
    import torch
    from paper_2503_18989_b200 import binding as B, runner
    sc = _batch("fp16", 5, 128, [700], [chunk], 13)
    ds = runner.DeviceStep(runner.DeviceCache(sc.cache, sc.k_pool, sc.v_pool, cuda_device), sc.steps[0])
    ds.attend(fused_append=True)
    ds.attend16(fused_append=True)
    torch.cuda.synchronize()
    assert B.hat_last_device_status(ds.plan) == B.HAT_OK
    assert torch.equal(ds.out16.view(torch.float16), ds.out.to(torch.float16))
