"""The streaming kernel where its tiling can go wrong: page and chunk edges, 8- and 16-row tiles, ring wrap-around with
several units per CTA, pieces and their merge, and batches whose pages are shared between a writer and a reader."""
import numpy as np
import pytest

from oracle import hat_oracle as O
from paper_2503_18989_b200 import workloads as W

from common import assert_parity, oracle_replay

pytestmark = pytest.mark.gpu


@pytest.fixture(autouse=True)
def _persistent(monkeypatch):
    monkeypatch.setenv("HAT_VERIFY_CLUSTER", "0")        # the short form is test_stream_short's


def _batch(dtype, H, d, prefix, chunk, seed, group=1, layout="paged", table=None, num_pages=None):
    rng = np.random.Generator(np.random.PCG64(seed))
    if table is None:
        table, num_pages = W._place_pages(rng, np.asarray(prefix) + np.asarray(chunk), slack_pages=5)
    st = W._make_step(seed + 100, dtype, H, d, prefix, chunk, table, q_heads=H * group)
    return W._scenario("stream", dtype, H, d, layout, num_pages, [st], seed + 100)


def _check(sc, device, repeat=1):
    """Every element and both pools, append fused and separate, the same bits either way and every time."""
    from paper_2503_18989_b200 import binding as B, runner
    kp, vp, want = oracle_replay(sc)
    first = None
    for fused in (True, False):
        cache = runner.DeviceCache(sc.cache, sc.k_pool, sc.v_pool, device)
        ds = runner.DeviceStep(cache, sc.steps[0])
        if not fused:
            ds.append()
        for _ in range(repeat):
            ds.attend(fused_append=fused)
        out, lse = ds.results()
        assert B.hat_last_device_status(ds.plan) == B.HAT_OK and ds.canaries_intact()
        assert_parity(out, want[0][0], "out")
        assert_parity(lse, want[0][1], "lse")
        gk, gv = cache.pools_to_host()
        assert np.array_equal(gk, kp) and np.array_equal(gv, vp)
        if first is None:
            first = (out, lse)
        assert np.array_equal(out, first[0]) and np.array_equal(lse, first[1])
        ds.close()


@pytest.mark.parametrize("dtype,d,layout", [("fp16", 128, "paged"), ("bf16", 128, "contiguous"), ("bf16", 64, "paged")])
@pytest.mark.parametrize("group", [1, 3, 8])          # 16-pair slabs: one, up to three, up to eight
def test_edges_of_pages_and_chunks(cuda_device, dtype, d, layout, group):
    prefix = [0, 0, 1, 15, 16, 17, 31, 32, 63, 64, 65, 127, 200, 511]
    chunk = [1, 16, 15, 1, 16, 2, 8, 9, 4, 16, 7, 1, 16, 3]
    _check(_batch(dtype, 2, d, prefix, chunk, 7 + group, group, layout), cuda_device)


@pytest.mark.parametrize("split", [16, 112, 160, 704, 100000])   # pieces of one page (32 at most), odd numbers of pages, uncut
def test_pieces_and_their_merge(cuda_device, split, monkeypatch):
    monkeypatch.setenv("HAT_VERIFY_SPLIT_LEN", str(split))
    _check(_batch("fp16", 3, 128, [703, 16, 0, 2500, 350], [4, 16, 3, 9, 1], 31), cuda_device, repeat=2)


@pytest.mark.parametrize("dtype", ["fp16", "bf16"])
def test_many_units_per_cta_back_to_back(cuda_device, dtype):
    """More units than CTAs and lengths of 1 to 60 pages, so that rings wrap and warps drift apart; repeated without a
    wait between the calls."""
    rng = np.random.default_rng(3)
    prefix = rng.integers(0, 950, size=60).tolist()
    chunk = rng.integers(1, 9, size=60).tolist()
    _check(_batch(dtype, 16, 128, prefix, chunk, 41), cuda_device, repeat=40)


@pytest.mark.parametrize("chunk", [[4, 5], [4, 40]])
def test_a_page_written_by_one_request_and_read_by_another(cuda_device, chunk):
    """Request 1's prefix contains the page request 0 appends to: it must see the appended rows."""
    table = np.asarray([[0, 1, 2, -1, -1, -1], [3, 2, 4, 5, 6, 7]], np.int32)        # page 2: chunk of 0, prefix of 1
    sc = _batch("fp16", 2, 128, [34, 50], chunk, 51, table=table, num_pages=9)
    kp, vp = sc.k_pool.copy(), sc.v_pool.copy()
    O.kv_append(sc.cache, kp, vp, sc.steps[0])
    _check(sc, cuda_device)
