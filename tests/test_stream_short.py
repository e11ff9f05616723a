"""The streaming kernel with a CTA per unit: clusters of 1, 2, 4 and 8 CTAs that share a request, through their shared memory."""
import numpy as np
import pytest

from paper_2503_18989_b200 import binding as B, workloads as W

from common import oracle_replay
from test_stream_kernel import _batch, _check

# beside the longest request ones with fewer pages than a cluster has CTAs (pieces without a page), page edges, 1 to 16 rows
PREFIX = [0, 5, 16, 17, 128]
CHUNK = [1, 16, 3, 8, 9, 4]
FORM = {0: 1, 1: 2, 2: 3, 4: 4, 8: 5}               # HAT_VERIFY_CLUSTER -> hat_plan_info.stream_kernel


def _form(sc):
    st = sc.steps[0]
    c = B.make_cache_desc(sc.cache.dtype, sc.cache.num_pages, sc.cache.num_heads, sc.cache.head_dim, 16 * sc.cache.num_heads * sc.cache.head_dim,
                          sc.cache.head_dim, 16 * sc.cache.head_dim, 1 << 30, 1 << 30)
    cu = np.concatenate([[0], np.cumsum(st.chunk_len)]).astype(np.int32)
    p = B.hat_plan_create(c, st.q.shape[1], cu, st.prefix_len, st.chunk_len, st.block_table, B.HAT_PLAN_HOST_ONLY)
    return B.hat_plan_get_info(p).as_dict()["stream_kernel"]


@pytest.mark.gpu
@pytest.mark.parametrize("dtype,d,layout", [("fp16", 128, "paged"), ("bf16", 128, "contiguous"), ("bf16", 64, "paged"), ("fp16", 64, "contiguous")])
@pytest.mark.parametrize("cluster", [1, 2, 4, 8])
@pytest.mark.parametrize("heads,longest", [(2, 3000), (20, 700)])
def test_clusters_and_pieces_without_pages(cuda_device, dtype, d, layout, heads, longest, cluster, monkeypatch):
    monkeypatch.setenv("HAT_VERIFY_CLUSTER", str(cluster))
    sc = _batch(dtype, heads, d, PREFIX + [longest], CHUNK, 60 + heads, 1, layout)
    assert _form(sc) == FORM[cluster]
    _check(sc, cuda_device, repeat=3)


@pytest.mark.gpu
@pytest.mark.parametrize("dtype,group", [("bf16", 4), ("fp16", 3), ("bf16", 8)])           # up to 4, 3 and 8 slabs; some requests have fewer
@pytest.mark.parametrize("cluster", [1, 2, 4, 8])
def test_slabs_of_grouped_heads_and_trees(cuda_device, dtype, group, cluster, monkeypatch):
    monkeypatch.setenv("HAT_VERIFY_CLUSTER", str(cluster))
    sc = _batch(dtype, 2, 128, PREFIX + [2000], CHUNK, 70 + group, group)
    sc.steps[0].tree_mask = W.random_tree_masks(70 + group, CHUNK)
    assert _form(sc) == FORM[cluster]
    _check(sc, cuda_device, repeat=3)


@pytest.mark.gpu
@pytest.mark.parametrize("dtype,heads,d,prefix", [("fp16", 32, 128, 700), ("bf16", 32, 128, 700), ("fp16", 32, 64, 700), ("fp16", 8, 64, 3000), ("bf16", 8, 64, 3000)])
def test_as_close_to_64_bits_as_the_persistent_kernel(cuda_device, dtype, heads, d, prefix, monkeypatch):
    """The plan's own choice against the persistent kernel's many short pieces, each with a reference maximum of its own.  The weights'
    roundings are the error of `out`: it is to be no larger (0.8 to 0.9 of it was measured).  An lse is rounded to 24 bits in any case."""
    from paper_2503_18989_b200 import runner
    sc = _batch(dtype, heads, d, [prefix], [6], 91)
    _, _, want = oracle_replay(sc)
    off = {}
    for cluster in ("0", None):
        if cluster:
            monkeypatch.setenv("HAT_VERIFY_CLUSTER", cluster)
        else:
            monkeypatch.delenv("HAT_VERIFY_CLUSTER")
        ds = runner.DeviceStep(runner.DeviceCache(sc.cache, sc.k_pool, sc.v_pool, cuda_device), sc.steps[0])
        assert ds.info["stream_kernel"] == 1 and ds.info["max_splits"] > 4 if cluster else ds.info["stream_kernel"] > 2
        ds.attend(fused_append=True)
        out, lse = ds.results()
        off[cluster] = np.linalg.norm(out - want[0][0]) / np.linalg.norm(want[0][0])
        assert np.linalg.norm(lse - want[0][1]) <= 2.0 ** -24 * np.linalg.norm(want[0][1])
        ds.close()
    assert off[None] <= off["0"], off


@pytest.mark.gpu
@pytest.mark.parametrize("dtype", ["fp16", "bf16"])
@pytest.mark.parametrize("cluster", ["1", "4"])
def test_infinite_and_undefined_scores_as_in_the_persistent_kernel(cuda_device, dtype, cluster, monkeypatch):
    """An infinite component of a cached key makes a score +inf or -inf by the sign of q: rows with the former are NaN (lse -inf), rows with
    the latter do without that key; a NaN component makes every row NaN.  In either form alike (of the persistent one, a request in one piece)."""
    from paper_2503_18989_b200 import runner
    sc = _batch(dtype, 4, 128, [700, 200, 300], [4, 3, 5], 95)
    k = sc.k_pool.reshape(-1, 4, 16, 128)
    table, inf = sc.steps[0].block_table, 0x7c00 if dtype == "fp16" else 0x7f80
    k[table[0, 20], 1, 3, 7] = inf
    k[table[0, 33], 2, 0, 9] = inf
    k[table[0, 34], 2, 5, 9] = inf
    k[table[1, 2], 0, 1, 5] = inf | 1                                             # NaN
    got = []
    for c in ("0", cluster):
        monkeypatch.setenv("HAT_VERIFY_CLUSTER", c)
        monkeypatch.setenv("HAT_VERIFY_SPLIT_LEN", "100000" if c == "0" else "0")
        ds = runner.DeviceStep(runner.DeviceCache(sc.cache, sc.k_pool, sc.v_pool, cuda_device), sc.steps[0])
        assert ds.info["stream_kernel"] == FORM[int(c)]
        ds.attend(fused_append=True)
        got.append(ds.results())
        ds.close()
    (o0, l0), (o1, l1) = got
    bad = np.isnan(o0).any(axis=2)
    assert bad[:4, 1:3].any() and not bad[:4, 1:3].all() and bad[4:7, 0].all() and bad.sum() <= 8 + 3
    assert np.array_equal(np.isnan(o0), np.isnan(o1)) and np.array_equal(np.isinf(l0), np.isinf(l1)) and np.array_equal(np.isnan(l0), np.isnan(l1))
    assert np.allclose(o0[~bad], o1[~bad], rtol=0, atol=2e-3) and np.allclose(l0[np.isfinite(l0)], l1[np.isfinite(l0)], rtol=0, atol=1e-5)


def test_batches_of_few_units_get_a_cta_or_a_cluster_each(hat_lib, monkeypatch):
    def form(heads, prefix, dtype="bf16", d=128, group=1, prompts=0):
        return _form(_batch(dtype, heads, d, prefix + [1000] * prompts, [4] * len(prefix) + [256] * prompts, 3, group))
    assert form(32, [200]) == FORM[2] and form(32, [700]) == FORM[4] and form(32, [700], "fp16") == FORM[4]
    assert form(8, [700]) == FORM[8] and form(8, [700], d=64) == FORM[8]      # few heads
    assert form(8, [700], group=4) == FORM[8]                                 # one slab of 16 (row, query head) pairs
    assert form(32, [300] * 9) == FORM[1]                                     # requests that need not be cut
    assert form(40, [3000]) == FORM[0] and form(32, [8000] * 12) == FORM[0]   # more units than CTAs, or as fast in pieces
    # with prompt chunks behind, clusters may take somewhat more, a CTA for each uncut request may not
    uneven = [4066, 3779, 936, 5501, 1210, 1568]
    assert form(40, uneven, "fp16") == FORM[0] and form(40, uneven, "fp16", prompts=3) == FORM[0]
    assert form(40, [1500]) == FORM[0] and form(40, [1500], prompts=3) == FORM[4]
    monkeypatch.setenv("HAT_VERIFY_CLUSTER", "0")
    assert form(32, [700]) == FORM[0]
    monkeypatch.delenv("HAT_VERIFY_CLUSTER")
    monkeypatch.setenv("HAT_VERIFY_SPLIT_LEN", "160")                         # a length asked for is the persistent kernel's
    assert form(32, [700]) == FORM[0]
