"""The streaming kernel with a CTA per unit: clusters of 1, 2, 4 and 8 CTAs that share a request, through their shared memory."""
import pytest

from paper_2503_18989_b200 import workloads as W

from test_stream_kernel import _batch, _check

pytestmark = pytest.mark.gpu

# beside the longest request ones with fewer pages than a cluster has CTAs (pieces without a page), page edges, 1 to 16 rows
PREFIX = [0, 5, 16, 17, 128]
CHUNK = [1, 16, 3, 8, 9, 4]


@pytest.mark.parametrize("dtype,d,layout", [("fp16", 128, "paged"), ("bf16", 128, "contiguous"), ("bf16", 64, "paged")])
@pytest.mark.parametrize("heads,longest", [(2, 3000), (8, 1500), (20, 700), (32, 60)])     # 12, 48, 120 and 192 units: clusters of 8, 4, 2 and 1
def test_clusters_and_pieces_without_pages(cuda_device, dtype, d, layout, heads, longest):
    _check(_batch(dtype, heads, d, PREFIX + [longest], CHUNK, 60 + heads, 1, layout), cuda_device, repeat=3)


@pytest.mark.parametrize("dtype,group", [("bf16", 4), ("fp16", 3), ("bf16", 8)])           # up to 4, 3 and 8 slabs; some requests have fewer
def test_slabs_of_grouped_heads_and_trees(cuda_device, dtype, group):
    sc = _batch(dtype, 2, 128, PREFIX + [2000], CHUNK, 70 + group, group)
    sc.steps[0].tree_mask = W.random_tree_masks(70 + group, CHUNK)
    _check(sc, cuda_device, repeat=3)
