"""Key ranges of verification batches with several slabs of 16 (row, query head) pairs per K/V head (host-only plans)."""
import numpy as np
import pytest

from paper_2503_18989_b200 import binding as B


@pytest.mark.parametrize("heads", [1, 2, 7, 8, 16])
@pytest.mark.parametrize("prefix,chunk", [([0], [16]), ([5], [9]), ([8000], [5]), ([60000, 10], [16, 3]), (list(range(100, 8000, 500)), [8] * 16)])
def test_pieces_cover_every_request(hat_lib, heads, prefix, chunk):
    need = [(p + c + 15) // 16 for p, c in zip(prefix, chunk)]
    table, at = np.zeros((len(prefix), max(need)), np.int32), 0
    for i, n in enumerate(need):
        table[i, :n] = np.arange(at, at + n)
        at += n
    desc = B.make_cache_desc("fp16", at, heads, 128, 16 * heads * 128, 128, 16 * 128, 1 << 30, 1 << 30)
    cu = np.concatenate([[0], np.cumsum(chunk)]).astype(np.int32)
    plan = B.hat_plan_create(desc, heads * 4, cu, np.array(prefix, np.int32), np.array(chunk, np.int32), table, flags=1)
    info = B.hat_plan_get_info(plan).as_dict()
    length = info["verify_split_len"]
    assert length >= 96 and length % 16 == 0 and info["max_splits"] <= 32
    # a range length below 1/32 of a request is lengthened for it
    pieces = sum(-(-(p + c) // max(length, -(-(-(-(p + c) // 32)) // 16) * 16)) for p, c in zip(prefix, chunk))
    assert info["num_verify_items"] == pieces
    cut = [c for p, c in zip(prefix, chunk) if p + c > length]
    assert info["num_merge_rows"] == sum(cut) and (info["workspace_bytes"] > 0) == bool(cut)
