"""wk_pool_compress_append at every row width and retention at which its kernels differ: the pool bytes, slot table and
keep-sets must equal those of wk_compress_chunk + wk_pool_append (whose keep-sets other tests hold against the oracle)."""
import numpy as np
import pytest
import torch

import wkinputs as wi
from wkinputs import device as wd

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("T,H,n_keep,L,per_head", [
    (33, 1, 16, 3, False),     # one column group per lane
    (32, 12, 16, 2, False),    # 1,536 columns, whole blocks of stored rows
    (31, 13, 30, 3, False),    # 1,664 columns: two warps per row, lanes without a column group
    (40, 16, 9, 2, False),     # 2,048 columns
    (45, 20, 44, 3, False),    # wide rows: both passes in one launch, rows stored from the staging buffer
    (65, 40, 32, 2, False),    # 5,120 columns
    (7, 40, 3, 5, False),      # groups of fewer than four rows
    (9, 65, 5, 2, False),      # rows of more than 8,192 columns: an anchor pass of their own
    (20, 72, 7, 3, False),
    (20, 3, 0, 2, False),      # nothing kept but the anchor: no scoring pass
    (20, 24, 40, 2, False),    # everything kept
    (50, 12, 25, 2, True),
    (37, 5, 18, 3, True),
    (20, 3, 0, 2, True),
])
def test_one_call_equals_two(T, H, n_keep, L, per_head):
    from paper_2605_22718_b200 import WorldKV, SCORE_PER_HEAD
    D, S = H * 128, 2
    kw = dict(n_layers=L, n_heads=H, tokens_per_frame=T, n_keep=n_keep, pool_slots=S, max_k=S, max_batch=L,
              score_mode=SCORE_PER_HEAD if per_head else 0)
    a, b = WorldKV(**kw), WorldKV(**kw)
    poses = wi.random_poses(7, 5)
    used = 2 * ((L * S * (T + n_keep) * D * 2 + 255) // 256 * 256)
    for c in range(4):      # fills the pool, then replaces the oldest chunk twice
        K = wd.to_device_bf16(np.stack([wi.key_chunk_bf16(3, l, c, T, D, 0.1) for l in range(L)]))
        V = wd.to_device_bf16(np.stack([wi.value_chunk_bf16(3, l, c, T, D) for l in range(L)]))
        slot, evicted, keep = a.pool_compress_append(0, L, K, V, poses[c], chunk_tag=c, evict_oldest_if_full=True)
        keep2 = b.compress_chunk(K)
        if c >= S:
            b.pool_evict(b.pool_oldest())
        assert b.pool_append(0, L, K, V, keep2, poses[c], chunk_tag=c) == slot == c % S
        assert evicted == (slot if c >= S else -1)
        assert torch.equal(keep, keep2)
        assert torch.equal(a.pool[:used], b.pool[:used])
        assert a.pool_count() == b.pool_count() and a.pool_tag(slot) == c
        assert torch.equal(a.retrieve(poses[4], S)[0], b.retrieve(poses[4], S)[0])
    assert a.poll_status() == (0, 0) and b.poll_status() == (0, 0)
    # the whole pool buffer: slot poses and validity flags as well
    assert torch.equal(a.pool, b.pool)


@pytest.mark.parametrize("T", [1385, 1400, 1414, 1445, 1446])
@pytest.mark.parametrize("H,per_head", [(1, False), (17, False), (1, True)])
def test_selection_space_around_48_kilobytes(T, H, per_head):
    """2 T scores take 17 bytes each in the selection's shared memory: just below 48 KB the kernel's static arrays push a
    launch over the default limit."""
    from paper_2605_22718_b200 import WorldKV, SCORE_PER_HEAD
    from oracle import worldkv_oracle as o
    D, n_keep = H * 128, T // 2
    kv = WorldKV(n_layers=1, n_heads=H, tokens_per_frame=T, n_keep=n_keep, pool_slots=1, max_k=1,
                 score_mode=SCORE_PER_HEAD if per_head else 0)
    bits = wi.key_chunk_bf16(4, 0, 1, T, D, 0.1)
    keep = kv.compress_chunk(wd.to_device_bf16(bits)[None]).cpu().numpy()[0]
    assert kv.poll_status() == (0, 0)
    if per_head:
        np.testing.assert_array_equal(keep, o.compress_chunk_per_head(bits, T, n_keep, H)[0])
    else:
        np.testing.assert_array_equal(keep, o.compress_chunk(bits, T, n_keep)[0])
