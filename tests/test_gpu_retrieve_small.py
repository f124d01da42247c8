"""Pose retrieval at the sizes where the one-pass kernel's thread layout changes, with ties, holes, NaN poses and a pose
table that is only 4-byte aligned, against the fp64 oracle (order and slots exact)."""
import numpy as np
import pytest
import torch

import wkinputs as wi
from oracle import worldkv_oracle as o

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("n", [1, 2, 31, 32, 33, 64, 65, 129, 250, 256, 257, 511, 513, 1000, 1023, 1024, 1025])
@pytest.mark.parametrize("offset", [0, 1])
def test_slot_tables_of_every_layout(n, offset):
    from paper_2605_22718_b200 import retrieve_noalloc
    poses = wi.random_poses(100 + n, n + 1)
    cur = poses[n]
    poses = poses[:n].copy()
    if n > 8:
        poses[5] = poses[3]                      # equal distances: the lower slot first
        poses[n - 1] = poses[3]
        poses[7, 4] = np.nan                     # not a candidate
    valid = np.ones(n, dtype=np.int32)
    valid[4::7] = 0
    max_k = min(n, 64) + 3
    buf = torch.zeros(n * 8 + 4, dtype=torch.float32, device="cuda")
    table = buf[offset:offset + n * 8].view(n, 8)
    table.copy_(torch.from_numpy(poses))
    slots = torch.full((max_k,), -7, dtype=torch.int32, device="cuda")
    dist = torch.full((max_k,), -7.0, dtype=torch.float64, device="cuda")
    ok = [i for i in range(n) if valid[i] and np.isfinite(poses[i]).all()]
    d = o.retrieval_distances(cur, poses[ok])
    order = sorted(range(len(ok)), key=lambda j: (d[j], ok[j]))
    for k in {0, 1, min(n, 64), max_k}:
        retrieve_noalloc(table, torch.from_numpy(valid).cuda(), cur, k, max_k, slots, dist)
        want = order[:min(k, len(ok))]
        got = slots.cpu().numpy()
        np.testing.assert_array_equal(got[:len(want)], [ok[j] for j in want])
        assert (got[len(want):] == -1).all()
        np.testing.assert_allclose(dist.cpu().numpy()[:len(want)], [d[j] for j in want], rtol=1e-12, atol=1e-14)
