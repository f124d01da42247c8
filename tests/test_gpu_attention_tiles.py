"""Memory attention at the edges of its KV tiles: short tiles run over ceil(rows / 16) * 16 keys only, in dense segments,
in pool slots and at the end of a split range."""
import numpy as np
import pytest
import torch

import wkinputs as wi
from wkinputs import device as wd
from oracle import worldkv_oracle as o
from wk_testlib import Scenario, assert_attention_close

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("seg_rows", [(1,), (15, 16), (17, 31), (32, 33), (63, 64, 65), (96, 97), (112, 127), (128,), (129, 1, 144),
                                      (255, 256, 257), (79, 80), (81, 159, 160), (161,), (512,), (513,), (480, 33), (720, 40, 641), (190, 256, 191, 161), (513, 512)])
@pytest.mark.parametrize("lq", [1, 129, 300])
def test_short_tiles_of_dense_segments(seg_rows, lq):
    from paper_2605_22718_b200 import WorldKV
    H = 2
    kv = WorldKV(n_layers=1, n_heads=H, tokens_per_frame=8, n_keep=4, pool_slots=1, max_k=1, max_lq=lq, max_splits=4)
    segs_d, segs_h = [], []
    for i, n in enumerate(seg_rows):
        K = wi.query_bf16(41, 0, i, 1, n, H * 128).reshape(n, H, 128)
        V = wi.query_bf16(42, 0, i, 2, n, H * 128).reshape(n, H, 128)
        segs_d.append((wd.to_device_bf16(K), wd.to_device_bf16(V)))
        segs_h.append((K, V))
    Qb = wi.query_bf16(43, 0, 0, 0, lq, H * 128).reshape(lq, H, 128)
    Q = wd.to_device_bf16(Qb)
    O_ref, L_ref = o.memory_attention(Qb, segs_h, o.PoolModel(n_slots=1, n_layers=1), 0, [])
    for splits in (0, 1, 3):
        lse = torch.empty((H, lq), dtype=torch.float32, device="cuda")
        O = kv.memory_attention(0, Q, segs_d, None, 0, lse_out=lse, kv_splits=splits)
        assert kv.poll_status() == (0, 0)
        assert_attention_close(O, O_ref, f"{seg_rows} lq={lq} splits={splits}")
        np.testing.assert_allclose(lse.cpu().numpy(), L_ref, atol=2e-3)


@pytest.mark.parametrize("T,n_keep", [(9, 1), (40, 24), (100, 27), (100, 28), (100, 29), (150, 40), (200, 56), (200, 57)])
def test_short_tiles_of_pool_slots(T, n_keep):
    """C = T + n_keep stored rows per chunk: 10, 64, 127, 128, 129, 190, 256 (tiled in 64 rows), 257."""
    from paper_2605_22718_b200 import WorldKV
    H, S, lq = 3, 6, 140
    kv = WorldKV(n_layers=1, n_heads=H, tokens_per_frame=T, n_keep=n_keep, pool_slots=S, max_k=S, max_batch=1, max_lq=lq,
                 max_splits=4)
    sc = Scenario(kv, 51, 0.1, 1, T, H, n_keep, S)
    poses = wi.random_poses(51, S)
    for c in range(S):
        sc.append_chunk(c, poses[c])
    Qb = wi.query_bf16(51, 0, 0, 0, lq, H * 128)
    Q = wd.to_device_bf16(Qb).view(lq, H, 128)
    seg_d, seg_h = sc.dense_segment(0, 9, min(3 * T, 83))
    ids = [3, 0, 5, 1]
    slots = torch.tensor(ids, dtype=torch.int32, device="cuda")
    O_ref, L_ref = o.memory_attention(Qb.reshape(lq, H, 128), [seg_h], sc.pool, 0, ids)
    for splits in (0, 1, 4):
        lse = torch.empty((H, lq), dtype=torch.float32, device="cuda")
        O = kv.memory_attention(0, Q, [seg_d], slots, len(ids), lse_out=lse, kv_splits=splits)
        assert kv.poll_status() == (0, 0)
        assert_attention_close(O, O_ref, f"C={T + n_keep} splits={splits}")
        np.testing.assert_allclose(lse.cpu().numpy(), L_ref, atol=2e-3)


@pytest.mark.parametrize("H,lq,rows,cut", [
    (1, 100, 4500, True),      # one unit in 12 pieces of five tiles
    (1, 100, 12000, True),     # one unit in as many pieces as a unit may have
    (7, 256, 2000, True),      # 7 units, every one cut into equal parts, one piece per CTA
    (9, 2000, 900, False),     # 72 units, not cut
    (10, 2048, 3600, True),    # 80 units of 45 tiles: a range per SM, most of them over the end of a unit
    (19, 2048, 1000, True),    # 152 units: one whole wave, the four others in equal parts
    (20, 2100, 640, False),    # 180 units: one whole wave and whole units behind it
    (29, 2048, 4000, True),    # 232 units: whole units and a range that crosses units on the same CTA
])
def test_work_distributions(H, lq, rows, cut):
    """The default distribution over the SMs (whole units, aligned cuts, ranges across units) against one CTA per unit,
    and one head against the oracle."""
    from paper_2605_22718_b200 import WorldKV
    kv = WorldKV(n_layers=1, n_heads=H, tokens_per_frame=8, n_keep=4, pool_slots=1, max_k=1, max_lq=lq)
    D = H * 128
    K = wi.query_bf16(61, 0, 0, 1, rows, D).reshape(rows, H, 128)
    V = wi.query_bf16(62, 0, 0, 2, rows, D).reshape(rows, H, 128)
    Qb = wi.query_bf16(63, 0, 0, 0, lq, D).reshape(lq, H, 128)
    Q, seg = wd.to_device_bf16(Qb), (wd.to_device_bf16(K), wd.to_device_bf16(V))
    out = {}
    for splits in (0, 1):
        lse = torch.empty((H, lq), dtype=torch.float32, device="cuda")
        launches = kv.launch_count()
        out[splits] = kv.memory_attention(0, Q, [seg], None, 0, lse_out=lse, kv_splits=splits).clone(), lse
        if torch.cuda.get_device_properties(0).multi_processor_count == 148:   # the sizes above are for that many
            assert kv.launch_count() - launches == (2 if cut and splits == 0 else 1)   # a second one merges pieces
        assert kv.poll_status() == (0, 0)
    # the two differ by one bf16 rounding of the output and the fp32 merge
    a, b = out[0][0].float(), out[1][0].float()
    assert float((a - b).norm() / b.norm()) < 4e-3
    assert float((out[0][1] - out[1][1]).abs().max()) < 1e-3
    h = H - 1
    O_ref, L_ref = o.memory_attention(Qb[:, h:h + 1], [(K[:, h:h + 1], V[:, h:h + 1])], o.PoolModel(n_slots=1, n_layers=1), 0, [])
    assert_attention_close(out[0][0][:, h:h + 1], O_ref, f"H={H}")
    np.testing.assert_allclose(out[0][1][h:h + 1].cpu().numpy(), L_ref, atol=2e-3)
