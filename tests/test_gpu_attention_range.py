"""Memory attention where logits leave the range in which a tile is streamed without a look at its maximum (a weight above
2^8 against the row's reference): such a tile is streamed again against its maximum.  Values scaled by a power of two (exact in
bf16) are compared after scaling back, so the tolerance is the usual one."""
import numpy as np
import pytest
import torch

import wkinputs as wi
from wkinputs import device as wd
from oracle import worldkv_oracle as o
from wk_testlib import assert_attention_close

pytestmark = pytest.mark.gpu
LOG2E = 1.4426950408889634
SCALE = 1.0 / np.sqrt(128.0)


def bf16(x):
    return wi.f32_to_bf16_bits(np.asarray(x, dtype=np.float32))


def normals(stream, shape):
    return wi.normal_f32(71, wi.STREAM_MISC + stream, np.arange(int(np.prod(shape)), dtype=np.uint64)).reshape(shape)


def run(H, lq, seg_rows, start, shift, moved, v_exp=0, splits_list=(1, 0, 3)):
    """moved: (head, row) pairs or None for all.  The first component of the moved queries is 16, of the others 0; that of
    a key makes 16 times it `start` log2 units, from key 40 of a segment on `start + shift`."""
    from paper_2605_22718_b200 import WorldKV
    kv = WorldKV(n_layers=1, n_heads=H, tokens_per_frame=8, n_keep=4, pool_slots=1, max_k=1, max_lq=lq, max_splits=8)
    q = normals(1, (lq, H, 128))
    q[:, :, 0] = 16.0 if moved is None else 0.0
    for h, r in moved or []:
        q[r, h, 0] = 16.0
    segs_h = []
    for i, n in enumerate(seg_rows):
        k = normals(10 + i, (n, H, 128))
        k[:, :, 0] = (start + shift * (np.arange(n) >= 40))[:, None] / (16.0 * SCALE * LOG2E)
        segs_h.append((bf16(k), bf16(np.ldexp(normals(20 + i, (n, H, 128)), v_exp))))
    Qb = bf16(q)
    O_ref, L_ref = o.memory_attention(Qb, segs_h, o.PoolModel(n_slots=1, n_layers=1), 0, [])
    segs_d = [(wd.to_device_bf16(k), wd.to_device_bf16(v)) for k, v in segs_h]
    Q = wd.to_device_bf16(Qb)
    for splits in splits_list:
        lse = torch.empty((H, lq), dtype=torch.float32, device="cuda")
        O = kv.memory_attention(0, Q, segs_d, None, 0, lse_out=lse, kv_splits=splits)
        assert kv.poll_status() == (0, 0)
        assert_attention_close(O.double() * 2.0 ** -v_exp, np.ldexp(O_ref, -v_exp),
                               f"start {start} shift {shift} v_exp {v_exp} splits {splits}")
        np.testing.assert_allclose(lse.cpu().numpy(), L_ref, rtol=2e-6, atol=2e-3)


@pytest.mark.parametrize("shift", [0, 40, 76, 84, 92, 100, 108, 112, 116, 120, 124, 130, 300, -300])
@pytest.mark.parametrize("start", [0, -250, 250])
def test_all_logits_moved(start, shift):
    run(2, 140, (300, 17), start, shift, None)


@pytest.mark.parametrize("shift,v_exp", [(0, 110), (0, -100), (60, 60), (60, 90), (60, -100), (-60, 90), (-60, -100)])
def test_large_and_small_values(shift, v_exp):
    run(1, 130, (300,), 0, shift, None, v_exp=v_exp)


@pytest.mark.parametrize("H,lq,rows", [(1, 256, 2000), (9, 2000, 900), (10, 2048, 3600), (20, 2100, 640)])
@pytest.mark.parametrize("shift", [90, 200])
def test_a_few_rows_moved(H, lq, rows, shift):
    """One row in the first Q tile of a pair, one in the last ragged one, one in a second tile: the other units of the CTAs that
    hold them, and all other CTAs, go on as before."""
    run(H, lq, (rows,), 0, shift, [(0, 3), (H - 1, lq - 1), (H // 2, 200)], splits_list=(0,))
