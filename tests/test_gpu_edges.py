"""Branches that ordinary inputs do not reach: a selection whose scores crowd into one value range beside an outlier, or are all
equal, and an attention output that is aligned to 16 bytes but not to 32."""
import numpy as np
import pytest
import torch

import wkinputs as wi
from wkinputs import device as wd
from oracle import worldkv_oracle as o

pytestmark = pytest.mark.gpu


def normals(stream, shape):
    return wi.normal_f32(91, wi.STREAM_MISC + stream, np.arange(int(np.prod(shape)), dtype=np.uint64)).reshape(shape)


@pytest.mark.parametrize("T,n_keep", [(100, 60), (500, 1), (500, 500), (500, 998)])
@pytest.mark.parametrize("spread", [0.02, 0.0])
def test_selection_of_crowded_scores(T, n_keep, spread):
    """spread 0.02: all scores but one within a few percent of their range (the keys are one vector and noise, one is its negative);
    0: all equal but that one, so the lowest indices are kept after it."""
    from paper_2605_22718_b200 import WorldKV
    D = 256
    k = normals(1, (1, D)) + spread * normals(2, (3 * T, D))
    k[T + T // 3] = -k[0]
    K = wi.f32_to_bf16_bits(k.astype(np.float32))
    kv = WorldKV(n_layers=1, n_heads=2, tokens_per_frame=T, n_keep=n_keep, pool_slots=1, max_k=1)
    keep = kv.compress_chunk(wd.to_device_bf16(K[None]))
    assert kv.poll_status() == (0, 0)
    np.testing.assert_array_equal(keep.cpu().numpy()[0], o.compress_chunk(K, T, n_keep)[0])


@pytest.mark.parametrize("n", [300, 700])
def test_output_aligned_to_16_bytes(n):
    from paper_2605_22718_b200 import WorldKV
    H, lq = 2, 300
    Q, K, V = (wd.to_device_bf16(wi.f32_to_bf16_bits(normals(3 + i, (m, H, 128)))) for i, m in enumerate((lq, n, n)))
    kv = WorldKV(n_layers=1, n_heads=H, tokens_per_frame=8, n_keep=4, pool_slots=1, max_k=1, max_lq=lq)
    want = kv.memory_attention(0, Q, [(K, V)], None, 0, kv_splits=1)
    buf = torch.zeros(lq * H * 128 + 16, dtype=torch.bfloat16, device="cuda")
    O = buf[8:8 + lq * H * 128].view(lq, H, 128)
    assert O.data_ptr() % 32 == 16
    kv.memory_attention(0, Q, [(K, V)], None, 0, O=O, kv_splits=1)
    assert kv.poll_status() == (0, 0)
    assert torch.equal(O, want) and not buf[:8].any() and not buf[-8:].any()
