"""Branches that ordinary inputs do not reach: a selection whose scores crowd into one value range beside an outlier, or are all
equal, an attention output that is aligned to 16 bytes but not to 32, and keys that are NaN."""
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


@pytest.mark.parametrize("n,lq", [(300, 140), (700, 300), (2000, 300)])
@pytest.mark.parametrize("at", [0, 3, 8, 9, 75, 150, 299])
def test_a_key_that_is_nan(n, lq, at):
    """Wherever it stands, every row of its head is NaN, log-sum-exp and all, and the other head is what it was."""
    from paper_2605_22718_b200 import WorldKV
    Q, K, V = (wd.to_device_bf16(wi.f32_to_bf16_bits(normals(6 + i, (m, 2, 128)))) for i, m in enumerate((lq, n, n)))
    kv = WorldKV(n_layers=1, n_heads=2, tokens_per_frame=8, n_keep=4, pool_slots=1, max_k=1, max_lq=lq, max_splits=4)
    for splits in (1, 0, 3):
        lse = torch.empty((2, 2, lq), dtype=torch.float32, device="cuda")
        want = kv.memory_attention(0, Q, [(K, V)], None, 0, lse_out=lse[0], kv_splits=splits)
        Kn = K.clone()
        Kn[at, 1, 5] = float("nan")
        O = kv.memory_attention(0, Q, [(Kn, V)], None, 0, lse_out=lse[1], kv_splits=splits)
        assert kv.poll_status() == (0, 0)
        assert bool(O[:, 1].isnan().all()) and bool(lse[1, 1].isnan().all()), f"splits {splits}"
        assert torch.equal(O[:, 0], want[:, 0]) and torch.equal(lse[1, 0], lse[0, 0])


@pytest.mark.parametrize("row", [0, 2, 9, 31, 60])
def test_query_retrieval_beside_a_chunk_with_a_nan_key(row):
    """The chunk counts for nothing, the others are ranked as if it were not there."""
    from paper_2605_22718_b200 import WorldKV
    H, T, S, lq = 2, 40, 4, 200
    kv = WorldKV(n_layers=1, n_heads=H, tokens_per_frame=T, n_keep=24, pool_slots=S, max_k=S, max_lq=lq, max_batch=1)
    for c in range(S):
        k, v = (wd.to_device_bf16(wi.f32_to_bf16_bits(normals(20 + 2 * c + i, (1, 3 * T, H * 128)))) for i in (0, 1))
        kv.pool_compress_append(0, 1, k, v, [float(c), 0, 0, 0, 1, 0, 0, 0], chunk_tag=c)
    K = kv.pool[:S * kv.C * H * 256].view(torch.bfloat16).view(S, kv.C, H, 128)
    K[1, row, :, 7] = float("nan")
    Q = wd.to_device_bf16(wi.f32_to_bf16_bits(normals(40, (lq, H, 128))))
    score = torch.empty((S,), dtype=torch.float32, device="cuda")
    slots, n = kv.retrieve_query(0, Q, S, score_out=score)
    assert kv.poll_status() == (0, 0)
    rest = [0, 2, 3]
    lse = torch.logsumexp(torch.einsum("qhd,skhd->shqk", Q.double(), K[rest].double()) / 128 ** 0.5, -1)
    mass = torch.softmax(lse, 0).mean((1, 2))
    got = dict(zip(slots.tolist(), score.tolist()))
    assert got[1] == 0.0
    assert [got[s] for s in rest] == pytest.approx(mass.tolist(), rel=1e-4)
