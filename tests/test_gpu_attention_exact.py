"""Attention where the result is known to the last bit: a key that outweighs all others by more than fp32 resolves has weight
1, so its V row comes back unchanged wherever the key stands; and a call that writes its output over its queries."""
import numpy as np
import pytest
import torch

import wkinputs as wi
from wkinputs import device as wd

pytestmark = pytest.mark.gpu
SCALE = 1.0 / np.sqrt(128.0)


def bf16(x):
    return wi.f32_to_bf16_bits(np.asarray(x, dtype=np.float32))


def normals(stream, shape):
    return wi.normal_f32(83, wi.STREAM_MISC + stream, np.arange(int(np.prod(shape)), dtype=np.uint64)).reshape(shape)


def context(H, lq):
    from paper_2605_22718_b200 import WorldKV
    return WorldKV(n_layers=1, n_heads=H, tokens_per_frame=8, n_keep=4, pool_slots=1, max_k=1, max_lq=lq, max_splits=8)


# the first tile's ends and the middle of its 32-column groups; the first, middle and last row of later and of short tiles
@pytest.mark.parametrize("n,at", [(390, at) for at in (0, 31, 32, 63, 64, 100, 127, 128, 200, 255, 256, 383, 384, 389)] +
                         [(440, 400), (440, 420), (440, 439), (480, 384), (480, 440), (480, 479)])
def test_dominating_key_returns_its_value_row(n, at):
    """Logits of the key: 43 to 56; of all others: below 7.  480 of them weigh 480 e^-33 < 2^-38 together: nothing beside 1
    in fp32, and far less than half a bf16 step in any output component."""
    H, lq = 2, 300
    q, k = normals(1, (lq, H, 128)), normals(2, (n, H, 128))
    q[:, :, 0] = (16.0 + np.arange(lq) % 17 / 4)[:, None]
    k[:, :, 0] = 0.0
    k[at] = 0.0
    k[at, :, 0] = 31.0
    Q, K, V = (wd.to_device_bf16(bf16(x)) for x in (q, k, normals(3, (n, H, 128))))
    logits = torch.einsum("qhd,khd->hqk", Q.float(), K.float()) * SCALE
    assert float(logits[:, :, at].min()) > 40.0
    logits[:, :, at] = 0.0
    assert float(logits.max()) < 7.0
    kv = context(H, lq)
    for splits in (1, 0, 3):
        O = kv.memory_attention(0, Q, [(K, V)], None, 0, kv_splits=splits)
        assert kv.poll_status() == (0, 0)
        assert torch.equal(O, V[at].expand(lq, H, 128)), f"splits {splits}"


@pytest.mark.parametrize("n,first,second", [(390, 5, 200), (390, 200, 5), (390, 60, 388), (390, 388, 60), (390, 130, 300),
                                            (200, 3, 150), (200, 150, 3), (512, 100, 511), (512, 511, 100), (512, 127, 128)])
def test_largest_weight_of_every_tile_in_short_pieces(n, first, second):
    """Two keys of different tiles share all of the weight, and their V rows no component, so each half of O is one rounded
    product w V.  Both weights are exact but for 2^x (1e-4), hence O is within half a bf16 step (2^-8) of it and 1e-4."""
    H, lq = 2, 300
    q, k, v = normals(7, (lq, H, 128)), normals(8, (n, H, 128)), normals(9, (n, H, 128))
    q[:, :, 0] = (16.0 + np.arange(lq) % 17 / 4)[:, None]
    q[:, :, 1] = q[:, :, 0] - (np.arange(lq) % 7 / 8)[:, None]     # the second logit: up to two natural units below
    k[:, :, :2] = 0.0
    k[[first, second]] = 0.0
    k[first, :, 0] = k[second, :, 1] = 31.0
    v[first, :, 64:] = v[second, :, :64] = 0.0
    Q, K, V = (wd.to_device_bf16(bf16(x)) for x in (q, k, v))
    P = torch.softmax(torch.einsum("qhd,khd->hqk", Q.double(), K.double()) * SCALE, -1)
    want = torch.einsum("hqk,khd->qhd", P, V.double())
    kv = context(H, lq)
    for splits in (1, 0, 2):
        O = kv.memory_attention(0, Q, [(K, V)], None, 0, kv_splits=splits)
        assert kv.poll_status() == (0, 0)
        assert bool(((O.double() - want).abs() <= (2.0 ** -8 + 1e-4) * want.abs() + 1e-12).all()), f"splits {splits}"


@pytest.mark.parametrize("H,lq,n", [(24, 256, 912), (24, 256, 1040), (12, 512, 1000), (36, 256, 1320), (40, 256, 1500), (14, 256, 816),
                                    (43, 256, 1560)])
def test_largest_weights_of_units_just_longer_than_short_pieces(H, lq, n):
    """Units of 11 to 20 tiles are cut, and every tile's largest weight is exact in the pieces.  At logits of deviation 2 the relative
    error of O is then 1.76 to 1.80e-3 (weights below their tile's largest and the output rounded to bf16), and 2.28 to 2.33e-3
    where one maximum stands for a whole unit: the bound lies between."""
    q, k, v = normals(13, (lq, H, 128)), normals(14, (n, H, 128)), normals(15, (n, H, 128))
    Q, K, V = (wd.to_device_bf16(bf16(x)) for x in (2.0 * q, k, v))
    P = torch.softmax(torch.einsum("qhd,khd->hqk", Q.double(), K.double()) * SCALE, -1)
    want = torch.einsum("hqk,khd->qhd", P, V.double())
    kv = context(H, lq)
    O = kv.memory_attention(0, Q, [(K, V)], None, 0).double()
    assert kv.poll_status() == (0, 0)
    assert float((O - want).norm() / want.norm()) < 2.05e-3


@pytest.mark.parametrize("H,lq,seg_rows", [(4, 300, (120,) * 8), (8, 1000, (100,) * 6), (2, 300, (255, 127, 127, 127, 127)), (2, 300, (40,) * 8)])
def test_log_sum_exp_over_short_segments(H, lq, seg_rows):
    """All exponentials of such calls are exact to 2^-22, so the log-sum-exp is off by that, by fp32 sums of at most 80 terms in
    four chains, 2^-19 if all roundings went one way, and by its own rounding: below 2.5e-6 (with a share of cubics 5e-6 to 1e-5)."""
    from paper_2605_22718_b200 import WorldKV
    kv = WorldKV(n_layers=1, n_heads=H, tokens_per_frame=8, n_keep=4, pool_slots=1, max_k=1, max_lq=lq, max_splits=8, max_dense_segments=8)
    q = wd.to_device_bf16(bf16(normals(16, (lq, H, 128))))
    segs = [tuple(wd.to_device_bf16(bf16(normals(17 + 2 * i + j, (n, H, 128)))) for j in (0, 1)) for i, n in enumerate(seg_rows)]
    K = torch.cat([k for k, _ in segs])
    want = torch.logsumexp(torch.einsum("qhd,khd->hqk", q.double(), K.double()) * SCALE, -1)
    for splits in (1, 0):
        lse = torch.empty((H, lq), dtype=torch.float32, device="cuda")
        kv.memory_attention(0, q, segs, None, 0, lse_out=lse, kv_splits=splits)
        assert kv.poll_status() == (0, 0)
        assert float((lse.double() - want).abs().max()) < 2.5e-6, f"splits {splits}"


def test_log_sum_exp_over_short_slots():
    """The same for stored chunks of fewer than 128 rows, beside a long segment and alone."""
    from paper_2605_22718_b200 import WorldKV
    H, T, keep, S, lq = 3, 96, 24, 9, 200
    kv = WorldKV(n_layers=1, n_heads=H, tokens_per_frame=T, n_keep=keep, pool_slots=S, max_k=S, max_lq=lq, max_batch=1)
    for c in range(S):
        x = [wd.to_device_bf16(bf16(normals(40 + 2 * c + j, (1, 3 * T, H * 128)))) for j in (0, 1)]
        kv.pool_compress_append(0, 1, x[0], x[1], [float(c), 0, 0, 0, 1, 0, 0, 0], chunk_tag=c)
    n = S * kv.C
    stored = kv.pool[:n * H * 256].view(torch.bfloat16).view(n, H, 128)
    q, k, v = (wd.to_device_bf16(bf16(normals(60 + i, (m, H, 128)))) for i, m in enumerate((lq, 640, 640)))
    slots = torch.arange(S, dtype=torch.int32, device="cuda")
    for segs in ([], [(k, v)]):
        K = torch.cat([s[0] for s in segs] + [stored])
        want = torch.logsumexp(torch.einsum("qhd,khd->hqk", q.double(), K.double()) * SCALE, -1)
        lse = torch.empty((H, lq), dtype=torch.float32, device="cuda")
        kv.memory_attention(0, q, segs, slots, S, lse_out=lse)
        assert kv.poll_status() == (0, 0)
        assert float((lse.double() - want).abs().max()) < 2.5e-6


@pytest.mark.parametrize("step", [-3, -7, -12, -15, -19, -30, 7, 15, 30])
@pytest.mark.parametrize("n,tile", [(512, 128), (470, 128), (1200, 128), (512, 64), (800, 80), (1200, 80)])
def test_large_values_under_falling_and_rising_logits(n, tile, step):
    """The logits move by `step` log2 units every `tile` keys, in step with the kernel's tiles (64 rows in short calls, 80) or not.  Values scaled by 2^115 are exact in bf16 and leave
    2^12 of fp32's range: O is the unscaled O times 2^115, bit for bit, as long as the sum that O is held against stays below 2^10."""
    H, lq = 2, 140
    q, k, v = normals(10, (lq, H, 128)), normals(11, (n, H, 128)), normals(12, (n, H, 128))
    q[:, :, 0] = 16.0
    k[:, :, 0] = (step * (np.arange(n) // tile) / (16.0 * SCALE * 1.4426950408889634))[:, None]
    Q, K, V = (wd.to_device_bf16(bf16(x)) for x in (q, k, v))
    kv = context(H, lq)
    for splits in (1, 0, 2):
        O = [kv.memory_attention(0, Q, [(K, x)], None, 0, kv_splits=splits) for x in (V, V * 2.0 ** 115)]
        assert kv.poll_status() == (0, 0)
        assert torch.equal(O[0].double() * 2.0 ** 115, O[1].double()), f"splits {splits}"


@pytest.mark.parametrize("rise", [0.0, 100.0])
@pytest.mark.parametrize("H,lq,n", [(2, 300, 700), (12, 880, 300), (40, 1100, 200)])
def test_output_over_the_queries(H, lq, n, rise):
    """O may be Q itself: each (head, query block) is read before it is written.  rise: logits of a few rows grow by that
    much (natural units) from key 150 on."""
    q, k = normals(4, (lq, H, 128)), normals(5, (n, H, 128))
    q[:, :, 0] = 0.0
    for h, r in ((0, 3), (H - 1, lq - 1), (H // 2, 200)):
        q[r, h, 0] = 16.0
    k[:, :, 0] = (rise * (np.arange(n) >= 150))[:, None] / (16.0 * SCALE)
    Q, K, V = (wd.to_device_bf16(bf16(x)) for x in (q, k, normals(6, (n, H, 128))))
    kv = context(H, lq)
    for splits in (1, 0, 3):
        want = kv.memory_attention(0, Q, [(K, V)], None, 0, kv_splits=splits)
        X = Q.clone()
        kv.memory_attention(0, X, [(K, V)], None, 0, O=X, kv_splits=splits)
        assert kv.poll_status() == (0, 0)
        assert torch.equal(X, want), f"splits {splits}"
