"""Calls issued back to back on one stream, each of which reads what the one before has just written (slot marks and poses,
retrieved slot ids, stored rows): the kernels are launched under the end of their predecessors, and the results must be those of
calls with a wait between them."""
import pytest
import torch

import wkinputs as wi
from wkinputs import device as wd

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("H,T,slots", [(1, 8, 3), (2, 40, 9), (12, 97, 4)])
def test_back_to_back_calls_see_each_other(H, T, slots):
    from paper_2605_22718_b200 import WorldKV
    D, k, rounds = H * 128, 3, 40
    poses = wi.loop_poses(11, rounds)
    K = [wd.to_device_bf16(wi.key_chunk_bf16(6, 0, c, T, D, 0.1))[None] for c in range(4)]
    V = [wd.to_device_bf16(wi.value_chunk_bf16(6, 0, c, T, D))[None] for c in range(4)]
    Q = V[0][0, :2 * T].reshape(2 * T, H, 128)

    def program(wait):
        kv = WorldKV(n_layers=1, n_heads=H, tokens_per_frame=T, n_keep=T // 2, pool_slots=slots, max_k=k, max_lq=2 * T)
        ids = torch.full((rounds, k), -7, dtype=torch.int32, device="cuda")
        dist = torch.zeros((rounds, k), dtype=torch.float64, device="cuda")
        O = torch.zeros((rounds, 2 * T, H, 128), dtype=torch.bfloat16, device="cuda")
        ranked = torch.full((rounds, k), -7, dtype=torch.int32, device="cuda")
        torch.cuda.synchronize()
        for r in range(rounds):
            kv.pool_compress_append(0, 1, K[r % 4], V[(r + 1) % 4], poses[r], chunk_tag=r, evict_oldest_if_full=True)
            wait()
            _, n = kv.retrieve(poses[(7 * r) % rounds], k, slots_out=ids[r], dist_out=dist[r])
            wait()
            kv.memory_attention(0, Q, [], ids[r], n, O=O[r])
            wait()
            kv.retrieve_query(0, Q, k, slots_out=ranked[r])
            wait()
        assert kv.poll_status() == (0, 0)
        return ids, dist, O, ranked, kv.pool

    for a, b in zip(program(lambda: None), program(torch.cuda.synchronize)):
        assert torch.equal(a, b)
