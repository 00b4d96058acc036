"""Runs of equal keys with a projection of exactly zero: every one of them is a doubtful sign, all in the
same few tiles. As many as a segment may have are settled exactly; more are reported."""
import numpy as np
import pytest

from oracle import laser_kv_oracle as O

from parity_util import to_np

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("n_equal,first", [(1, 0), (225, 0), (225, 1777), (257, 640)])
def test_run_of_doubtful_keys(n_equal, first):
    import torch
    from paper_2602_02199_b200 import binding as Bn
    # about a dozen of the other (key, table) pairs are doubtful too
    S, K, L, W, G = 2048, 8, 16, 32, 4                         # 2048 * 16 / 256 < 256: the list's smallest capacity
    gen = torch.Generator(device="cuda").manual_seed(9)
    k = torch.randn(1, 1, S, 128, generator=gen, device="cuda")
    planes = torch.randn(L * K, 128, generator=gen, device="cuda")
    planes[11] = 0.0
    planes[11, 5] = 1.0                                        # table 1, bit 3
    odd = torch.randn(128, generator=gen, device="cuda")
    odd[5] = 0.0
    k[:, :, first:first + n_equal] = odd
    q = torch.randn(1, G, W, 128, generator=gen, device="cuda").bfloat16()
    k, planes = k.bfloat16(), planes.bfloat16()
    eng = Bn.LaserKV(Bn.make_config(n_layers=1, batch=1, n_q_heads=G, n_kv_heads=1, block_size=S, window=W, max_blocks=1,
                                    max_blocks_per_call=1, lsh_bits=K, lsh_tables=L, protection_divisor=4,
                                    budget_per_block=512, alpha=0.5, debug=1), planes)
    eng.laser_kv_select_block(0, k, k, q, 1)
    if n_equal > 256:
        with pytest.raises(Bn.LaserKVError) as e:
            eng.laser_kv_poll_status()
        assert e.value.status == Bn.ERR_CAPACITY
        return
    eng.laser_kv_poll_status()
    bits = [to_np(t.view(torch.int16)).view(np.uint16) for t in (k[0, 0], q[0].reshape(-1, 128), planes)]
    kb, _ = O.simhash_buckets(bits[0], bits[2], K, L)
    qb, _ = O.simhash_buckets(bits[1], bits[2], K, L)
    rest = np.setdiff1d(np.arange(S), np.arange(first, first + n_equal))
    counts = to_np(eng.laser_kv_debug_view().counts)[0, 0, 0].astype(np.int64)
    want = O.collision_counts(qb, kb)
    assert (counts[first:first + n_equal] == want[first]).all()
    assert (counts[rest] == want[rest]).all()
