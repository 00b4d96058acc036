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


@pytest.mark.parametrize("n_bits,n_tables", [(10, 16), (8, 16), (6, 16), (4, 32), (12, 8), (4, 8), (6, 8), (6, 32)])
def test_more_doubtful_keys_than_a_ctas_list_holds(n_bits, n_tables):
    """The segments' lists are shared out over the CTAs of the projection pass: a run of doubtful keys in two
    tiles is longer than the share of the CTAs that meet it, so most of its items are settled by single threads."""
    import torch
    from paper_2602_02199_b200 import binding as Bn
    H, S, nb, W, G = 2, 1000, 3, 32, 2
    gen = torch.Generator(device="cuda").manual_seed(n_bits)
    k = torch.randn(1, H, nb * S, 128, generator=gen, device="cuda")
    planes = torch.randn(n_tables * n_bits, 128, generator=gen, device="cuda")
    for row, dim in ((2 * n_bits, 5), (3 * n_bits - 1, 6)):            # first and last bit of table 2
        planes[row] = 0.0
        planes[row, dim] = -1.0
    first = S + 100
    k[:, 1, first:first + 200, 5:7] = 0.0                              # second head, second block: 200 different keys
    q = torch.randn(1, H * G, W, 128, generator=gen, device="cuda").bfloat16()
    k, planes = k.bfloat16(), planes.bfloat16()
    got, status = Bn.laser_kv_collision_counts(k, q, planes, S, nb, n_bits, n_tables)
    got = to_np(got).astype(np.int64).reshape(H, nb, S)
    pb = to_np(planes.view(torch.int16)).view(np.uint16)
    for h in range(H):
        qb, _ = O.simhash_buckets(to_np(q[0, h * G:(h + 1) * G].reshape(-1, 128).view(torch.int16)).view(np.uint16), pb, n_bits, n_tables)
        kb, _ = O.simhash_buckets(to_np(k[0, h].view(torch.int16)).view(np.uint16), pb, n_bits, n_tables)
        assert (got[h].reshape(-1) == O.collision_counts(qb, kb)).all(), h
    assert int(status.view(torch.int32)[0]) == 0


@pytest.mark.parametrize("n_bits,n_tables", [(8, 16), (10, 16), (4, 32), (6, 32)])
def test_tables_of_zero_hyperplanes(n_bits, n_tables):
    """The scale of the threshold is that of the chunk's first sixteen hyperplanes for every table of the chunk. Where
    those are all zero no sign is doubtful, and another table of zero hyperplanes does not fill the list either."""
    import torch
    from paper_2602_02199_b200 import binding as Bn
    H, S, W, G = 2, 1024, 32, 2
    gen = torch.Generator(device="cuda").manual_seed(60 + n_bits)
    k = torch.randn(1, H, S, 128, generator=gen, device="cuda").bfloat16()
    q = torch.randn(1, H * G, W, 128, generator=gen, device="cuda").bfloat16()
    planes = torch.randn(n_tables, n_bits, 128, generator=gen, device="cuda")
    planes[:-(-16 // n_bits)] = 0.0
    planes[n_tables // 4] = 0.0
    planes = planes.reshape(-1, 128).bfloat16()
    got, status = Bn.laser_kv_collision_counts(k, q, planes, S, 1, n_bits, n_tables)
    got, status = to_np(got).astype(np.int64).reshape(H, S), int(status.view(torch.int32)[0])
    pb = to_np(planes.view(torch.int16)).view(np.uint16)
    for h in range(H):
        qb, _ = O.simhash_buckets(to_np(q[0, h * G:(h + 1) * G].reshape(-1, 128).view(torch.int16)).view(np.uint16), pb, n_bits, n_tables)
        kb, _ = O.simhash_buckets(to_np(k[0, h].view(torch.int16)).view(np.uint16), pb, n_bits, n_tables)
        assert (got[h] == O.collision_counts(qb, kb)).all(), h
    assert status == 0
