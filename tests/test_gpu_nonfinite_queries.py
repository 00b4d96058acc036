"""Window queries with NaN or infinite elements: a projection that is not a number has sign bit 0, as the
comparison with zero gives it, whatever the NaN's own sign; infinite projections keep their sign."""
import numpy as np
import pytest

from oracle import laser_kv_oracle as O

from parity_util import check_signatures, to_np

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("n_bits,n_tables,window", [(8, 16, 32), (10, 8, 64), (5, 24, 16)])
def test_signatures_of_nonfinite_queries(n_bits, n_tables, window):
    import torch
    from paper_2602_02199_b200 import binding as Bn
    G, S = 4, 256
    gen = torch.Generator(device="cuda").manual_seed(n_bits)
    q = torch.randn(1, G, window, 128, generator=gen, device="cuda")
    q[0, 0, 3, 7] = float("nan")
    q[0, 1, 5, 9] = float("inf")
    q[0, 2, 6, 1], q[0, 2, 6, 2] = float("inf"), -float("inf")     # NaN where the two hyperplane elements agree in sign
    q = q.bfloat16()
    k = torch.randn(1, 1, S, 128, generator=gen, device="cuda").bfloat16()
    planes = torch.randn(n_bits * n_tables, 128, generator=gen, device="cuda").bfloat16()
    eng = Bn.LaserKV(Bn.make_config(n_layers=1, batch=1, n_q_heads=G, n_kv_heads=1, block_size=S, window=window, max_blocks=1,
                                    max_blocks_per_call=1, lsh_bits=n_bits, lsh_tables=n_tables, protection_divisor=4,
                                    budget_per_block=64, alpha=0.5, debug=1), planes)
    eng.laser_kv_select_block(0, k, k, q, 1)
    view = eng.laser_kv_debug_view()
    eng.laser_kv_poll_status()
    bits = [to_np(t.view(torch.int16)).view(np.uint16) for t in (k[0, 0], q[0].reshape(-1, 128), planes)]
    with np.errstate(invalid="ignore"):
        proj = O.simhash_projections(bits[1], bits[2]).reshape(-1, n_tables, n_bits)
        assert np.isnan(proj[3]).all() and np.isnan(proj[2 * window + 6]).any() and not np.isnan(proj[window + 5]).any()
        codes = to_np(view.query_buckets)[0, 0]
        # the rows with NaN bit by bit (their difference from zero cannot be compared), the others as usual
        code_bits = max(4, (n_bits + 1) // 2 * 2)
        for row in (3, window + 5, 2 * window + 6):
            got = (codes[row, :n_tables, None].astype(np.int64) >> (code_bits - 1 - np.arange(n_bits))) & 1
            assert (got == (proj[row] >= 0.0)).all(), row
        finite = np.isfinite(proj).all(axis=(1, 2))
        qb, _ = O.simhash_buckets(bits[1], bits[2], n_bits, n_tables)
    check_signatures(codes[finite], bits[1][finite], bits[2], n_bits, n_tables, "finite queries")
    kb, _ = O.simhash_buckets(bits[0], bits[2], n_bits, n_tables)
    assert (to_np(view.counts)[0, 0, 0].astype(np.int64) == O.collision_counts(qb, kb)).all()
