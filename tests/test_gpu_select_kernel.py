"""The selection kernel against the oracle's two-stage rule, bit for bit, at the sizes where its rows of
keys begin and end and on values that strain its radix rounds: wide and narrow ranges, few distinct
values, ties that fill the boundary bin, extremes of the types."""
import numpy as np
import pytest

from oracle import laser_kv_oracle as O

from parity_util import to_np

pytestmark = pytest.mark.gpu


def _values(rng, kind, shape):
    if kind == "equal":
        return np.full(shape, 0.25, np.float32), np.full(shape, 7, np.uint32)
    if kind == "few":
        return rng.integers(0, 3, shape).astype(np.float32) * 1e-3, rng.integers(0, 2, shape).astype(np.uint32)
    if kind == "wide":        # zeros, denormals, negatives, infinities; counts over all 32 bits
        s = (rng.standard_normal(shape) * 10.0 ** rng.integers(-44, 38, shape)).astype(np.float32)
        s[rng.random(shape) < 0.05] = 0.0
        s[rng.random(shape) < 0.01] = np.inf
        s += 0.0                                          # no -0.0
        return np.abs(s) if shape[1] % 16 else s, rng.integers(0, 2 ** 32, shape, dtype=np.uint32)
    s = np.exp(rng.standard_normal(shape)).astype(np.float32) * 1e-2
    return s, rng.poisson(40.0, shape).astype(np.uint32)


def _want(s, c, cand, kept, k_exact, k_lsh):
    exact = O.topk_lower_index(cand, s.astype(np.float64), k_exact)
    resid = np.setdiff1d(cand, exact, assume_unique=True)
    return np.sort(np.concatenate([kept, exact, O.topk_lower_index(resid, c.astype(np.int64), k_lsh)]))


@pytest.mark.parametrize("kind", ["usual", "equal", "few", "wide"])
@pytest.mark.parametrize("n_seg,S", [(3, 8), (2, 1000), (2, 1024), (2, 1025), (2, 2049), (2, 4097), (2, 6145), (1, 8193),
                                     (1, 10241), (1, 16384), (300, 1000), (300, 1032), (300, 2056), (300, 4096)])
def test_rounds_and_ties(kind, n_seg, S):
    import torch
    from paper_2602_02199_b200 import binding as Bn
    rng = np.random.default_rng(S * 7 + n_seg)
    s, c = _values(rng, kind, (n_seg, S))
    a = S // 16
    left = S - 2 * a
    for k_exact, k_lsh in [(left // 4, left // 9), (0, left // 3), (left // 2, 0), (1, 1), (left - 1, 1)]:
        idx = to_np(Bn.laser_kv_two_stage_topk(torch.from_numpy(s).cuda(), torch.from_numpy(c.view(np.int32)).cuda(), a,
                                               k_exact, k_lsh))
        kept = np.concatenate([np.arange(a), np.arange(S - a, S)])
        for i in range(n_seg) if n_seg < 10 else (0, n_seg - 1):
            want = _want(s[i], c[i], np.arange(a, S - a), kept, k_exact, k_lsh)
            assert (idx[i] == want).all(), (kind, i, k_exact, k_lsh)


def test_longest_segment():
    """Look-back with the largest block and half of it held back: 24576 scored keys per segment."""
    import torch
    from paper_2602_02199_b200 import binding as Bn
    S, B, n = 16384, 16384, 2
    gen = torch.Generator(device="cuda").manual_seed(5)
    k, v = (torch.randn(1, 1, 2 * S, 128, generator=gen, device="cuda").bfloat16() for _ in range(2))
    q = torch.randn(1, 1, 32, 128, generator=gen, device="cuda").bfloat16()
    planes = torch.randn(16 * 8, 128, generator=gen, device="cuda").bfloat16()
    eng = Bn.LaserKV(Bn.make_config(n_layers=1, batch=1, n_q_heads=1, n_kv_heads=1, block_size=S, window=32, max_blocks=2,
                                    max_blocks_per_call=1, lsh_bits=8, lsh_tables=16, protection_divisor=n,
                                    budget_per_block=B, alpha=0.75, lookback=1), planes)
    for t in range(2):
        eng.laser_kv_select_block(0, k[:, :, t * S:(t + 1) * S], v[:, :, t * S:(t + 1) * S], q, 1)
    eng.laser_kv_poll_status()
    dbg = eng.laser_kv_debug_view()
    a, _, b_long, k_e, k_l = O.lookback_partition(B, n, 0.75, B // n)
    assert dbg.segment_keys == S + a == 24576
    cand = np.concatenate([np.arange(0, a), np.arange(2 * a, a + S - a)])
    want = _want(to_np(dbg.s_exact)[0, 0, 0], to_np(dbg.counts)[0, 0, 0], cand, np.arange(a, 2 * a), k_e, k_l)
    assert (to_np(dbg.idx)[0, 0, 0][:a + b_long] == want).all()


@pytest.mark.parametrize("n_seg,keep", [(1, 1), (4, 4096), (5, 4096)])
def test_gather_status_of_few_and_many_indices(n_seg, keep):
    """The status word is stored by the gather itself (up to 16384 indices) or cleared before it."""
    import torch
    from paper_2602_02199_b200 import binding as Bn
    rows = 5000
    src = torch.randn(n_seg, rows, 128, device="cuda").bfloat16()
    idx = torch.sort(torch.stack([torch.randperm(rows, device="cuda")[:keep] for _ in range(n_seg)]), dim=1)[0].int()
    k, v = (torch.zeros(n_seg, keep, 128, dtype=torch.bfloat16, device="cuda") for _ in range(2))
    pos = torch.zeros(n_seg, keep, dtype=torch.int32, device="cuda")
    status = torch.full((1,), 99, dtype=torch.int32, device="cuda")
    for bad in (False, True, False):
        use = idx.clone()
        if bad:
            use[n_seg - 1, keep - 1] = rows
        Bn.laser_kv_gather_append(src, src, use, k, v, pos, 0, 0, status)
        assert int(status) == (Bn.ERR_INVALID_ARG if bad else 0)
        if not bad:
            want = torch.gather(src, 1, idx.long()[:, :, None].expand(-1, -1, 128))
            assert torch.equal(k, want) and torch.equal(v, want) and torch.equal(pos, idx)
