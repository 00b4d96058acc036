"""Decode attention over one to 112 tiles, which merge in clusters of up to eight and of sixteen splits, against fp64
(test_gpu_decode_memory.py has the shapes whose splits merge by way of memory). The numerators keep 24 bits: what is left is the rounding of the
fp32 sums, 1.0e-7 (one tile) to 3.1e-7 of the result's norm over these lengths and six seeds each. Numerators of
two bf16 terms, 2^-17 off at most, would leave 1.3e-6 to 2.4e-6: the bound of 8e-7 tells the two apart."""
import pytest

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("length,n_kv_heads,group", [(8, 1, 8), (512, 2, 4), (520, 2, 4), (1536, 8, 4), (1544, 4, 7), (1736, 8, 1),
                                                     (7104, 8, 4), (7112, 2, 7)])
def test_lengths_around_the_split_rule(length, n_kv_heads, group):
    import torch
    from paper_2602_02199_b200 import binding as Bn
    gen = torch.Generator(device="cuda").manual_seed(length)
    k, v = (torch.randn(1, n_kv_heads, length, 128, generator=gen, device="cuda").bfloat16() for _ in range(2))
    qw = torch.randn(1, n_kv_heads * group, 16, 128, generator=gen, device="cuda").bfloat16()
    planes = torch.randn(64, 128, generator=gen, device="cuda").bfloat16()
    # a budget of the whole block keeps every token: the cache is the input, in order
    eng = Bn.LaserKV(Bn.make_config(n_layers=1, batch=1, n_q_heads=n_kv_heads * group, n_kv_heads=n_kv_heads, block_size=length,
                                    window=16, max_blocks=1, max_blocks_per_call=1, lsh_bits=8, lsh_tables=8,
                                    protection_divisor=2, budget_per_block=length, alpha=1.0), planes)
    eng.laser_kv_select_block(0, k, v, qw, 1)
    q = torch.randn(1, n_kv_heads * group, 128, generator=gen, device="cuda").bfloat16()
    out = eng.laser_kv_decode_attention(0, q).double()
    eng.laser_kv_poll_status()
    w = torch.softmax(torch.einsum("bhgd,bhnd->bhgn", q.double().view(1, n_kv_heads, group, 128), k.double()) / 128 ** 0.5, -1)
    want = torch.einsum("bhgn,bhnd->bhgd", w, v.double()).view(1, n_kv_heads * group, 128)
    assert ((out - want).norm() / want.norm()).item() < 8e-7
