"""Decode attention whose splits merge by way of global memory, against attention in fp64 over the same cache: ragged last tiles, up to
296 splits, merges in one and in several rounds, strided queries, reference maxima that are raised late. That these shapes take this
route is checked on the host (test_launch_rules.py)."""
import pytest

pytestmark = pytest.mark.gpu

# batch, KV heads, queries per head, block, blocks, softmax scale (0: the usual one); every token is kept
SHAPES = [
    (1, 8, 4, 8456, 2, 0.0),          # 265 tiles, the last of 16 rows, 37 splits
    (1, 2, 2, 6376, 1, 0.0),          # 100 tiles, the last of 40 rows, 34 splits
    (1, 1, 2, 12776, 2, 0.0),         # 400 tiles, 134 splits
    (1, 1, 1, 15128, 4, 6.0),         # 946 tiles, 296 splits; logits hundreds apart
    (1, 10, 8, 6088, 1, 0.0),         # 96 tiles, 29 splits: a merge in two rounds
    (1, 10, 8, 6088, 1, 6.0),
    (2, 16, 7, 4168, 1, 0.0),         # nine splits of seven or eight tiles
    (3, 11, 3, 4232, 1, 0.0),         # eight splits of 33 heads
    (1, 16, 5, 7112, 1, 6.0),         # eighteen splits
    (37, 4, 1, 1000, 1, 0.0),         # two splits of 148 heads
]


def entries(shape):
    return shape[3] * shape[4]


@pytest.mark.parametrize("shape", SHAPES, ids=lambda s: "x".join(map(str, s)))
@pytest.mark.parametrize("strided", [False, True])
def test_against_fp64(shape, strided):
    import torch
    from paper_2602_02199_b200 import binding as Bn
    batch, heads, group, block, blocks, scale = shape
    gen = torch.Generator(device="cuda").manual_seed(heads * 1000 + group)
    n, hq, W = entries(shape), heads * group, 16
    planes = torch.randn(8 * 8, 128, generator=gen, device="cuda").bfloat16()
    eng = Bn.LaserKV(Bn.make_config(n_layers=1, batch=batch, n_q_heads=hq, n_kv_heads=heads, block_size=block, window=W, max_blocks=blocks,
                                    max_blocks_per_call=blocks, lsh_bits=8, lsh_tables=8, protection_divisor=2, budget_per_block=block,
                                    alpha=1.0), planes)
    q = torch.randn(batch, hq, W, 128, generator=gen, device="cuda").bfloat16()
    k, v = (torch.randn(batch, heads, n, 128, generator=gen, device="cuda").bfloat16() for _ in range(2))
    eng.laser_kv_select_block(0, k, v, q, blocks)
    d = q[:, :, W - 1] if strided else q[:, :, 0].contiguous()
    got = [eng.laser_kv_decode_attention(0, d, softmax_scale=scale) for _ in range(3)]
    eng.laser_kv_poll_status()
    assert torch.equal(got[0], got[1]) and torch.equal(got[0], got[2])
    x = torch.einsum("bhgd,bhkd->bhgk", d.double().reshape(batch, heads, group, 128), k.double()) * (scale or 128 ** -0.5)
    want = torch.einsum("bhgk,bhkd->bhgd", torch.softmax(x, -1), v.double()).reshape(batch, hq, 128)
    # a few roundings of 2^-24 in weights and sums; a tile of a split is three steps of accumulators that cut off at 2^-24 of their
    # value, half of it on average; a logit of |x| is rounded at 2^-24 |x| before the exponential and at about that in its sum
    splits = max(1, min(296 // (batch * heads), -(-n // 64) // 3))
    bound = 4e-7 + 1.5 * 2.0 ** -24 * -(-n // 64) / splits + 2.0 ** -23 * float(x.abs().max())
    assert ((got[0].double() - want).norm() / want.norm()).item() <= bound
