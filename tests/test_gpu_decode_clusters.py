"""Decode attention whose splits merge inside a thread-block cluster: one to eight splits, sixteen, and just beyond the sizes
at which they do, against attention in fp64 over the same cache."""
import pytest

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("batch,n_kv_heads,group,entries", [
    (1, 8, 4, 8), (1, 8, 4, 72), (1, 3, 5, 7 * 64), (1, 8, 4, 8 * 64), (1, 8, 4, 9 * 64 + 8), (1, 6, 3, 48 * 64),  # up to eight
    (1, 6, 3, 48 * 64 + 8), (1, 2, 1, 57 * 64), (1, 1, 8, 64 * 64),                                             # sixteen
    (1, 8, 4, 65 * 64), (1, 4, 7, 80 * 64 - 8), (1, 1, 8, 130 * 64), (1, 2, 8, 255 * 64),
    (1, 4, 2, 80 * 64), (5, 8, 4, 9 * 64), (8, 8, 4, 12 * 64), (13, 8, 2, 128), (16, 8, 1, 5 * 64), (20, 8, 3, 200)])  # many heads
def test_against_fp64(batch, n_kv_heads, group, entries):
    import torch
    from paper_2602_02199_b200 import binding as Bn
    gen = torch.Generator(device="cuda").manual_seed(entries)
    hq, W = n_kv_heads * group, 16
    planes = torch.randn(8 * 8, 128, generator=gen, device="cuda").bfloat16()
    eng = Bn.LaserKV(Bn.make_config(n_layers=2, batch=batch, n_q_heads=hq, n_kv_heads=n_kv_heads, block_size=entries, window=W,
                                    max_blocks=1, max_blocks_per_call=1, lsh_bits=8, lsh_tables=8, protection_divisor=2,
                                    budget_per_block=entries, alpha=1.0), planes)
    q = torch.randn(batch, hq, W, 128, generator=gen, device="cuda").bfloat16()
    k, v = (torch.randn(batch, n_kv_heads, entries, 128, generator=gen, device="cuda").bfloat16() for _ in range(2))
    for layer in range(2):                               # the second layer's call starts beside the first one's
        eng.laser_kv_select_block(layer, k if layer else v, v if layer else k, q, 1)
    d = torch.randn(batch, hq, 128, generator=gen, device="cuda").bfloat16()
    got = [eng.laser_kv_decode_attention(layer, d) for layer in (0, 1, 0, 1)]
    eng.laser_kv_poll_status()
    for layer, (kk, vv) in ((0, (v, k)), (1, (k, v))):
        assert torch.equal(got[layer], got[layer + 2])
        w = torch.softmax(torch.einsum("bhgd,bhkd->bhgk", d.double().view(batch, n_kv_heads, group, 128), kk.double()) / 128 ** 0.5, -1)
        want = torch.einsum("bhgk,bhkd->bhgd", w, vv.double()).reshape(batch, hq, 128)
        # fp32 logits, weights and sums: a few roundings of 2^-24 each
        assert ((got[layer].double() - want).norm() / want.norm()).item() <= 4e-7
