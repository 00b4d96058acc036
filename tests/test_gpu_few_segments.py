"""Calls over one or two long segments: every CTA of the log-sum-exp pass contributes to the same
segment, more partials than a warp has lanes, and the score pass that runs beside it has to wait for
all of them. Calls follow one another without a pause and with new keys, so that a partial read too
early is one of other keys."""
import pytest

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("n_kv_heads,block_size", [(1, 16384), (2, 16384), (4, 8192)])
def test_every_partial_is_waited_for(n_kv_heads, block_size):
    import torch
    from paper_2602_02199_b200 import binding as Bn
    gen = torch.Generator(device="cuda").manual_seed(3)
    group, window, calls = 4, 64, 24
    q = torch.randn(1, n_kv_heads * group, window, 128, generator=gen, device="cuda").bfloat16()
    planes = torch.randn(16 * 8, 128, generator=gen, device="cuda").bfloat16()
    # another scale from call to call: the normalisers differ by far more than rounding
    keys = [(torch.randn(1, n_kv_heads, block_size, 128, generator=gen, device="cuda") * (1 + i % 3)).bfloat16() for i in range(calls)]
    eng = Bn.LaserKV(Bn.make_config(n_layers=1, batch=1, n_q_heads=n_kv_heads * group, n_kv_heads=n_kv_heads,
                                    block_size=block_size, window=window, max_blocks=calls, max_blocks_per_call=1, lsh_bits=8,
                                    lsh_tables=16, protection_divisor=4, budget_per_block=512, alpha=1.0), planes)
    got = []
    for k in keys:
        eng.laser_kv_select_block(0, k, k, q, 1)
        got.append(eng.laser_kv_debug_view().s_exact.clone())
    eng.laser_kv_poll_status()
    for k, s in zip(keys, got):
        # the probabilities of every window query sum to one over the block (fp32 sums: a few 1e-6)
        total = s.double().sum(-1) / (group * window)
        assert (total - 1).abs().max().item() < 1e-4
        want = Bn.laser_kv_window_scores(k, q, block_size, 1)
        assert (s.view_as(want) - want).abs().max().item() <= 1e-5 * want.abs().max().item()


@pytest.mark.parametrize("block_size", [64, 128])
def test_every_stationary_operand_is_waited_for(block_size):
    """Blocks of one tile, one block per head, more heads than SMs: the stationary operand changes with
    every tile and each issuing warp works on every second one of them."""
    import torch
    from paper_2602_02199_b200 import binding as Bn
    gen = torch.Generator(device="cuda").manual_seed(4)
    batch, n_kv_heads, group, window = 100, 8, 4, 32
    for i in range(4):
        q = torch.randn(batch, n_kv_heads * group, window, 128, generator=gen, device="cuda").bfloat16()
        k = torch.randn(batch, n_kv_heads, block_size, 128, generator=gen, device="cuda").bfloat16()
        s = Bn.laser_kv_window_scores(k, q, block_size, 1)[:, :, 0]
        logits = torch.einsum("bhgd,bhkd->bhgk", q.double().view(batch, n_kv_heads, group * window, 128), k.double())
        want = torch.softmax(logits / 128 ** 0.5, dim=-1).sum(2)
        assert (s.double() - want).abs().max().item() <= 1e-5 * want.abs().max().item()
