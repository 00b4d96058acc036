"""Calls of one stage only, whose first streaming pass starts beside whatever is ahead in the stream: queued back to back, behind
kernels that write their keys and queries or directly behind one another (then beside the append of the call before, which
itself may wait beside its selection), they give what each gives alone."""
import pytest

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("alpha", [0.0, 1.0])
@pytest.mark.parametrize("group,window,size,bits,tables", [(4, 32, 512, 8, 16), (2, 16, 136, 8, 16), (4, 128, 1024, 8, 16),   # the third: a window
                                                            (2, 32, 1000, 7, 24)])         # in parts; the last: eight tables per chunk
@pytest.mark.parametrize("between", [True, False])
def test_back_to_back(alpha, group, window, size, bits, tables, between):
    import torch
    from paper_2602_02199_b200 import binding as Bn
    heads, calls, B = 4, 24, 48
    gen = torch.Generator(device="cuda").manual_seed(size)
    planes = torch.randn(bits * tables, 128, generator=gen, device="cuda").bfloat16()
    src_k = [torch.randn(1, heads, size, 128, generator=gen, device="cuda") for _ in range(calls)]
    src_q = [torch.randn(1, heads * group, window, 128, generator=gen, device="cuda") for _ in range(calls)]

    def engine():
        return Bn.LaserKV(Bn.make_config(n_layers=1, batch=1, n_q_heads=heads * group, n_kv_heads=heads, block_size=size,
                                         window=window, max_blocks=calls, max_blocks_per_call=1, lsh_bits=bits, lsh_tables=tables,
                                         protection_divisor=4, budget_per_block=B, alpha=alpha), planes)

    queued, alone = engine(), engine()
    k, q = torch.empty(1, heads, size, 128, dtype=torch.bfloat16, device="cuda"), torch.empty(1, heads * group, window, 128, dtype=torch.bfloat16, device="cuda")
    if between:
        for x, y in zip(src_k, src_q):                   # the same buffers, written again in front of every call
            k.copy_(x)
            q.copy_(y)
            queued.laser_kv_select_block(0, k, k, q, 1)
    else:
        ready = [(x.bfloat16(), y.bfloat16()) for x, y in zip(src_k, src_q)]
        torch.cuda.synchronize()
        for x, y in ready:                               # nothing between the calls
            queued.laser_kv_select_block(0, x, x, y, 1)
    queued.laser_kv_poll_status()
    for x, y in zip(src_k, src_q):
        torch.cuda.synchronize()
        alone.laser_kv_select_block(0, x.bfloat16(), x.bfloat16(), y.bfloat16(), 1)
        torch.cuda.synchronize()
    for a, b in zip(queued.laser_kv_cache_view(0), alone.laser_kv_cache_view(0)):
        assert torch.equal(a, b) if torch.is_tensor(a) else a == b
