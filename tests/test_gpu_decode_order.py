"""Decode attention on a handle whose cache changes between the calls, and right behind the call that fills it:
the kernel starts beside that call's last kernel, and a layer's tensor maps are kept while its length stands."""
import pytest

pytestmark = pytest.mark.gpu

H, G, S, B = 4, 4, 1024, 400


def _engine(Bn, planes, blocks, layers=1):
    return Bn.LaserKV(Bn.make_config(n_layers=layers, batch=1, n_q_heads=H * G, n_kv_heads=H, block_size=S, window=32,
                                     max_blocks=blocks, max_blocks_per_call=blocks, lsh_bits=8, lsh_tables=16,
                                     protection_divisor=4, budget_per_block=B, alpha=0.75), planes)


def _inputs(torch, seed, blocks):
    gen = torch.Generator(device="cuda").manual_seed(seed)
    k, v = (torch.randn(1, H, blocks * S, 128, generator=gen, device="cuda").bfloat16() for _ in range(2))
    q = torch.randn(1, H * G, 32, 128, generator=gen, device="cuda").bfloat16()
    return k, v, q


def _expect(torch, eng, layer, q):
    k, v, _, n = eng.laser_kv_cache_view(layer)
    # (the view's rows are bf16 bit patterns)
    k, v = (x[:, :, :n].view(torch.bfloat16).double() for x in (k, v))
    w = torch.softmax(torch.einsum("bhgd,bhnd->bhgn", q.double().view(1, H, G, 128), k) / 128 ** 0.5, -1)
    return torch.einsum("bhgn,bhnd->bhgd", w, v).view(1, H * G, 128), n


def _check(torch, eng, layer, q, entries):
    out = eng.laser_kv_decode_attention(layer, q).double()
    want, n = _expect(torch, eng, layer, q)
    assert n == entries
    assert ((out - want).norm() / want.norm()).item() < 8e-7


def test_cache_that_grows_shrinks_and_is_refilled():
    import torch
    from paper_2602_02199_b200 import binding as Bn
    gen = torch.Generator(device="cuda").manual_seed(1)
    eng = _engine(Bn, torch.randn(128, 128, generator=gen, device="cuda").bfloat16(), 4, layers=2)
    q = torch.randn(1, H * G, 128, generator=gen, device="cuda").bfloat16()
    k, v, qw = _inputs(torch, 2, 4)
    for layer in (0, 1):
        for t in range(4):                                     # one more block, and a decode after each
            eng.laser_kv_select_block(layer, k[:, :, t * S:(t + 1) * S], v[:, :, t * S:(t + 1) * S], qw, 1)
            _check(torch, eng, layer, q, (t + 1) * B)
            _check(torch, eng, layer, q, (t + 1) * B)
    for seed, blocks in ((3, 1), (4, 2), (5, 2)):              # shorter than before, longer, as long with other rows
        eng.laser_kv_reset(0)
        k, v, qw = _inputs(torch, seed, blocks)
        eng.laser_kv_select_block(0, k, v, qw, blocks)
        _check(torch, eng, 0, q, blocks * B)
        _check(torch, eng, 1, q, 4 * B)                        # the other layer is as it was
    eng.laser_kv_poll_status()


@pytest.mark.parametrize("blocks", [1, 4])
def test_decode_queued_right_behind_the_selection(blocks):
    import torch
    from paper_2602_02199_b200 import binding as Bn
    gen = torch.Generator(device="cuda").manual_seed(6)
    planes = torch.randn(128, 128, generator=gen, device="cuda").bfloat16()
    q = torch.randn(1, H * G, 128, generator=gen, device="cuda").bfloat16()
    eng = _engine(Bn, planes, blocks)
    inputs = [_inputs(torch, 10 + i, blocks) for i in range(12)]

    def run(wait):
        outs = []
        for k, v, qw in inputs:
            eng.laser_kv_reset(0)
            eng.laser_kv_select_block(0, k, v, qw, blocks)
            if wait:
                torch.cuda.synchronize()
            outs.append(eng.laser_kv_decode_attention(0, q))
            if wait:
                torch.cuda.synchronize()
        return outs
    queued, alone = run(False), run(True)
    eng.laser_kv_poll_status()
    for a, b in zip(queued, alone):
        assert torch.equal(a, b)
