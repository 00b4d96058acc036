"""The gather + append of a select call at the edges of its row groups (64 rows a CTA, 16 at a time), in grids that
start beside the selection and in one that does not: every kept row is the source row its position names, and the
rows behind the last one stay as they were."""
import pytest

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("budget,nb,n_kv_heads,batch", [(1, 3, 2, 1), (15, 2, 3, 2), (64, 2, 8, 1), (65, 5, 2, 2), (127, 3, 8, 1),
                                                        (200, 16, 8, 2)])
def test_kept_rows_are_the_rows_named(budget, nb, n_kv_heads, batch):
    import torch
    from paper_2602_02199_b200 import binding as Bn
    S, W = 264, 16
    gen = torch.Generator(device="cuda").manual_seed(budget)
    k, v = (torch.randn(batch, n_kv_heads, 2 * nb * S, 128, generator=gen, device="cuda").bfloat16() for _ in range(2))
    q = torch.randn(batch, n_kv_heads, W, 128, generator=gen, device="cuda").bfloat16()
    planes = torch.randn(8 * 8, 128, generator=gen, device="cuda").bfloat16()
    eng = Bn.LaserKV(Bn.make_config(n_layers=1, batch=batch, n_q_heads=n_kv_heads, n_kv_heads=n_kv_heads, block_size=S, window=W,
                                    max_blocks=2 * nb + 1, max_blocks_per_call=nb, lsh_bits=8, lsh_tables=8,
                                    protection_divisor=4, budget_per_block=budget, alpha=0.5), planes)
    eng.cache_mem.zero_()
    for t in range(2):                                   # the second call starts beside the first one's append
        eng.laser_kv_select_block(0, k[:, :, t * nb * S:(t + 1) * nb * S], v[:, :, t * nb * S:(t + 1) * nb * S], q, nb)
    eng.laser_kv_poll_status()
    kc, vc, pos, n = eng.laser_kv_cache_view(0)
    assert n == 2 * nb * budget
    p = pos[:, :, :n].long()
    assert (p.diff(dim=-1) > 0).all() and int(p.min()) >= 0 and int(p.max()) < 2 * nb * S
    assert (torch.bincount((p // S).flatten(), minlength=2 * nb) == budget * batch * n_kv_heads).all()
    want = p[..., None].expand(-1, -1, -1, 128)
    assert torch.equal(kc[:, :, :n], torch.gather(k, 2, want).view(torch.int16))
    assert torch.equal(vc[:, :, :n], torch.gather(v, 2, want).view(torch.int16))
    assert not kc[:, :, n:].any() and not vc[:, :, n:].any() and not pos[:, :, n:].any()
