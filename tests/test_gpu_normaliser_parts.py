"""Segments whose log-sum-exp partials are few enough for every warp of the score pass to fetch them all, and more, so that the
four warps of a group share the fetching (above five), for every width of a group's query columns: the scores are those
of a softmax in fp64. Blocks of one head follow one another, so that a CTA goes from segment to segment."""
import pytest

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("n_kv_heads,nb", [(37, 1), (21, 1), (9, 2), (6, 3), (2, 4), (1, 2)])
@pytest.mark.parametrize("group,window", [(1, 16), (2, 48), (5, 32), (7, 32), (4, 64)])
def test_scores_against_fp64(n_kv_heads, nb, group, window):
    import torch
    from paper_2602_02199_b200 import binding as Bn
    S = 3080
    gen = torch.Generator(device="cuda").manual_seed(n_kv_heads * 100 + group)
    q = torch.randn(1, n_kv_heads * group, window, 128, generator=gen, device="cuda").bfloat16()
    k = torch.randn(1, n_kv_heads, nb * S, 128, generator=gen, device="cuda").bfloat16()
    logits = torch.einsum("hqd,hkd->hqk", q[0].double().view(n_kv_heads, group * window, 128), k[0].double()) / 128 ** 0.5
    want = torch.softmax(logits.view(n_kv_heads, group * window, nb, S), dim=-1).sum(1)
    planes = torch.randn(8 * 8, 128, generator=gen, device="cuda").bfloat16()
    eng = Bn.LaserKV(Bn.make_config(n_layers=1, batch=1, n_q_heads=n_kv_heads * group, n_kv_heads=n_kv_heads, block_size=S,
                                    window=window, max_blocks=nb, max_blocks_per_call=nb, lsh_bits=8, lsh_tables=8,
                                    protection_divisor=4, budget_per_block=64, alpha=1.0), planes)
    eng.laser_kv_select_block(0, k, k, q, nb)
    got = eng.laser_kv_debug_view().s_exact
    eng.laser_kv_poll_status()
    for s in (got[0], Bn.laser_kv_window_scores(k, q, S, nb)[0]):
        # probabilities from exponentials of 2.7e-6 and sums of a few thousand fp32 terms
        assert ((s.double() - want).abs() / want).max().item() <= 1e-4
