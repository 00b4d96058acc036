"""The projection pass of a select call cuts its tiles into unequal slices, one behind the other or abreast in the hyperplane
chunks: every key's collisions are those that the step-level entry point counts over equal slices."""
import pytest

pytestmark = pytest.mark.gpu


# (KV heads, block size, blocks, bits, tables): one tile in all; fewer tiles than CTAs; one to eight chunks, among them counts
# that do not divide the grid; more query-signature CTAs than SMs; keys above and below the size from which slices lie abreast
@pytest.mark.parametrize("n_kv_heads,size,nb,bits,tables", [
    (1, 128, 1, 8, 8), (2, 1000, 3, 8, 16), (8, 1864, 2, 10, 64), (4, 2048, 4, 10, 48), (3, 776, 5, 10, 40), (8, 512, 3, 12, 24),
    (8, 4096, 8, 10, 64), (8, 4096, 9, 10, 64), (8, 4104, 9, 8, 64), (8, 4096, 9, 12, 64), (8, 4096, 9, 6, 24), (20, 4096, 4, 10, 64)])
def test_counts_of_unequal_slices(n_kv_heads, size, nb, bits, tables):
    import torch
    from paper_2602_02199_b200 import binding as Bn
    G, W = 2, 32
    gen = torch.Generator(device="cuda").manual_seed(size + tables)
    q = torch.randn(1, n_kv_heads * G, W, 128, generator=gen, device="cuda").bfloat16()
    k = torch.randn(1, n_kv_heads, nb * size, 128, generator=gen, device="cuda").bfloat16()
    planes = torch.randn(tables * bits, 128, generator=gen, device="cuda").bfloat16()
    eng = Bn.LaserKV(Bn.make_config(n_layers=1, batch=1, n_q_heads=n_kv_heads * G, n_kv_heads=n_kv_heads, block_size=size, window=W,
                                    max_blocks=2 * nb, max_blocks_per_call=nb, lsh_bits=bits, lsh_tables=tables,
                                    protection_divisor=4, budget_per_block=64, alpha=0.5), planes)
    want, status = Bn.laser_kv_collision_counts(k, q, planes, size, nb, bits, tables)
    for _ in range(2):                                   # the second call starts beside the first one's append
        eng.laser_kv_select_block(0, k, k, q, nb)
        got = eng.laser_kv_debug_view().counts.clone()
        eng.laser_kv_poll_status()
        assert torch.equal(got.view_as(want), want)
    assert int(status.view(torch.int32)[0]) == 0
