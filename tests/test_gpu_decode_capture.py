"""The first decode call of a handle inside a stream capture: what the call asks the device for does not disturb the capture."""
import subprocess
import sys

import pytest

pytestmark = pytest.mark.gpu

FIRST = """
import torch
from paper_2602_02199_b200 import binding as Bn
for heads, entries in ((8, 1640), (4, 56 * 64), (16, 72 * 64)):            # clusters of eight, of sixteen, by way of memory
    gen = torch.Generator(device="cuda").manual_seed(entries)
    planes = torch.randn(64, 128, generator=gen, device="cuda").bfloat16()
    eng = Bn.LaserKV(Bn.make_config(n_layers=1, batch=1, n_q_heads=4 * heads, n_kv_heads=heads, block_size=entries, window=16, max_blocks=1,
                                    max_blocks_per_call=1, lsh_bits=8, lsh_tables=8, protection_divisor=2, budget_per_block=entries,
                                    alpha=1.0), planes)
    k, v = (torch.randn(1, heads, entries, 128, generator=gen, device="cuda").bfloat16() for _ in range(2))
    q = torch.randn(1, 4 * heads, 16, 128, generator=gen, device="cuda").bfloat16()
    eng.laser_kv_select_block(0, k, v, q, 1)
    d, graph = q[:, :, 3].contiguous(), torch.cuda.CUDAGraph()
    torch.cuda.synchronize()
    with torch.cuda.graph(graph):
        out = eng.laser_kv_decode_attention(0, d)
    graph.replay()
    eng.laser_kv_poll_status()
    assert torch.equal(out, eng.laser_kv_decode_attention(0, d))
print("captured")
"""


def test_first_decode_of_a_process_inside_a_capture():
    run = subprocess.run([sys.executable, "-c", FIRST], capture_output=True, text=True, timeout=300)
    assert run.returncode == 0 and "captured" in run.stdout, run.stderr[-2000:]
