"""Encoding with most threads of a block idle, when they stage the tables and the others wait for them half way, and with all of
them at work, when a block meets once first; a tile or two a team, ragged at the end; against the oracle."""
import numpy as np
import pytest
import torch

from oracle import beta_codebook as bc
from oracle import pvq_oracle as po
from paper_2410_16926_b200 import inputs, pvq

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("N,bits", [(8, 24), (8, 40), (16, 30), (16, 48), (16, 80), (32, 32), (32, 64), (32, 96), (32, 128), (64, 64), (64, 128)])
@pytest.mark.parametrize("rows,G", [(1, 2), (149, 32), (300, 33), (2001, 96)])
def test_idle_and_busy_blocks(N, bits, rows, G):
    b = 5
    K = pvq.max_pulses(N, bits)
    W = pvq.code_words(N, K)
    rng = np.random.default_rng(N * bits + rows)
    x = (rng.standard_normal((rows, G * N)) * 0.02).astype(np.float32)
    e_np = bc.edges_f32(N, G, b)
    edges, table = torch.from_numpy(e_np).cuda(), pvq.build_count_table(N, K)
    for kind in ("bf16", "f32"):
        x_np = inputs.f32_to_bf16_bits(x) if kind == "bf16" else x
        x_dev = torch.from_numpy(x_np.view(np.int16)).cuda().view(torch.bfloat16) if kind == "bf16" else torch.from_numpy(x_np).cuda()
        codes, sidx, rnorm = pvq.encode(x_dev, N, K, b, table, edges)
        torch.cuda.synchronize()
        o = po.encode(x_np, N, K, b, e_np, W=W)
        assert np.array_equal(codes.cpu().numpy().view(np.uint32), o[0]), kind
        assert np.array_equal(sidx.cpu().numpy(), o[1]) and np.array_equal(rnorm.cpu().numpy().view(np.uint32), o[2].view(np.uint32)), kind
