"""The rotated round trip over the sizes of a rotation block: inside a lane, a warp, and across 2 to 16 warps of a thread
block; one tile and many for a thread block, rows that share one; both input types."""
import numpy as np
import pytest
import torch

from oracle import beta_codebook as bc
from oracle import pvq_oracle as po
from paper_2410_16926_b200 import inputs, pvq

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("N,bits,b", [(32, 64, 8), (64, 256, 6), (128, 512, 16), (256, 768, 6), (16, 48, 4)])
@pytest.mark.parametrize("block,blocks,rows", [(0, 5, 3000), (0, 32, 40), (512, 3, 900), (1024, 1, 2600), (1024, 3, 300), (2048, 1, 1300), (2048, 3, 70),
                                               (4096, 1, 1300), (4096, 2, 60), (8192, 1, 400), (8192, 2, 11), (16384, 1, 160)])
def test_block_sizes(N, bits, b, block, blocks, rows):
    block = block or N             # the smallest: a group
    if N == 16 and block > 8192:   # (a lane holds 16 values, a thread block 512 lanes)
        block = 8192
    cols = block * blocks
    if cols < 2 * N:
        cols *= 2
    G = cols // N
    rng = np.random.default_rng(N + block + rows)
    x = rng.standard_normal((rows, cols)).astype(np.float32)
    x[:, ::257] *= 20
    signs = rng.choice([-1.0, 1.0], size=block).astype(np.float32)
    K = pvq.max_pulses(N, bits)
    e_np, l_np = (None, None) if b == 16 else (bc.edges_f32(N, G, b), bc.levels_amp_f32(N, G, b))
    edges, levels = (None, None) if b == 16 else (torch.from_numpy(e_np).cuda(), torch.from_numpy(l_np).cuda())
    table = pvq.build_count_table(N, K)
    for kind in ("bf16", "f32"):
        n = rows if kind == "bf16" else min(rows, 40)
        x_np = inputs.f32_to_bf16_bits(x) if kind == "bf16" else x[:n]
        y = po.rotate(x_np, block, signs)
        want = po.decode(*po.encode(y, N, K, b, e_np, W=pvq.code_words(N, K)), N, K, b, l_np)[0]
        x_dev = torch.from_numpy(x_np.view(np.int16)).cuda().view(torch.bfloat16) if kind == "bf16" else torch.from_numpy(x_np).cuda()
        got = pvq.rotate_roundtrip(x_dev, block, torch.from_numpy(signs).cuda(), N, K, b, table, edges, levels)
        assert np.array_equal(got.view(torch.int16).cpu().numpy().view(np.uint16), want), kind
