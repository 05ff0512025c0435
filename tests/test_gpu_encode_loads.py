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


# Enough values that teams make do with one input buffer where that lets more of them fit (more than 8 x 148 x 896 lanes):
# which is asked for in the middle of a chunk, over values that least-squares amplitudes have just read.  Teams of one warp, and
# of several; rows of one chunk, and of several.
@pytest.mark.parametrize("N,bits,G,kind,amp_mode", [(32, 96, 96, "bf16", 0), (32, 96, 128, "f32", 0), (32, 96, 130, "bf16", 1), (32, 128, 64, "f32", 1),
                                                    (64, 128, 48, "bf16", 0), (64, 128, 50, "f32", 1), (32, 96, 700, "f32", 1), (32, 128, 1500, "bf16", 1),
                                                    (64, 96, 1021, "f32", 0), (16, 64, 256, "f32", 1)])
def test_long_launches(N, bits, G, kind, amp_mode):
    b = 4
    K = pvq.max_pulses(N, bits)
    W = pvq.code_words(N, K)
    lanes = G * max(1, N // 32)
    rows = (1 << 20) // lanes + 150
    gen = torch.Generator(device="cuda")
    gen.manual_seed(N * bits + G)
    x = torch.randn((rows, G * N), generator=gen, device="cuda", dtype=torch.float32)
    if kind == "bf16":
        x = x.to(torch.bfloat16)
    table = pvq.build_count_table(N, K)
    edges, _ = pvq.build_scale_codebook(N, G, b)
    whole = pvq.encode(x, N, K, b, table, edges, amp_mode=amp_mode)
    step = rows // 9 + 1               # launches with two input buffers a team
    for r in range(0, rows, step):
        part = pvq.encode(x[r:r + step], N, K, b, table, edges, amp_mode=amp_mode)
        for got, want in zip(whole, part):
            assert torch.equal(got[r:r + step].view(torch.uint8), want.view(torch.uint8)), r
    some = x[rows // 2:rows // 2 + 2]
    x_np = some.cpu().view(torch.int16).numpy().view(np.uint16) if kind == "bf16" else some.cpu().numpy()
    o = po.encode(x_np, N, K, b, edges.cpu().numpy(), W=W, amp_mode=amp_mode)
    assert np.array_equal(whole[0][rows // 2:rows // 2 + 2].cpu().numpy().view(np.uint32), o[0])
    assert np.array_equal(whole[1][rows // 2:rows // 2 + 2].cpu().numpy(), o[1])
