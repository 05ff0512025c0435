"""Rows of few and of many groups through every encode-side call, against the oracle bit for bit: rows that a thread block
holds, one group beyond that, and the longest (4096 groups); more pulses than a byte holds."""
import numpy as np
import pytest
import torch

from oracle import beta_codebook as bc
from oracle import pvq_oracle as po
from paper_2410_16926_b200 import inputs, pvq

pytestmark = pytest.mark.gpu

# direction bits; 8 / 56, 16 / 90, 32 / 200: more than 127 pulses
SETTINGS = [(8, 24), (8, 56), (16, 48), (16, 90), (32, 64), (32, 96), (32, 200), (64, 128), (64, 192), (64, 320), (128, 384), (128, 512),
            (256, 600)]


def bf16_bits(t):
    return t.view(torch.int16).cpu().numpy().view(np.uint16)


@pytest.mark.parametrize("N,bits", SETTINGS)
@pytest.mark.parametrize("G,rows,kind", [(2, 5, "bf16"), (511, 3, "f32"), (513, 3, "bf16"), (4096, 2, "bf16"), (4096, 1, "f32")])
def test_every_call(N, bits, G, rows, kind):
    if N * G > 1 << 19:
        rows = 1
    K = pvq.max_pulses(N, bits)
    W = pvq.code_words(N, K)
    b = 6 if N <= 64 else 16
    rng = np.random.default_rng(N * bits + G)
    x = (rng.standard_normal((rows, G * N)) * 0.02).astype(np.float32)
    x[:, ::31] *= 8
    x_np = inputs.f32_to_bf16_bits(x) if kind == "bf16" else x
    x_dev = torch.from_numpy(x_np.view(np.int16)).cuda().view(torch.bfloat16) if kind == "bf16" else torch.from_numpy(x_np).cuda()
    e_np = l_np = edges = levels = None
    if b != 16:
        e_np, l_np = bc.edges_f32(N, G, b), bc.levels_amp_f32(N, G, b)
        edges, levels = torch.from_numpy(e_np).cuda(), torch.from_numpy(l_np).cuda()
    table = pvq.build_count_table(N, K)
    for amp_mode in (None, 1):
        codes, sidx, rnorm = pvq.encode(x_dev, N, K, b, table, edges, amp_mode=amp_mode)
        torch.cuda.synchronize()
        o = po.encode(x_np, N, K, b, e_np, W=W, amp_mode=amp_mode or 0)
        assert np.array_equal(codes.cpu().numpy().view(np.uint32), o[0]), amp_mode
        assert np.array_equal(sidx.cpu().numpy(), o[1]) and np.array_equal(rnorm.cpu().numpy().view(np.uint32), o[2].view(np.uint32)), amp_mode
        if amp_mode is None:
            want = po.decode(*o, N, K, b, l_np)[0]
            assert np.array_equal(bf16_bits(pvq.decode(codes, sidx, rnorm, N, K, b, table, levels)), want)
            assert np.array_equal(bf16_bits(pvq.roundtrip(x_dev, N, K, b, table, edges, levels)), want)


# the rotated round trip takes rows of any length, with more pulses than a byte holds too
@pytest.mark.parametrize("N,bits,G,block", [(8, 56, 128, 64), (8, 56, 1024, 4096), (16, 90, 640, 512), (32, 64, 1024, 4096), (64, 320, 600, 256)])
def test_rotated_round_trip(N, bits, G, block):
    rows, b = 3, 16
    K = pvq.max_pulses(N, bits)
    rng = np.random.default_rng(G + bits)
    x = rng.standard_normal((rows, G * N)).astype(np.float32)
    signs = rng.choice([-1.0, 1.0], size=block).astype(np.float32)
    y = po.rotate(x, block, signs)
    o = po.encode(y, N, K, b, None, W=pvq.code_words(N, K))
    want = po.decode(*o, N, K, b, None)[0]
    got = pvq.rotate_roundtrip(torch.from_numpy(x).cuda(), block, torch.from_numpy(signs).cuda(), N, K, b, pvq.build_count_table(N, K), None, None)
    assert np.array_equal(bf16_bits(got), want)


# Rows of whole warps, a power of two of them or not (lanes a row; N / 32 lanes a group): a warp's part of a row's energy and the
# zeros between the rows' parts; rows that leave a thread block's lanes idle; input and output in wider rows.
@pytest.mark.parametrize("N,bits,b", [(32, 64, 8), (64, 256, 3), (128, 512, 16), (256, 768, 5)])
@pytest.mark.parametrize("lanes", [32, 64, 72, 80, 96, 160, 352])
@pytest.mark.parametrize("block", [0, 256])
def test_round_trip_lanes(N, bits, b, lanes, block):
    rows, cols = 401, lanes * 32
    if cols % max(block, N) != 0:
        pytest.skip("rows of whole groups and rotation blocks")
    G = cols // N
    K = pvq.max_pulses(N, bits)
    rng = np.random.default_rng(N + lanes)
    x = np.zeros((rows, cols + 24), dtype=np.uint16)
    x[:, :cols] = inputs.f32_to_bf16_bits(rng.standard_normal((rows, cols)).astype(np.float32))
    e_np, l_np = (None, None) if b == 16 else (bc.edges_f32(N, G, b), bc.levels_amp_f32(N, G, b))
    edges, levels = (None, None) if b == 16 else (torch.from_numpy(e_np).cuda(), torch.from_numpy(l_np).cuda())
    table = pvq.build_count_table(N, K)
    out = torch.full((rows, cols + 8), 7.0, dtype=torch.bfloat16, device="cuda")
    x_dev = torch.from_numpy(x.view(np.int16)).cuda().view(torch.bfloat16)[:, :cols]
    values = np.ascontiguousarray(x[:, :cols])
    if block:
        signs = rng.choice([-1.0, 1.0], size=block).astype(np.float32)
        values = po.rotate(values, block, signs)
        pvq.rotate_roundtrip(x_dev, block, torch.from_numpy(signs).cuda(), N, K, b, table, edges, levels, out=out[:, :cols])
    else:
        pvq.roundtrip(x_dev, N, K, b, table, edges, levels, out=out[:, :cols])
    want = po.decode(*po.encode(values, N, K, b, e_np, W=pvq.code_words(N, K)), N, K, b, l_np)[0]
    assert np.array_equal(bf16_bits(out[:, :cols].contiguous()), want)
    assert bool((out[:, cols:] == 7.0).all())
