"""Groups whose residuals agree in their leading bits: which of them get the last pulses is decided on the exact fp32
values, lowest position first among equals.  One to all values of a group differ by a few units in the last place or not
at all, so that between none and all of a lane's residuals are left for that decision; every lane count and both point forms."""
import numpy as np
import pytest
import torch

from oracle import beta_codebook as bc
from oracle import pvq_oracle as po
from paper_2410_16926_b200 import inputs, pvq

pytestmark = pytest.mark.gpu


# (8, 56), (16, 90), (64, 256), (128, 512): more than 127 pulses
@pytest.mark.parametrize("N,bits", [(8, 24), (8, 56), (16, 48), (16, 90), (32, 64), (32, 96), (64, 192), (64, 256), (128, 384), (128, 512), (256, 768)])
@pytest.mark.parametrize("kind", ["bf16", "f32"])
def test_near_and_exact_ties(N, bits, kind):
    G, b = 4, 6
    rng = np.random.default_rng(7 * N + bits)
    rows = []
    for alike in sorted({1, 2, 3, 4, 5, N // 4, N // 2, N - 1, N}):
        for spread in (0, 1, 40):  # units of 2^-20 between neighbours: equal, apart in the last bits, apart in some bits more
            for _ in range(2):
                row = rng.standard_normal((G, N))
                for g in range(G):
                    where = rng.permutation(N)[:alike]
                    row[g, where] = abs(rng.standard_normal() + 0.2) * (1 + spread * 2.0 ** -20 * rng.integers(0, 8, size=alike)) * rng.choice([-1, 1], size=alike)
                rows.append(row.reshape(-1))
    x = np.array(rows, dtype=np.float32)
    K = pvq.max_pulses(N, bits)
    W = pvq.code_words(N, K)
    e_np, l_np = bc.edges_f32(N, G, b), bc.levels_amp_f32(N, G, b)
    x_np = inputs.f32_to_bf16_bits(x) if kind == "bf16" else x
    x_dev = torch.from_numpy(x_np.view(np.int16)).cuda().view(torch.bfloat16) if kind == "bf16" else torch.from_numpy(x_np).cuda()
    table = pvq.build_count_table(N, K)
    edges, levels = torch.from_numpy(e_np).cuda(), torch.from_numpy(l_np).cuda()
    o = po.encode(x_np, N, K, b, e_np, W=W)
    o_out, _ = po.decode(*o, N, K, b, l_np)
    codes, sidx, rnorm = pvq.encode(x_dev, N, K, b, table, edges)
    back = pvq.roundtrip(x_dev, N, K, b, table, edges, levels)
    torch.cuda.synchronize()
    assert np.array_equal(codes.cpu().numpy().view(np.uint32), o[0]), "codes"
    assert np.array_equal(sidx.cpu().numpy(), o[1]) and np.array_equal(rnorm.cpu().numpy().view(np.uint32), o[2].view(np.uint32))
    assert np.array_equal(back.view(torch.int16).cpu().numpy().view(np.uint16), o_out), "round trip"
