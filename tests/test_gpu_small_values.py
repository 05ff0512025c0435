"""Values whose squares are not representable: with |x| below 2^-67 the square of a bf16 value has bits below the last
place of the smallest fp32 number, so rounding the products before they are added (one rounding an operation, as
the oracle) and adding them in one go give different energies.  Every encoder and the round trip."""
import numpy as np
import pytest
import torch

from oracle import beta_codebook as bc
from oracle import pvq_oracle as po
from paper_2410_16926_b200 import inputs, pvq

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("N,bits", [(8, 24), (16, 48), (32, 96), (64, 128), (64, 192), (128, 384), (256, 768)])
@pytest.mark.parametrize("kind", ["bf16", "f32"])
def test_energies_of_tiny_values(N, bits, kind):
    rows, G, b = 24, 8, 6
    rng = np.random.default_rng(N + bits)
    # magnitudes from 1e-24 to 1e-19, neighbours of different size; every third row squares to subnormal sums only
    x = rng.choice([-1.0, 1.0], size=(rows, G * N)) * 10.0 ** rng.uniform(-24, -19, size=(rows, G * N))
    x[::3] = rng.choice([-1.0, 1.0], size=x[::3].shape) * 10.0 ** rng.uniform(-22.5, -21, size=x[::3].shape)
    x = x.astype(np.float32)
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
    assert np.array_equal(rnorm.cpu().numpy().view(np.uint32), o[2].view(np.uint32)), "row norms"
    assert np.array_equal(sidx.cpu().numpy(), o[1]), "amplitude indices"
    assert np.array_equal(codes.cpu().numpy().view(np.uint32), o[0]), "codes"
    assert np.array_equal(back.view(torch.int16).cpu().numpy().view(np.uint16), o_out), "round trip"
