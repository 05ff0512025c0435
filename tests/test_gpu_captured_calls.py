"""Encode and decode recorded in a CUDA graph and replayed on other inputs, also after more count tables have been built
than windowed tables are kept (tests/test_host_fake_gpu.py checks who frees what)."""
import numpy as np
import pytest
import torch

from oracle import pvq_oracle as po
from paper_2410_16926_b200 import inputs, pvq

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("N,bits", [(32, 96), (64, 192), (128, 384), (64, 320)])
def test_replay_after_other_tables(N, bits):
    rows, G = 40, 6
    K = pvq.max_pulses(N, bits)
    W = pvq.code_words(N, K)
    table = pvq.build_count_table(N, K)
    rng = np.random.default_rng(bits)
    x = torch.zeros((rows, G * N), dtype=torch.bfloat16, device="cuda")
    side = torch.cuda.Stream()
    side.wait_stream(torch.cuda.current_stream())
    with torch.cuda.stream(side):
        enc = pvq.encode(x, N, K, 16, table, None)
        out = pvq.decode(*enc, N, K, 16, table, None)
    torch.cuda.current_stream().wait_stream(side)
    graph = torch.cuda.CUDAGraph()
    with torch.cuda.graph(graph):
        pvq.encode(x, N, K, 16, table, None, out=enc)
        pvq.decode(*enc, N, K, 16, table, None, out=out)
    for turn in range(3):
        if turn == 2:
            for k in range(86, 97):
                pvq.build_count_table(64, k)
        x_np = inputs.f32_to_bf16_bits((rng.standard_normal((rows, G * N)) * 0.02).astype(np.float32))
        x.copy_(torch.from_numpy(x_np.view(np.int16)).view(torch.bfloat16))
        graph.replay()
        torch.cuda.synchronize()
        o = po.encode(x_np, N, K, 16, None, W=W)
        assert np.array_equal(enc[0].cpu().numpy().view(np.uint32), o[0])
        assert np.array_equal(out.view(torch.int16).cpu().numpy().view(np.uint16), po.decode(*o, N, K, 16, None)[0])


@pytest.mark.parametrize("N,bits", [(64, 168), (128, 360), (256, 768)])
def test_tables_built_and_used_on_a_side_stream(N, bits):
    """No synchronisation between building a count table and the calls that use it, on a stream that does not wait for the
    legacy stream.  (Pulse counts that nothing else builds: the tables are made here.)"""
    rows, G = 64, 8
    K = pvq.max_pulses(N, bits)
    W = pvq.code_words(N, K)
    x = (np.random.default_rng(bits).standard_normal((rows, G * N)) * 0.02).astype(np.float32)
    x_dev = torch.from_numpy(x).cuda()
    torch.cuda.synchronize()
    with torch.cuda.stream(torch.cuda.Stream()):
        table = pvq.build_count_table(N, K)
        enc = pvq.encode(x_dev, N, K, 16, table, None)
        out = pvq.decode(*enc, N, K, 16, table, None)
    torch.cuda.synchronize()
    o = po.encode(x, N, K, 16, None, W=W)
    assert np.array_equal(enc[0].cpu().numpy().view(np.uint32), o[0])
    assert np.array_equal(out.view(torch.int16).cpu().numpy().view(np.uint16), po.decode(*o, N, K, 16, None)[0])
