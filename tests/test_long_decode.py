"""Decoding in launches of several rounds (codes of up to four words): the searching decoder then rewrites its buckets and looks
up the last four positions at once.  Codes that sit on thresholds among random ones, the first and the last code, against
the oracle; and on the CPU that a rewritten entry leads to the index or says that the key bits leave it open."""
import numpy as np
import pytest
import torch

from oracle import beta_codebook as bc
from oracle import pvq_oracle as po
from oracle import pvq_pyref as pr
from paper_2410_16926_b200 import pvq

import blob_sections as bs

SETTINGS = [(8, 6), (8, 127), (16, 27), (16, 127), (32, 22), (32, 50), (32, 63), (64, 20), (64, 31)]


def threshold_codes(rng, N, K, want):
    """Codes whose path meets a threshold: random beginnings, then all pulses left on one coordinate; and their neighbours."""
    total = pr.count_table(N, K)[N][K]
    out = [0, 1, total - 1]
    while len(out) < want:
        y, left = [0] * N, K
        p = int(rng.integers(0, N - 1))
        for i in range(p):
            v = int(rng.integers(0, min(left, 4) + 1))
            y[i] = v if rng.integers(0, 2) else -v
            left -= v
        y[int(rng.choice([p, N - 1]))] += left if rng.integers(0, 2) else -left
        if sum(map(abs, y)) == K:
            c = pr.enumerate_point(y, K)
            out += [c + d for d in (0, -1, 1) if 0 <= c + d < total]
    return out[:want]


@pytest.mark.parametrize("N,K", SETTINGS)
def test_rewritten_entries(N, K):
    count = pr.count_table(N, K)
    sec = bs.section(count, N, K, pvq.code_words(N, K), 0)
    rng = np.random.default_rng(N + K)
    left_open = 0
    for c in threshold_codes(rng, N, K, 300):
        q = count[N][K] - c
        for i in range(N):
            n = N - 1 - i
            sh, tab, T = sec["shifts"][n], sec["tables"][n], sec["T"][n]
            key = bs.key_bits(q)
            b = (key >> sh) - (bs.KEY_OF_ONE >> sh)
            e = tab[b]
            entry = ((e << 24) + 0xFFFFFF - ((e >> 8) & 1) - 2 * ((((bs.KEY_OF_ONE >> sh) + b) << sh) + (e >> (32 - sh)))) & 0xFFFFFFFF
            total = (2 * key + entry) & 0xFFFFFFFF
            m = total >> 24
            if total & 0xFFFFFF == 0xFFFFFF:
                assert T[m] >= 1 << 24 and bs.key_bits(T[m]) == key
                left_open += 1
                m += 1 if T[m] < q else 0
            assert T[m] >= q and (m == 0 or T[m - 1] < q)
            q += (sec["T"][n - 1][2 * (m >> 1)] if n >= 1 else 0) - T[m]
    if pvq.code_words(N, K) > 1:
        assert left_open > 0           # these codes do reach the case


def long_rows(N, K, G, sms):
    """Rows of G groups for rounds enough of two tiles of 32 groups for each of 32 warps an SM that the buckets are rewritten
    (launch_search_g; that these sizes do it is tested in test_host_fake_gpu.py)."""
    sec = bs.section(pr.count_table(N, K), N, K, pvq.code_words(N, K), 0)
    rounds = 1.02 * max(3.0, (sec["t_off"] - sec["b_off"]) / 4 / (80 * N))
    return int(rounds * 2 * sms * 32 * 32 / G) + 1


@pytest.mark.gpu
def test_last_four_positions():
    """Every q of the table of the last four positions: behind 6 pulses and 27 zeros every point of four positions with 16, and
    some with 17, whose q are partly beyond the table."""
    N, K, G, b = 32, 22, 64, 16
    W = pvq.code_words(N, K)
    count = pr.count_table(N, K)
    first = pr.enumerate_point([K - 16] + [0] * 27 + [0, 0, 0, 16], K)   # the lowest code of them
    assert first + count[4][16] - 1 == pr.enumerate_point([K - 16] + [0] * 27 + [-16, 0, 0, 0], K)
    some = list(range(first, first + count[4][16]))
    some += [pr.enumerate_point([K - 17] + [0] * 27 + p, K) for p in ([17, 0, 0, 0], [-9, 8, 0, 0], [0, 0, 0, 17], [0, 0, 0, -17], [0, -1, 16, 0])]
    rows = long_rows(N, K, G, torch.cuda.get_device_properties(0).multi_processor_count)
    base = np.array([po.int_to_code(c, W) for c in some], dtype=np.uint32)
    codes = np.resize(base, (rows * G, W)).reshape(rows, G, W)
    sidx = np.random.default_rng(1).integers(0, 120, size=(rows, int(pvq.scale_row_stride(G, b))), dtype=np.uint8)  # finite binary16 amplitudes
    rnorm = np.ones(rows, dtype=np.float32)
    want, _ = po.decode(codes, sidx, rnorm, N, K, b, None)
    got = pvq.decode(torch.from_numpy(codes.view(np.int32)).cuda(), torch.from_numpy(sidx).cuda(), torch.from_numpy(rnorm).cuda(), N, K, b,
                     pvq.build_count_table(N, K), None)
    assert np.array_equal(got.view(torch.int16).cpu().numpy().view(np.uint16), want)


@pytest.mark.gpu
@pytest.mark.parametrize("N,K", SETTINGS)
def test_long_launch(N, K):
    G, b = 64, 8
    rows = long_rows(N, K, G, torch.cuda.get_device_properties(0).multi_processor_count)
    W = pvq.code_words(N, K)
    rng = np.random.default_rng(3 * N + K)
    total = pr.count_table(N, K)[N][K]
    some = threshold_codes(rng, N, K, 1500) + [int.from_bytes(rng.bytes(4 * W), "little") % total for _ in range(1500)]
    base = np.array([po.int_to_code(c, W) for c in some], dtype=np.uint32)
    codes = base[rng.integers(0, len(some), size=rows * G)].reshape(rows, G, W)
    if total < 1 << (32 * W):
        codes[7, 3] = 0xFFFFFFFF      # not a code: zeros, and the status says so
    sidx = rng.integers(0, 256, size=(rows, int(pvq.scale_row_stride(G, b))), dtype=np.uint8)
    rnorm = rng.random(rows).astype(np.float32) + np.float32(0.5)
    l_np = bc.levels_amp_f32(N, G, b)
    want, want_status = po.decode(codes, sidx, rnorm, N, K, b, l_np)
    status = torch.zeros(1, dtype=torch.int32, device="cuda")
    got = pvq.decode(torch.from_numpy(codes.view(np.int32)).cuda(), torch.from_numpy(sidx).cuda(), torch.from_numpy(rnorm).cuda(), N, K, b,
                     pvq.build_count_table(N, K), torch.from_numpy(l_np).cuda(), status=status)
    torch.cuda.synchronize()
    assert int(status.item()) == want_status
    bad = np.argwhere(got.view(torch.int16).cpu().numpy().view(np.uint16) != want)
    assert bad.size == 0, "decoded values differ first at %s" % (bad[0],)
