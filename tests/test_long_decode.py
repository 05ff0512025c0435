"""Decoding in launches of several rounds (codes of up to four words): the searching decoder then rewrites its buckets, looks
up the last four positions at once, and finds out afterwards that key bits could not decide.  Codes that sit on thresholds
among random ones, the first and the last code, against the oracle; and on the CPU that what is not decided does show."""
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
def test_undecided_key_bits_show(N, K):
    count = pr.count_table(N, K)
    sec = bs.section(count, N, K, pvq.code_words(N, K), 0)
    rng = np.random.default_rng(N + K)
    missed = 0
    for c in threshold_codes(rng, N, K, 300):
        q, k, shown, m_all = count[N][K] - c, K, False, []
        for i in range(N):
            n = N - 1 - i
            sh, tab = sec["shifts"][n], sec["tables"][n]
            last = (((bs.KEY_OF_ONE >> sh) + len(tab)) << sh) - 1
            assert q >= 1
            key = min(bs.key_bits(q), last)
            b = (key >> sh) - (bs.KEY_OF_ONE >> sh)
            entry = ((tab[b] << 24) + 0xFFFFFF - ((((bs.KEY_OF_ONE >> sh) + b) << sh) + (tab[b] >> (32 - sh)))) & 0xFFFFFFFF
            m = ((key + entry) & 0xFFFFFFFF) >> 24
            assert m <= 2 * K + 1
            shown = shown or m > 2 * k
            m_all.append(m)
            e = sec["E"][n][m] if m <= 2 * K else 0     # (the entry behind the last threshold is zero)
            q = (q + e) % (1 << (32 * sec["words"][n]))
            k = m >> 1
        right = bs.decode_with(sec, count, c, N, K)
        k, y = K, []
        for m in m_all:
            y.append(k - (m >> 1) if m & 1 else (m >> 1) - k)
            k = m >> 1
        assert shown or list(y) == list(right)
        missed += list(y) != list(right)
    if pvq.code_words(N, K) > 1:
        assert missed > 0           # these codes do reach the case


@pytest.mark.gpu
@pytest.mark.parametrize("N,K", SETTINGS)
def test_long_launch(N, K):
    G, rows, b = 64, 5001, 8        # 320064 groups: more than a round of 148 x 32 warps of two tiles
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
