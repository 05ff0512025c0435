"""The kernels for wide codes (windowed tables: group size 64 with codes of 5 to 8 words, 128 with 9 to 12, 256 with 24)
against the CPU oracle, bit for bit, where they can go wrong: every code width, tiles that are not full, rows
that do not fit a block, paths that leave the windows, values of 128 pulses and more, codes that sit on
thresholds, several matrices in a call, tables that are not there.  And the encoder's tables of 112 entries a row."""
import numpy as np
import pytest
import torch

from oracle import pvq_oracle as po
from paper_2410_16926_b200 import inputs, pvq

pytestmark = pytest.mark.gpu

DEV = "cuda"
WIDTHS = [(64, 160), (64, 192), (64, 224), (64, 256), (128, 288), (128, 320), (128, 352), (128, 384), (256, 768)]


def as_u32(t):
    return t.cpu().numpy().view(np.uint32)


def bf16_bits(t):
    return t.view(torch.int16).cpu().numpy().view(np.uint16)


def source(rng, kind, rows, cols, N):
    x = rng.standard_normal((rows, cols))
    i = np.arange(cols) % N
    if kind == "outliers":
        x[:, ::37] *= 25
    elif kind == "one value":         # |y| of 128 and more where there are that many pulses
        x[:, ::61] *= 2000
    elif kind == "front":             # the pulses early in the group, then late: paths below and above the windows
        x *= np.exp(-i / 8.0)
    elif kind == "back":
        x *= np.exp(i / 8.0)
    elif kind == "sparse":
        x *= rng.random((rows, cols)) < 0.05
        x[0, :2 * N] = 0.0            # whole groups of zeros, and one with a single negative value
        x[0, N] = -1.0
    return (x * 0.02).astype(np.float32)


def check(x, kind, N, K, b=16, amp_mode=0):
    W = pvq.code_words(N, K)
    x_np = inputs.f32_to_bf16_bits(x) if kind == "bf16" else x
    x_dev = torch.from_numpy(x_np.view(np.int16)).to(DEV).view(torch.bfloat16) if kind == "bf16" else torch.from_numpy(x_np).to(DEV)
    table = pvq.build_count_table(N, K)
    edges = levels = e_np = l_np = None
    if b != 16:
        edges, levels = pvq.build_scale_codebook(N, x.shape[1] // N, b)
        e_np, l_np = edges.cpu().numpy(), levels.cpu().numpy()
    o = po.encode(x_np, N, K, b, e_np, W=W, amp_mode=amp_mode)
    o_out, _ = po.decode(*o, N, K, b, l_np)
    codes, sidx, rnorm = pvq.encode(x_dev, N, K, b, table, edges, amp_mode=amp_mode)
    out = pvq.decode(codes, sidx, rnorm, N, K, b, table, levels)
    torch.cuda.synchronize()
    assert np.array_equal(as_u32(codes), o[0]), "codes"
    assert np.array_equal(sidx.cpu().numpy(), o[1]) and np.array_equal(as_u32(rnorm), o[2].view(np.uint32)), "amplitudes"
    assert np.array_equal(bf16_bits(out), o_out), "decoded"


@pytest.mark.parametrize("N,bits", WIDTHS)
@pytest.mark.parametrize("kind", ["gauss", "outliers", "one value", "front", "back", "sparse"])
def test_sources(N, bits, kind):
    rng = np.random.default_rng(bits)
    x = source(rng, kind, 5, 13 * N, N)
    check(x, "f32" if bits % 64 else "bf16", N, pvq.max_pulses(N, bits), 16 if kind == "gauss" else 6, 1 if kind == "front" else 0)


# one group short of and one beyond what a block of the encoder holds in a row, and the smallest row; rows that leave
# the last tile nearly empty
@pytest.mark.parametrize("N,bits", [(64, 192), (64, 256), (128, 384)])
@pytest.mark.parametrize("rows,G", [(1, 2), (33, 2), (3, 895), (2, 897), (150, 7)])
def test_shapes(N, bits, rows, G):
    rng = np.random.default_rng(rows * G)
    check(source(rng, "gauss", rows, G * N, N), "bf16", N, pvq.max_pulses(N, bits))


@pytest.mark.parametrize("N,bits", [(64, 192), (64, 256), (128, 384), (256, 768)])
def test_codes_on_thresholds(N, bits):
    """Points whose remainder after a random prefix is the largest or smallest of its kind: the number searched equals
    a threshold or is one above it, key bits the same as the threshold's."""
    K = pvq.max_pulses(N, bits)
    W = pvq.code_words(N, K)
    rng = np.random.default_rng(N + bits)
    points = []
    for n in range(32 * 8):
        a = np.abs(rng.standard_normal(N)) * K / (0.8 * N)
        y = np.zeros(N, dtype=np.int32)
        cut, left = int(rng.integers(0, N - 1)), K
        for i in range(cut):
            y[i] = min(left, int(a[i]), 127)
            left -= y[i]
        y[:cut] *= rng.choice([-1, 1], size=cut)
        at = cut if n % 2 else N - 1       # all that is left in the next place, or in the last
        y[at] = left if n % 4 < 2 else -left
        points.append(y)
    codes = np.stack([po.enumerate_point(y, K, W) for y in points]).reshape(8, 32, W)
    sidx = rng.integers(0, 120, size=(8, int(pvq.scale_row_stride(32, 16))), dtype=np.uint8)  # finite binary16 amplitudes
    rnorm = np.ones(8, dtype=np.float32)
    o_out, _ = po.decode(codes, sidx, rnorm, N, K, 16, None)
    table = pvq.build_count_table(N, K)
    out = pvq.decode(torch.from_numpy(codes.view(np.int32)).to(DEV), torch.from_numpy(sidx).to(DEV), torch.from_numpy(rnorm).to(DEV), N, K, 16,
                     table, None)
    torch.cuda.synchronize()
    assert np.array_equal(bf16_bits(out), o_out)


# position: value.  The pulses left at the beginning of a block of positions are 125 to 127 above the window's lower end, and the
# positions that follow are outside the window.
MANY_LEFT = [
    (64, 140, {1: -5, 48: 50, 52: 85}), (64, 140, {22: 4, 48: 51, 50: 85}), (64, 140, {29: 1, 46: 1, 48: 53, 54: -52, 62: 33}),
    (64, 165, {21: 23, 48: 36, 53: -46, 63: 60}), (64, 165, {2: -17, 9: 3, 17: -5, 48: 34, 51: 83, 63: 23}),
    (64, 169, {16: -33, 48: 30, 51: 20, 53: -35, 60: 51}), (64, 169, {21: -5, 32: 25, 48: 33, 50: 30, 51: 70, 59: 6}),
    (64, 180, {32: 39, 33: -4, 42: 39, 54: 7, 55: -16, 63: -75}), (64, 199, {7: -29, 22: 43, 61: -127}),
    (128, 187, {32: 34, 84: -1, 103: 14, 104: -68, 119: -70}), (128, 187, {3: -1, 6: 5, 40: -5, 66: 27, 92: -59, 95: 28, 97: 11, 109: 51}),
]


@pytest.mark.parametrize("N,K", sorted({p[:2] for p in MANY_LEFT}))
def test_many_pulses_left(N, K):
    """Points whose path is as far above the windows as an index outside of them says.  Each beside 31 ordinary ones: a warp
    looks closer for all its groups when it does for one."""
    W = pvq.code_words(N, K)
    rng = np.random.default_rng(N + K)
    points = []
    for value in (p[2] for p in MANY_LEFT if p[:2] == (N, K)):
        y = np.zeros((32, N), dtype=np.int32)
        y[:] = np.diff(np.arange(N + 1) * K // N)
        y *= rng.choice([-1, 1], size=y.shape).astype(np.int32)
        y[11] = 0
        y[11, list(value)] = list(value.values())
        points.append(y)
    codes = np.stack([[po.enumerate_point(y, K, W) for y in tile] for tile in points])
    rows = len(points)
    sidx = rng.integers(0, 120, size=(rows, int(pvq.scale_row_stride(32, 16))), dtype=np.uint8)  # finite binary16 amplitudes
    rnorm = np.ones(rows, dtype=np.float32)
    o_out, _ = po.decode(codes, sidx, rnorm, N, K, 16, None)
    out = pvq.decode(torch.from_numpy(codes.view(np.int32)).to(DEV), torch.from_numpy(sidx).to(DEV), torch.from_numpy(rnorm).to(DEV), N, K, 16,
                     pvq.build_count_table(N, K), None)
    torch.cuda.synchronize()
    assert np.array_equal(bf16_bits(out), o_out)


def test_several_matrices_and_streams():
    N, bits, b = 64, 192, 6
    K = pvq.max_pulses(N, bits)
    W = pvq.code_words(N, K)
    table = pvq.build_count_table(N, K)
    rng = np.random.default_rng(3)
    items, want = [], []
    for rows, G in ((37, 5), (2, 64), (130, 3)):
        x = source(rng, "gauss", rows, G * N, N)
        edges, levels = pvq.build_scale_codebook(N, G, b)
        want.append(po.encode(x, N, K, b, edges.cpu().numpy(), W=W))
        codes, sidx, rnorm = pvq.alloc_encoded(rows, G, W, b)
        items.append(dict(x=torch.from_numpy(x).to(DEV), codes=codes, scale_idx=sidx, row_norm=rnorm, edges=edges, levels=levels, cols=G * N,
                          out=torch.empty((rows, G * N), dtype=torch.bfloat16, device=DEV)))
    torch.cuda.synchronize()
    with torch.cuda.stream(torch.cuda.Stream()):
        pvq.encode_batched(items, torch.float32, N, K, b, table)
        pvq.decode_batched(items, N, K, b, table)
    torch.cuda.synchronize()
    for it, o in zip(items, want):
        assert np.array_equal(as_u32(it["codes"]), o[0]) and np.array_equal(it["scale_idx"].cpu().numpy(), o[1])
        assert np.array_equal(bf16_bits(it["out"]), po.decode(*o, N, K, b, it["levels"].cpu().numpy())[0])


def test_more_tables_than_are_kept():
    """Ten pulse counts, then the first one's table again: its windowed tables are gone, the calls go on without."""
    N = 64
    K0 = pvq.max_pulses(N, 192)
    first = pvq.build_count_table(N, K0)
    for K in range(K0 - 10, K0):
        pvq.build_count_table(N, K)
    rng = np.random.default_rng(9)
    x = source(rng, "gauss", 3, 4 * N, N)
    o = po.encode(x, N, K0, 16, None, W=6)
    codes, sidx, rnorm = pvq.encode(torch.from_numpy(x).to(DEV), N, K0, 16, first, None)
    out = pvq.decode(codes, sidx, rnorm, N, K0, 16, first, None)
    torch.cuda.synchronize()
    assert np.array_equal(as_u32(codes), o[0]) and np.array_equal(bf16_bits(out), po.decode(*o, N, K0, 16, None)[0])
    check(x, "f32", N, K0)


# 2 K + 2 = 112 is the last that rows of 112 entries hold; wide rows of 4, 13 and 0 positions' worth of upper halves
@pytest.mark.parametrize("N,K", [(32, 32), (32, 55), (32, 56), (16, 40), (64, 31), (32, 18)])
def test_encoder_tables(N, K):
    rng = np.random.default_rng(K)
    check(source(rng, "outliers", 7, 19 * N, N), "bf16", N, K, 5)
