"""The library's host code on a CUDA runtime without a GPU (tests/fake_cudart.cpp): who owns the memory that launches are
given, what is waited for, who waits for whom."""
import ctypes as C
import glob
import os
import shutil
import subprocess
import sys
import threading

import pytest

from oracle import pvq_pyref as pr
from paper_2410_16926_b200 import build as lib_build
from paper_2410_16926_b200 import pvq

import test_long_decode

ROOT = os.path.dirname(os.path.dirname(os.path.abspath(__file__)))
P = 1 << 20  # an address, aligned; nothing is read there
CAPTURED, PLAIN = C.c_void_p(0x100), C.c_void_p(0x200)


@pytest.fixture(scope="module")
def fake_lib(tmp_path_factory):
    """The library's objects linked with the fake runtime."""
    objs = sorted(glob.glob(os.path.join(lib_build.OBJDIR, "*.o")))
    cuda = os.environ.get("CUDA_HOME", "/usr/local/cuda")
    want = {f[:-3] for f in os.listdir(lib_build.CSRC) if f.endswith(".cu")}
    objs = [o for o in objs if os.path.basename(o)[:-2] in want]
    if len(objs) != len(want) or shutil.which("g++") is None:
        pytest.skip("needs the library's objects (python -m paper_2410_16926_b200.build) and g++")
    tmp = tmp_path_factory.mktemp("fake")
    out = str(tmp / "libpvq_fake.so")
    subprocess.run(["g++", "-std=c++17", "-O1", "-shared", "-fPIC", "-pthread", "-Wl,-Bsymbolic", "-Wl,-s", "-I", os.path.join(cuda, "include"),
                    os.path.join(ROOT, "tests", "fake_cudart.cpp")] + objs + ["-o", out], check=True)
    return out


@pytest.fixture()
def fake(fake_lib, tmp_path):
    """A fresh instance for every test (the library's caches live as long as the process)."""
    copy = str(tmp_path / "lib.so")
    shutil.copyfile(fake_lib, copy)
    L = load(copy)
    os.unlink(copy)
    return L


def load(path):
    L = C.CDLL(path)
    i32, i64, vp = C.c_int, C.c_int64, C.c_void_p
    L.pvq_build_count_table.argtypes = [i32, i32, vp, C.c_size_t, vp]
    L.pvq_encode.argtypes = [vp, i32, i64, i64, i64, i32, i32, i32, vp, vp, vp, vp, vp, vp]
    L.pvq_decode.argtypes = [vp, vp, vp, i64, i64, i32, i32, i32, vp, vp, vp, i64, vp, vp]
    L.pvq_encode_amp.argtypes = [vp, i32, i64, i64, i64, i32, i32, i32, i32, vp, vp, vp, vp, vp, vp]
    L.pvq_roundtrip.argtypes = [vp, i32, i64, i64, i64, i32, i32, i32, vp, vp, vp, vp, i64, vp]
    L.pvq_rotate_roundtrip.argtypes = [vp, i32, i64, i64, i64, i32, vp, i32, i32, i32, vp, vp, vp, vp, i64, vp]
    L.fake_capture.argtypes = [vp, i32]
    L.fake_launch_name.restype = C.c_char_p
    L.fake_launch_table.restype = C.c_uint64
    L.fake_live.argtypes = [C.c_uint64]
    return L


def build(L, N, K, stream=PLAIN):
    return L.pvq_build_count_table(N, K, P, 1 << 40, stream)


def encode(L, N, K, stream=PLAIN, rows=8, G=4):
    return L.pvq_encode(P, 1, rows, G * N, G * N, N, K, 16, P, None, P, P, P, stream)


def decode(L, N, K, stream=PLAIN, rows=8, G=4):
    return L.pvq_decode(P, P, P, rows, G * N, N, K, 16, P, None, P, G * N, None, stream)


def roundtrip(L, N, K, rows, cols, bf16=True, block=0):
    dtype = 1 if bf16 else 0
    if block:
        return L.pvq_rotate_roundtrip(P, dtype, rows, cols, cols, block, P, N, K, 16, P, None, None, P, cols, PLAIN)
    return L.pvq_roundtrip(P, dtype, rows, cols, cols, N, K, 16, P, None, None, P, cols, PLAIN)


def last_tables(L):
    """Name and tables of the last launch: ('', ...) unless it was a windowed kernel."""
    i = L.fake_launches() - 1
    name = L.fake_launch_name(i).decode()
    return name, [L.fake_launch_table(i, w) for w in (0, 1)]


@pytest.mark.parametrize("call", [encode, decode])
@pytest.mark.parametrize("N,bits", [(64, 192), (128, 384)])
def test_tables_of_a_captured_call_stay(fake, call, N, bits):
    """A graph replays a captured launch with the addresses it was given: they are not freed for other tables."""
    K = pvq.max_pulses(N, bits)
    assert build(fake, N, K) == 0
    fake.fake_capture(CAPTURED, 1)
    assert call(fake, N, K, CAPTURED) == 0
    fake.fake_capture(CAPTURED, 0)
    name, tables = last_tables(fake)
    assert "window" in name and all(fake.fake_live(t) for t in tables)
    for k in range(K - 12, K):
        assert build(fake, N, k) == 0
    assert all(fake.fake_live(t) for t in tables)
    # and the number kept stays bounded, also when every one of them has been captured
    assert fake.fake_allocations() <= 8
    for k in range(K - 30, K + 1):
        assert build(fake, N, k) == 0
        fake.fake_capture(CAPTURED, 1)
        assert call(fake, N, k, CAPTURED) == 0
        fake.fake_capture(CAPTURED, 0)
    assert fake.fake_allocations() <= 8 and all(fake.fake_live(t) for t in tables)
    assert call(fake, N, K) == 0 and last_tables(fake)[1] == tables


def test_tables_that_no_capture_holds_make_room(fake):
    K = pvq.max_pulses(64, 192)
    for k in range(K - 12, K + 1):
        assert build(fake, 64, k) == 0 and decode(fake, 64, k) == 0
        name, tables = last_tables(fake)
        assert "window" in name and all(fake.fake_live(t) for t in tables)
    assert fake.fake_allocations() == 8


def test_a_hot_call_never_frees(fake):
    """Tables that make room while another thread is launching with them stay until it is through, and that
    thread does not free them (cudaFree waits for the device and ends a capture)."""
    K = pvq.max_pulses(64, 192)
    assert build(fake, 64, K) == 0
    fake.fake_forget_frees()
    fake.fake_hold(1, 0)
    status = []
    launching = threading.Thread(target=lambda: status.append(decode(fake, 64, K)))
    launching.start()
    assert fake.fake_wait_until_held(20)
    for k in range(K - 9, K):
        assert build(fake, 64, k) == 0
    fake.fake_hold(0, 0)
    launching.join()
    assert status == [0]
    name, tables = last_tables(fake)
    assert "window" in name and all(fake.fake_live(t) for t in tables)
    assert fake.fake_frees_by_others() == 0
    for k in range(K - 20, K - 9):
        assert build(fake, 64, k) == 0
    assert fake.fake_allocations() == 8 and fake.fake_frees() == 1 + 9 + 11 - 8 and fake.fake_frees_by_others() == 0


@pytest.mark.parametrize("N,bits", [(64, 192), (128, 384), (256, 768)])
def test_tables_are_on_the_device_before_a_launch_can_find_them(fake, N, bits):
    """Streams that do not wait for the legacy stream follow: nothing may still be on its way when the build returns."""
    K = pvq.max_pulses(N, bits)
    assert build(fake, N, K) == 0
    assert fake.fake_uploads_pending() == 0
    assert decode(fake, N, K) == 0 and "window" in last_tables(fake)[0]


def test_a_hot_call_does_not_wait_for_another_threads_build(fake):
    """Tables are computed, allocated, copied and freed (which waits for the device) beside the calls of other threads."""
    K = pvq.max_pulses(64, 192)
    assert build(fake, 64, K) == 0
    fake.fake_hold(0, 1)
    builder = threading.Thread(target=build, args=(fake, 64, K - 1))
    builder.start()
    assert fake.fake_wait_until_held(20)
    done = []
    calls = [threading.Thread(target=lambda n=n, k=k: done.append(decode(fake, n, k)), daemon=True) for n, k in ((64, K), (64, K - 1), (32, 50))]
    for c in calls:
        c.start()
    for c in calls:
        c.join(20)
    finished = len(done)
    fake.fake_hold(0, 0)
    builder.join()
    assert finished == 3 and done == [0, 0, 0]


def test_which_launches_may_start_early(fake):
    """Kernels that fill the GPU and read tables through L1 start when the one before has ended; the others early."""
    def early():
        return bool(fake.fake_launch_early(fake.fake_launches() - 1))
    K = pvq.max_pulses(64, 320)          # tables in global memory, both ways
    assert decode(fake, 64, K, rows=4096, G=64) == 0 and not early()
    assert decode(fake, 64, K) == 0 and not early()
    assert encode(fake, 64, K, rows=256, G=64) == 0 and not early()  # two lanes a group
    assert encode(fake, 64, K, rows=255, G=64) == 0 and early()
    assert decode(fake, 32, 50, rows=4096, G=128) == 0 and early()
    assert encode(fake, 32, 50, rows=4096, G=128) == 0 and early()


@pytest.mark.parametrize("N,K,rows,G,lanes", [(8, 12, 1024, 512, 1), (16, 27, 1024, 256, 1), (32, 50, 1024, 128, 1), (64, 26, 1024, 64, 2),
                                              (32, 1000, 600, 128, 1)])
def test_few_rows_still_fill_the_gpu(fake, N, K, rows, G, lanes):
    """The encoder's teams: a matrix of medium size is given as many threads as it has groups (lanes), up to what an SM
    holds, not one warp a row that takes the row's chunks one after the other."""
    assert encode(fake, N, K, rows=rows, G=G) == 0
    i = fake.fake_launches() - 1
    assert "encode_lanes" in fake.fake_launch_name(i).decode()
    threads = fake.fake_launch_grid(i) * fake.fake_launch_block(i)
    assert threads >= 0.75 * min(rows * G * lanes, 148 * 768)


@pytest.mark.parametrize("N,K", test_long_decode.SETTINGS)
def test_decoding_launches_that_rewrite_the_buckets(fake, N, K):
    """The sizes that test_long_decode.py decodes take the kernels for launches of several rounds, with the table of the last
    four positions where N = 32 has it; launches half as long do not."""
    rows, quads = test_long_decode.long_rows(N, K, 64, 148), 0
    for n, long_launch in ((rows, True), (int(rows / 2.1), False)):
        assert decode(fake, N, K, rows=n, G=64) == 0
        i = fake.fake_launches() - 1
        name = fake.fake_launch_name(i).decode()
        assert "decode_search" in name and ("ELb1EE" in name) == long_launch and ("ELb0EE" in name) != long_launch
        tables = fake.fake_launch_shared(i) - 2 * (N + 4) * fake.fake_launch_block(i)  # (slots of two groups a thread)
        quads = tables if long_launch else quads - tables
    assert quads in (0, 4 * pr.count_table(4, 16)[4][16]) and (quads != 0 or (N, K) != (32, 22))


@pytest.mark.parametrize("K,G,bf16,amp_mode,bufs", [(50, 4096, 1, 0, 2), (50, 4096, 1, 1, 2), (63, 4096, 1, 0, 2), (63, 128, 1, 1, 1), (50, 128, 0, 0, 1)])
def test_one_input_buffer_only_for_more_teams(fake, K, G, bf16, amp_mode, bufs):
    """Long encoder launches: a team gives up the buffer that its next input is asked for ahead only where more teams fit
    without.  (Rows of 4096 groups: as many either way.)"""
    assert fake.pvq_encode_amp(P, bf16, 2000000 // G, G * 32, G * 32, 32, K, 8, amp_mode, P, P, P, P, P, PLAIN) == 0
    i = fake.fake_launches() - 1
    assert "encode_lanes" in fake.fake_launch_name(i).decode()
    assert fake.fake_launch_teams(i, 2) == bufs


@pytest.mark.parametrize("bf16", [True, False])
@pytest.mark.parametrize("N,K,rows,cols,block", [(32, 22, 100, 8192, 8192), (32, 22, 600, 2048, 2048), (32, 22, 100, 8192, 0), (128, 155, 256, 4096, 0),
                                                 (16, 27, 100, 1664, 0), (32, 22, 1, 512, 0), (32, 22, 2000, 512, 512)])
def test_a_round_trip_of_few_blocks_spreads(fake, N, K, rows, cols, block, bf16):
    """No more blocks fit an SM than its share of the launch."""
    assert roundtrip(fake, N, K, rows, cols, bf16, block) == 0
    i = fake.fake_launches() - 1
    grid, shared = fake.fake_launch_grid(i), fake.fake_launch_shared(i)
    share = -(-grid // 148)
    assert shared <= 232448 and 233472 // (shared + 1024) <= share or grid >= 148 * (1024 // fake.fake_launch_block(i))


@pytest.mark.parametrize("N,K", [(16, 27), (32, 22), (64, 199), (128, 155)])
@pytest.mark.parametrize("cols", [1152, 1664, 2304, 2560, 3072, 3328, 3584, 4096])
def test_round_trip_blocks_waste_few_lanes(fake, N, K, cols):
    """bf16, rows enough: the lanes without values are no more than in the best block of up to 256 threads, but for the 3 %
    that those above 128 cost."""
    rows, lanes = (1 << 24) // cols, cols // min(N, 32)

    def cost(threads):
        return -(-rows // (threads // lanes)) * threads

    assert roundtrip(fake, N, K, rows, cols) == 0
    threads = fake.fake_launch_block(fake.fake_launches() - 1)
    need = -(-lanes // 32) * 32
    assert cost(threads) <= 1.03 * min(cost(t) for t in range(max(64, need), max(256, need) + 1, 32))


@pytest.mark.parametrize("call,N,K", [(decode, 32, 50), (encode, 32, 50), (decode, 64, 96), (decode, 64, 300), (encode, 64, 300)])
def test_a_failed_launch_is_reported_once(fake, call, N, K):
    assert build(fake, 64, 96) == 0
    fake.fake_fail_launches(701)
    assert call(fake, N, K) == 5 and fake.pvq_last_cuda_error() == 701
    fake.fake_fail_launches(0)
    assert build(fake, 32, 22) == 0, "found the error of an earlier call"
    assert call(fake, N, K) == 0


OUT_OF_HOST_MEMORY = """
import resource, sys
sys.path.insert(0, sys.argv[2])
import test_host_fake_gpu as t
L = t.load(sys.argv[1])
K = t.pvq.max_pulses(256, 768)
assert t.build(L, 256, 8) == 0  # (the library's first call, with what it allocates once)
now = int(open("/proc/self/statm").read().split()[0]) * resource.getpagesize()
resource.setrlimit(resource.RLIMIT_AS, (now + (8 << 20), resource.RLIM_INFINITY))
assert t.build(L, 256, K) == 0
resource.setrlimit(resource.RLIMIT_AS, (resource.RLIM_INFINITY, resource.RLIM_INFINITY))
assert t.decode(L, 256, K) == 0 and "big" in t.last_tables(L)[0]
assert t.build(L, 256, K) == 0 and t.decode(L, 256, K) == 0 and "window" in t.last_tables(L)[0]
"""


def test_no_exception_leaves_a_build_without_host_memory(fake_lib):
    r = subprocess.run([sys.executable, "-c", OUT_OF_HOST_MEMORY, fake_lib, os.path.dirname(os.path.abspath(__file__))], cwd=ROOT,
                       env=dict(os.environ, PYTHONPATH=ROOT), capture_output=True, text=True, timeout=300)
    assert r.returncode == 0, (r.returncode, r.stderr[-2000:])
