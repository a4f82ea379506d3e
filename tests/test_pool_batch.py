"""The size of the batches that go through a pool of seeded particles, on the host (CPU only)."""
import ctypes
import os
import subprocess

import pytest

ROOT = os.path.dirname(os.path.dirname(os.path.abspath(__file__)))
CSRC = os.path.join(ROOT, "paper_1312_3691_gb300", "csrc")
CUDA_INC = os.path.join(os.environ.get("CUDA_HOME", "/usr/local/cuda"), "include")
MIB = 1 << 20


@pytest.fixture(scope="module")
def pool_batch(tmp_path_factory):
    d = tmp_path_factory.mktemp("pool")
    src, lib = d / "pool.cpp", d / "pool.so"
    src.write_text('#include "runtime.h"\n'
                   'extern "C" uint64_t batch(uint64_t n, uint64_t most, size_t room, uint64_t* entries, size_t* bytes) {'
                   ' *entries = tpmc::pool_entries(n, most, room);'
                   ' *bytes = tpmc::pool_bytes(*entries);'
                   ' return *entries ? tpmc::pool_batch(*entries, n, most) : 0; }\n')
    subprocess.check_call(["g++", "-O1", "-std=c++17", "-shared", "-fPIC", "-I", CSRC, "-I", CUDA_INC, str(src), "-o", str(lib)])
    f = ctypes.CDLL(str(lib)).batch
    f.restype = ctypes.c_uint64
    f.argtypes = [ctypes.c_uint64, ctypes.c_uint64, ctypes.c_size_t, ctypes.POINTER(ctypes.c_uint64),
                  ctypes.POINTER(ctypes.c_size_t)]

    def sizes(n, most, room):
        entries, size = ctypes.c_uint64(), ctypes.c_size_t()
        b = f(n, most, room, ctypes.byref(entries), ctypes.byref(size))
        return b, entries.value, size.value

    return sizes


@pytest.mark.parametrize("room", [24, 80, 160, 300, 536, 600, 1100, 1200, 2400, 4800, 20_000, 250_000])
@pytest.mark.parametrize("most", [1 << 25, 1 << 26])
def test_batches_are_long_and_fit(pool_batch, most, room):
    """A pool takes at most half of the room; a launch that it splits has batches of 2^23 particles and more (smaller
    ones lose to the launch that seeds inside the trace kernel); sizes are powers of two."""
    for n in (1, 2048, 2049, (1 << 22) - 1, 1 << 22, (1 << 22) + 1, 12_000_001, 1 << 23, (1 << 23) + 1, 10 ** 8, 1 << 34, 1 << 50):
        b, entries, size = pool_batch(n, most, room * MIB)
        assert entries & (entries - 1) == 0 and b <= most and b % 2048 == 0
        whole = 1 << max(12, (n - 1).bit_length())  # a pool for one batch
        if b == 0:
            assert 32 * (min(whole, 1 << 24) if n <= most else 1 << 24) * 1.01 > room * MIB / 2
            continue
        assert size <= room * MIB / 2
        halves = 1 if n <= b else 2
        assert halves * (32 * b + 4 * b // 32 + 255) <= size  # with each half's start rounded down to 256 bytes
        assert n <= b or b >= 1 << 23
        assert entries == whole if n <= b else entries == 2 * b
