"""The host pipeline's order of copies, kernels, events and waits, followed on the CPU: its object is linked with stand-ins for
the CUDA runtime (``host_fake``) that log every call with the bytes that it reads and writes."""
import ctypes
import os
import shutil
import subprocess

import pytest

from paper_2502_16886_b200 import binding, build

HERE = os.path.dirname(os.path.abspath(__file__))
UNITS, ROWS = 3, 5


@pytest.fixture(scope="module")
def built(tmp_path_factory):
    build.build()
    d = tmp_path_factory.mktemp("host_fake")
    obj, lib = str(d / "fake_launch.o"), str(d / "libhostfake.so")
    fake, cuda = os.path.join(HERE, "host_fake"), os.path.dirname(os.path.dirname(os.path.realpath(shutil.which(build._nvcc()))))
    subprocess.run([build._nvcc()] + build.NVCC_FLAGS + ["-c", os.path.join(fake, "fake_launch.cu"), "-o", obj], check=True)
    subprocess.run(["g++", "-shared", "-fPIC", "-std=c++17", "-Wl,-Bsymbolic", "-I", os.path.join(cuda, "include"), "-o", lib,
                    os.path.join(fake, "fake_runtime.cpp"), obj, os.path.join(build.OBJ_DIR, "host_pipeline.o")], check=True)
    return lib


class Pipeline:
    """The linked pipeline with its own copy of the pool (a library file of its own)."""

    def __init__(self, built, tmp_path):
        path = str(tmp_path / "lib.so")
        with open(built, "rb") as f, open(path, "wb") as g:
            g.write(f.read())
        self.lib = ctypes.CDLL(path)
        self.lib.fake_log.restype = ctypes.c_char_p
        self.lib.fake_live.restype = ctypes.c_long
        self.memory = []

    def _buffer(self, n):
        self.memory.append(ctypes.create_string_buffer(n + 256))
        return (ctypes.addressof(self.memory[-1]) + 255) & ~255

    def run(self, layers=4, rank=binding.RANK_POSITION, status=0):
        p = binding.Params(num_seqs=1, num_q_heads=UNITS, num_kv_heads=UNITS, head_dim=64, window=1, sink=0, threshold=0.01, rank_mode=rank,
                           dtype=binding.DTYPE_F32, kv_tokens=8, k_strides=(0, 64, 512), v_strides=(0, 64, 512)).c_struct()
        kv, total, cap = UNITS * 512, 8, UNITS * 8
        need = ctypes.c_size_t(0)
        self.lib.refree_host_pipeline_arena_size(ctypes.byref(p), ctypes.c_int64(total), ctypes.c_int64(kv), ctypes.c_int64(cap), ctypes.byref(need))
        arena = self._buffer(need.value)
        sizes = [UNITS * 256, kv * 4, kv * 4, cap * 256, cap * 256, UNITS * 4, (UNITS + 1) * 8]
        arrays = [(ctypes.c_void_p * layers)(*[self._buffer(n) for _ in range(layers)]) for n in sizes]
        self.lib.fake_reset(ctypes.c_longlong(ROWS), status)
        rc = self.lib.refree_compress_layers_host(
            ctypes.byref(p), layers, *arrays[:3], ctypes.c_int64(kv), ctypes.c_void_p(self._buffer(4)), ctypes.c_void_p(self._buffer(4)),
            ctypes.c_int64(total), *arrays[3:5], ctypes.c_int64(cap), *arrays[5:7], ctypes.c_void_p(arena), ctypes.c_size_t(need.value))
        return rc, self.lib.fake_log().decode().splitlines()


@pytest.fixture
def pipeline(built, tmp_path):
    return Pipeline(built, tmp_path)


def races(log):
    """Pairs of operations of two streams that touch the same bytes, one of them writing, with nothing that orders them."""
    streams, events, host, ops, found = {}, {}, {}, [], []

    def join(a, b):
        for s, n in b.items():
            a[s] = max(a.get(s, 0), n)
    for line in log:
        w = line.split()
        if w[0] == "op":
            at = streams.setdefault(w[1], {})
            join(at, host)
            at[w[1]] = at.get(w[1], 0) + 1
            what = [(w[i], int(w[i + 1]), int(w[i + 2])) for i in range(3, len(w) - 2, 3)]
            for s, n, other, name in ops:
                if s == w[1] or at.get(s, 0) >= n:
                    continue
                for kind, a, la in what:
                    for kind2, b, lb in other:
                        if "w" in (kind, kind2) and a < b + lb and b < a + la:
                            found.append((name, w[2], a))
            ops.append((w[1], at[w[1]], what, w[2]))
        elif w[0] == "record":
            at = streams.setdefault(w[1], {})
            join(at, host)
            events[w[2]] = dict(at)
        elif w[0] == "wait":
            join(streams.setdefault(w[1], {}), events.get(w[2], {}))
        elif w[0] == "hostwait":
            join(host, events.get(w[1], {}))
        elif w[0] == "hostsync":
            join(host, streams.get(w[1], {}))
    return found


@pytest.mark.parametrize("rank", [binding.RANK_POSITION, binding.RANK_SCORE])
@pytest.mark.parametrize("layers", [1, 2, 5])
def test_no_two_streams_touch_the_same_bytes_unordered(pipeline, rank, layers):
    rc, log = pipeline.run(layers=layers, rank=rank)
    assert rc == 0 and sum(line.split()[2] == "rows" for line in log if line.startswith("op")) == 2 * layers
    assert races(log) == []


def test_kept_streams_serve_the_next_call(pipeline):
    pipeline.run()
    first = pipeline.lib.fake_live()
    rc, log = pipeline.run()
    assert rc == 0 and pipeline.lib.fake_live() == first and not any(line.startswith(("pinned", "destroy")) for line in log)


@pytest.mark.parametrize("status,error", [(binding.DEV_CAPACITY, binding.ERR_CAPACITY), (0, 0)])
def test_streams_of_a_context_that_is_gone_are_not_touched(pipeline, status, error):
    """After a reset of the device a call makes its own streams, once; what was kept before is neither used nor destroyed."""
    assert pipeline.run(status=status)[0] == error
    for _ in range(2):
        pipeline.lib.fake_new_context()
        for made in (True, False):
            rc, log = pipeline.run()
            assert rc == 0 and not any("dead" in line for line in log)
            assert any(line.startswith("pinned") for line in log) == made
