"""Which launches a call makes, on the CPU: the library's host code (cat_api.cu,
cat_tune.cu) linked with a CUDA runtime and launchers that keep a record
(tests/host/fake_cuda.cpp), under which bit planes are preferred wherever the
host code asks about them."""
import ctypes
import json
import os
import subprocess

import pytest

from paper_2406_17284_gb300 import build, cat, inputs

CUDA_INCLUDE = os.path.join(os.path.dirname(os.path.dirname(build._nvcc())), "include")


class Host:
    """The C ABI on the fake runtime."""

    def __init__(self, lib):
        self.lib = lib

    def __getattr__(self, name):
        def call(*args):
            rc = getattr(self.lib, name)(*[ctypes.c_int64(a) if isinstance(a, int) else a for a in args])
            assert rc == cat.CAT_OK, (name, rc, self.lib.cat_last_error())
        return call

    def rc(self, name, *args):
        return getattr(self.lib, name)(*[ctypes.c_int64(a) if isinstance(a, int) else a for a in args])

    def grid(self, H, W, r, C=2, storage=0, boundary=0):
        h = ctypes.c_void_p()
        rule = cat.make_rule(**inputs.scaled_rule(r, C=C))
        self.cat_create_ex(H, W, ctypes.byref(rule), boundary, storage, ctypes.byref(h))
        return h

    def options(self, h):
        v = [ctypes.c_int32() for _ in range(6)]
        self.cat_get_options(h, *[ctypes.byref(x) for x in v])
        return dict(zip(("kernel", "dtype", "storage", "steps_per_launch", "tile", "window"), (x.value for x in v)))

    def log(self):
        out = ctypes.create_string_buffer(1 << 16)
        assert self.lib.fake_log(out, len(out)) >= 0
        return out.value.decode().split("\n")[:-1]


@pytest.fixture(scope="module")
def lib(tmp_path_factory):
    so = str(tmp_path_factory.mktemp("host") / "libcat_host.so")
    src = [os.path.join(build.CSRC, f) for f in ("cat_api.cu", "cat_tune.cu")]
    src.append(os.path.join(os.path.dirname(os.path.abspath(__file__)), "host", "fake_cuda.cpp"))
    cmd = ["g++", "-std=c++17", "-O1", "-shared", "-fPIC", "-fvisibility=hidden", "-I", CUDA_INCLUDE, "-I", build.CSRC,
           "-x", "c++", *src, "-o", so]
    subprocess.run(cmd, check=True)
    return ctypes.CDLL(so)


@pytest.fixture
def host(lib):
    h = Host(lib)
    lib.cat_last_error.restype = ctypes.c_char_p
    yield h
    lib.fake_fail(None)
    lib.fake_capturing(0)
    h.log()


# Buffers that no launch touches here: only their addresses and pitch matter.
A, B = 1 << 44, 1 << 45


@pytest.mark.parametrize("pitch,route", [((1 << 32) - 16, "planes u8 to u8"), (1 << 32, "tensor cores"),
                                         ((1 << 32) + 4096, "tensor cores")])
def test_pitches_that_the_bit_planes_take(host, pitch, route):
    """The bit-plane kernels multiply a row by a pitch of 32 bits; longer ones,
    which cat_bind accepts, go to the tensor cores, in every way to step."""
    h = host.grid(3, 200, 4)
    host.cat_bind(h, A, B, pitch)
    host.cat_step(h, 1, None)
    assert host.log() == [route]
    host.cat_step(h, 4, None)
    assert all((x == "tensor cores") == (route == "tensor cores") for x in host.log())
    host.cat_destroy(h)
    if route == "tensor cores":
        large = host.grid(8192, 8192, 4)   # enough cells for a batch to step on bit planes
        host.cat_bind(large, A, B, pitch)
        host.cat_batch_step((ctypes.c_void_p * 1)(large), 1, 8, None)
        assert "batch planes" not in host.log()
        host.cat_destroy(large)


@pytest.mark.parametrize("bound", [False, True])
def test_steps_of_a_callers_buffers_end_from_bytes_to_bytes(host, bound):
    """Several steps keep the states between as bits; on a caller's buffers the
    last one reads bytes, so that the other buffer holds the generation before.
    A batch does so only on buffers of the library's own."""
    h = host.grid(8192, 8192, 4)
    if bound:
        host.cat_bind(h, A, B, 8192)
    host.cat_step(h, 4, None)
    last = "planes u8 to u8" if bound else "planes bit1 to u8"
    assert host.log() == ["planes u8 to bit1", "planes bit1 to bit1", *(["planes bit1 to u8"] if bound else
                                                                        ["planes bit1 to bit1"]), last]
    host.cat_batch_step((ctypes.c_void_p * 1)(h), 1, 8, None)
    assert ("batch tiles" in host.log()) == bound
    host.cat_destroy(h)


def cache_line(H, W, r, **choice):
    key = f"H={H} W={W} r={r} C=2 nbhd=M boundary=0 storage=0 gpu=fake/152"
    return json.dumps({"key": key, **choice, "cell_updates_per_s": 1.0}) + "\n"


FP16_TILES = dict(kernel=cat.KERNEL_TCGEN05, dtype=cat.DTYPE_FP16, tile=128, window=160, steps_per_launch=1)


def test_the_autotuner_times_what_the_library_would_choose(host, tmp_path, monkeypatch):
    """Tuning again while CAT_AUTOTUNE_CACHE names an older, explicit choice:
    the candidate that leaves the options to the library is timed as that."""
    old, new = tmp_path / "old.jsonl", tmp_path / "new.jsonl"
    old.write_text(cache_line(64, 96, 4, **FP16_TILES))
    h = host.grid(64, 96, 4)
    monkeypatch.setenv("CAT_AUTOTUNE_CACHE", str(old))
    host.cat_autotune(h, 8, str(new).encode(), cat.CAT_TUNE_REMEASURE, None)
    line = json.loads(new.read_text())
    assert line["left"] == 1 and line["dtype"] == cat.DTYPE_FP8_E4M3
    assert line["cell_updates_per_s"] == pytest.approx(64 * 96 * 8 / 8e-3)   # eight launches of a millisecond
    assert host.options(h)["dtype"] == cat.DTYPE_FP8_E4M3
    host.log()
    host.cat_step(h, 1, None)
    assert host.log() == ["planes u8 to u8"]
    host.cat_destroy(h)


@pytest.mark.parametrize("left", [False, True])
def test_auto_takes_the_cached_choice(host, tmp_path, monkeypatch, left):
    """CAT_KERNEL_AUTO takes the choice that CAT_AUTOTUNE_CACHE names in place of
    the other arguments, also when that is to leave every option to the library."""
    cache = tmp_path / "tune.jsonl"
    default = dict(FP16_TILES, dtype=cat.DTYPE_FP8_E4M3, window=144)
    cache.write_text(cache_line(64, 96, 4, **FP16_TILES))
    if left:
        cache.write_text(cache.read_text() + cache_line(64, 96, 4, **default).replace("}", ', "left": 1}'))
    h = host.grid(64, 96, 4)
    host.cat_set_tile(h, 128, 128, 160)
    monkeypatch.setenv("CAT_AUTOTUNE_CACHE", str(cache))
    host.cat_set_options(h, cat.KERNEL_AUTO, cat.DTYPE_FP16, cat.STORE_U8, 4)
    assert host.options(h) == dict(default if left else FP16_TILES, storage=cat.STORE_U8)
    host.cat_step(h, 1, None)
    assert host.log() == ["planes u8 to u8" if left else "tensor cores"]
    host.cat_destroy(h)


@pytest.mark.parametrize("boundary,fails", [(0, "planes u8 to bit1"), (0, "planes bit1 to bit1"), (0, "planes bit1 to u8"),
                                            (1, "bit frame"), (1, "planes bit1 to u8")])
def test_steps_that_cannot_all_be_launched_leave_the_state(host, boundary, fails):
    """Several steps write bits over states, also in the buffer that holds the
    state: a kernel that cannot be loaded is found before the first launch."""
    h = host.grid(64, 96, 4, boundary=boundary)
    at, pitch = ctypes.c_void_p(), ctypes.c_int64()
    host.cat_state_ptr(h, ctypes.byref(at), ctypes.byref(pitch))
    host.lib.fake_fail(fails.encode())
    assert host.rc("cat_step", h, 5, None) == cat.CAT_ERR_CUDA
    assert host.log() == []
    now = ctypes.c_void_p()
    host.cat_state_ptr(h, ctypes.byref(now), ctypes.byref(pitch))
    assert now.value == at.value
    host.lib.fake_fail(None)
    host.cat_step(h, 5, None)
    assert host.log()[-1] == "planes bit1 to u8"
    host.cat_destroy(h)


def test_a_batch_asks_for_the_capture_only_where_it_matters(host):
    """The legacy stream has no capture status while another stream is captured
    (cudaErrorStreamCaptureImplicit): calls that launch nothing, or nothing that a
    capture changes, do not ask for it."""
    u8, bits = host.grid(64, 96, 4), host.grid(64, 96, 4, storage=cat.STORE_BIT1)
    host.lib.fake_capturing(906)
    host.cat_batch_step((ctypes.c_void_p * 1)(u8), 1, 0, None)
    host.cat_batch_step((ctypes.c_void_p * 1)(bits), 1, 2, None)
    assert host.rc("cat_batch_step", (ctypes.c_void_p * 2)(u8, u8), 2, 2, None) == cat.CAT_ERR_INVALID_ARG
    assert host.rc("cat_batch_step", (ctypes.c_void_p * 1)(u8), 1, 2, None) == cat.CAT_ERR_CUDA
    host.lib.fake_capturing(0)
    host.cat_destroy(u8)
    host.cat_destroy(bits)


@pytest.mark.parametrize("radii,n,planes", [((9, 9, 9, 9), 8, True), ((4, 4, 4, 10), 8, True), ((4, 4, 10, 10), 8, False),
                                            ((4, 4, 10, 10), 12, True), ((4, 10, 10, 10), 16, False), ((4,) * 4, 7, False)])
def test_batches_of_large_radii_keep_to_the_tiles(host, radii, n, planes):
    """The bit planes of a batch gain up to r = 9; larger radii may make up a
    quarter of the cells, or half of them from twelve steps on."""
    grids = [host.grid(3000, 3000, r) for r in radii]
    host.cat_batch_step((ctypes.c_void_p * 4)(*grids), 4, n, None)
    assert ("batch planes" in host.log()) == planes
    for g in grids:
        host.cat_destroy(g)


@pytest.mark.parametrize("W,planes", [(128, False), (2048, True)])
def test_batches_of_narrow_grids_keep_to_the_tiles(host, W, planes):
    grids = [host.grid((1 << 24) // W, W, 4) for _ in range(2)]
    host.cat_batch_step((ctypes.c_void_p * 2)(*grids), 2, 8, None)
    assert ("batch planes" in host.log()) == planes
    for g in grids:
        host.cat_destroy(g)
