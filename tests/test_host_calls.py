"""The device memory that a context keeps, and what it launches, on the CPU: the
library runs with a stand-in for the CUDA runtime (fake_cudart.cpp) that counts
its calls and holds a budget of device memory.  Each scenario runs in a process of its own, which
the stand-in is preloaded into."""
import ctypes
import os
import shutil
import subprocess
import sys
import threading
from pathlib import Path

import numpy as np
import pytest

HERE = Path(__file__).resolve().parent
ROOT = HERE.parent
MiB = 1 << 20


def _fake():
    f = ctypes.CDLL(None)
    f.fake_used.restype = ctypes.c_size_t
    f.fake_total.argtypes = [ctypes.c_size_t]
    f.fake_calls.argtypes = [ctypes.c_char_p]
    f.cudaMallocHost.argtypes = [ctypes.POINTER(ctypes.c_void_p), ctypes.c_size_t]
    return f


def _calls(f, name):
    return f.fake_calls(name.encode())


def _elsewhere(fn, *args):
    """A call on another thread (whose CUDA errors are its own)."""
    t = threading.Thread(target=fn, args=args)
    t.start()
    t.join()


def free_during_a_capture(bh, f):
    """While any stream of the device is captured, the device cannot be
    synchronised, so nothing shows that a freed handle's memory is idle: no later
    call may get it before a synchronisation succeeds."""
    ctx = bh.bh_create(0, 0)
    make = {"tables": lambda: bh.bh_precompute_tables(ctx, 66, 10, 6),
            "cube": lambda: bh.bh_build_star_cubemap(ctx, np.zeros((0, 5), np.float32), 64, 1)}
    free = {"tables": bh.bh_tables_free, "cube": bh.bh_cubemap_free}
    for kind in make:
        free[kind](make[kind]())  # kept, and idle
        f.fake_clear()
        first = make[kind]()
        assert _calls(f, "cudaMalloc") == 0  # the kept memory
        f.fake_capture(1)
        _elsewhere(free[kind], first)
        second = make[kind]()
        assert _calls(f, "cudaMalloc") == 1, kind  # not the memory of `first`
        third = make[kind]()
        assert _calls(f, "cudaMalloc") == 2, kind
        assert _calls(f, "cudaFree") == 0
        free[kind](third)  # the error of its synchronisation stays with it
        fourth = make[kind]()
        assert _calls(f, "cudaMalloc") == 3, kind
        f.fake_capture(0)
        f.fake_clear()
        free[kind](second)  # synchronises: first, second and third are idle
        handles = [fourth] + [make[kind]() for _ in range(3)]
        assert _calls(f, "cudaMalloc") == 0, kind
        for h in handles:
            free[kind](h)
    # what waits for a synchronisation is bounded with the rest
    maps = [bh.bh_build_star_cubemap(ctx, np.zeros((0, 5), np.float32), 1024, 1) for _ in range(12)]  # 69 MB each
    f.fake_capture(1)
    for m in maps:
        bh.bh_cubemap_free(m)
    assert f.fake_used() <= 512 * MiB + 16 * MiB
    f.fake_capture(0)
    bh.bh_destroy(ctx)
    assert f.fake_used() == 0


class _DeviceStars:
    """n stars in device memory, as the binding sees them."""
    is_cuda, dtype = True, np.dtype(np.float32)

    def __init__(self, n):
        self.shape = (n, 5)

    def is_contiguous(self):
        return True

    def data_ptr(self):
        return 1 << 30


WAITS = ("cudaDeviceSynchronize", "cudaStreamSynchronize", "cudaEventSynchronize", "cudaFree")


def builds_only_enqueue(bh, f):
    """Scratch that cannot be kept goes back in the order of its stream: no call
    that waits for the device, whatever the scratch's size and however full the
    kept memory is."""
    ctx = bh.bh_create(0, 0)
    fill = [bh.bh_build_star_cubemap(ctx, _DeviceStars(0), 1024, 1) for _ in range(7)]  # 69 MB each
    for full in (False, True):
        if full:
            for m in fill:
                bh.bh_cubemap_free(m)
        for n in (1000, 1_000_000, 12_000_000):  # 48 bytes of scratch each
            f.fake_clear()
            cube = bh.bh_build_star_cubemap(ctx, _DeviceStars(n), 64, 1, 1)
            tables = bh.bh_precompute_tables(ctx, 66, 10, 6, bh.BH_F32, 1)
            assert [w for w in WAITS if _calls(f, w)] == [], (full, n)
            bh.bh_cubemap_free(cube)
            bh.bh_tables_free(tables)
            assert f.fake_used() <= 512 * MiB + 16 * MiB + (0 if full else 7 * 71 * MiB)
    bh.bh_destroy(ctx)
    assert f.fake_used() == 0


def kept_memory_follows_the_work(bh, f):
    """Memory kept for sizes that are no longer asked for makes room for what is, and
    the stream-ordered allocator, whose first use costs a process 2 ms, is only
    used for scratch that there is no room for."""
    ctx = bh.bh_create(0, 0)
    for m in [bh.bh_build_star_cubemap(ctx, _DeviceStars(0), 1024, 1) for _ in range(8)]:
        bh.bh_cubemap_free(m)
    bh.bh_tables_free(bh.bh_precompute_tables(ctx, 66, 10, 6))
    assert _calls(f, "cudaMallocAsync") == 0
    for face, n in ((2048, 100), (512, 2_000_000), (512, 3_000_000), (512, 1_000_000), (2048, 7_000_000)):
        for _ in range(3):
            f.fake_clear()
            m = bh.bh_build_star_cubemap(ctx, _DeviceStars(n), face, 1)
            bh.bh_cubemap_free(m)
            f.cudaDeviceSynchronize()  # the stream-ordered allocator keeps nothing past it
            assert f.fake_used() <= 512 * MiB + MiB
        fits = 8 * bh.bh_cubemap_records(face) + 48 * n < 480 * MiB
        assert _calls(f, "cudaMalloc") == 0 and _calls(f, "cudaMallocAsync") == (0 if fits else 1), (face, n)
    bh.bh_destroy(ctx)
    assert f.fake_used() == 0


def allocations_take_the_kept_memory(bh, f):
    """Every allocation of a context that finds the device full gets the memory
    that the context keeps, whatever it is for."""
    from paper_2010_08735_gb300 import synth
    frame = 1 << 32  # an output in device memory
    cam, small = synth.camera(6.0, 85.0, width=1920, height=1080), synth.camera(6.0, 85.0, width=8, height=4)
    disc, sh = synth.disc(), bh.make_shading(1.0, 0.05)

    class Pinned:
        dtype = np.dtype(np.float32)

        def __init__(self):
            self.p = ctypes.c_void_p()
            f.cudaMallocHost(ctypes.byref(self.p), 1920 * 1080 * 16)

        def is_contiguous(self):
            return True

        def numel(self):
            return 1920 * 1080 * 4

        def data_ptr(self):
            return self.p.value

    def orbits(ctx, t):
        bh.bh_render_orbits(ctx, t, None, 1, frame, disc, sh, [frame])

    def autotune(ctx, t):
        f.fake_clear()
        bh.bh_autotune_batch(ctx, t, None, [small] * 1000, disc, sh, [frame] * 1000)
        assert _calls(f, "cudaMalloc") == 3  # the flush buffer, refused once, and the cameras

    calls = {
        "bloom": lambda ctx, t: bh.bh_bloom(ctx, frame, frame, 1920, 1080, np.ones(7) / 7),
        "to host": lambda ctx, t: bh.bh_render_to_host(ctx, t, None, cam, disc, sh,
                                                       np.zeros((1080, 1920, 4), np.float32)),
        "to host, in flight": lambda ctx, t: bh.bh_render_to_host_async(ctx, t, None, cam, disc, sh, Pinned(), False),
        "batch": lambda ctx, t: bh.bh_render_batch(ctx, t, None, [small] * 100, disc, sh, [frame] * 100),
        "autotune": autotune,
        "orbits": orbits,
        "particles": lambda ctx, t: bh.bh_disc_particles_free(
            bh.bh_disc_particles_create(ctx, synth.disc_particles(256, 5))),
        "served": lambda ctx, t: bh.bh_serve_submit(ctx, t, None, 0, small, disc, sh, frame),
        "tables": lambda ctx, t: bh.bh_tables_free(bh.bh_precompute_tables(ctx, 512, 64, 32)),
        "map": lambda ctx, t: bh.bh_cubemap_free(bh.bh_build_star_cubemap(ctx, _DeviceStars(10_000_000), 64, 1)),
    }
    for name, call in calls.items():
        for held in (False, True):  # kept as idle, or freed while nothing could be waited for
            ctx = bh.bh_create(0, 0)
            t = bh.bh_precompute_tables(ctx, 66, 10, 6)
            maps = [bh.bh_build_star_cubemap(ctx, _DeviceStars(0), 1024, 1) for _ in range(7)]
            f.fake_capture(int(held))
            for m in maps:
                bh.bh_cubemap_free(m)
            f.fake_capture(0)
            f.fake_total(f.fake_used() + 64)
            try:
                call(ctx, t)
            except bh.BhError as e:
                raise AssertionError((name, held)) from e
            bh.bh_tables_free(t)
            bh.bh_destroy(ctx)
            f.cudaDeviceSynchronize()
            assert f.fake_used() == 0, name
            f.fake_total(280 << 30)


def many_stars_in_little_memory(bh, f):
    """Where the device has no room for a sorted copy of the stars, the build makes
    do with the sums of the texels (240 bytes a level-0 texel)."""
    for face, n, room in ((128, 20_000_000, 32 * MiB), (64, 1_000_000, 16 * MiB), (8192, 1_000_000, 100 * MiB)):
        ctx = bh.bh_create(0, 0)
        records = 8 * bh.bh_cubemap_records(face)
        f.fake_total(f.fake_used() + records + records // 8 + room)
        cube = bh.bh_build_star_cubemap(ctx, _DeviceStars(n), face, 1)
        bh.bh_cubemap_free(cube)
        bh.bh_destroy(ctx)
        assert f.fake_used() == 0
        f.fake_total(280 << 30)


def tuned_launches_are_resident(bh, f):
    """The render's warps take their first tiles by their place in the grid, which
    is only even while every block of the launch is resident: 1,024 threads of 64
    registers an SM, in every shape that the autotuner tries."""
    from paper_2010_08735_gb300 import synth
    ctx = bh.bh_create(0, 0)
    t = bh.bh_precompute_tables(ctx, 66, 10, 6)
    cam = synth.camera(6.0, 85.0, width=1920, height=1080)
    bh.bh_autotune_batch(ctx, t, None, [cam] * 8, synth.disc(), bh.make_shading(1.0, 0.05), [1 << 32] * 8)
    assert f.fake_node_threads() == 152 * 1024
    bh.bh_tables_free(t)
    bh.bh_destroy(ctx)


SCENARIOS = [tuned_launches_are_resident, many_stars_in_little_memory, allocations_take_the_kept_memory, free_during_a_capture, builds_only_enqueue, kept_memory_follows_the_work]


@pytest.fixture(scope="module")
def fake_runtime(tmp_path_factory):
    from paper_2010_08735_gb300 import build
    build.build()
    cxx = shutil.which("g++")
    if cxx is None:
        pytest.skip("no C++ compiler")
    so = tmp_path_factory.mktemp("fake") / "libfake_cudart.so"
    include = Path(build.nvcc()).resolve().parent.parent / "include"
    subprocess.run([cxx, "-std=c++17", "-O1", "-shared", "-fPIC", "-I", str(include), str(HERE / "fake_cudart.cpp"),
                    "-o", str(so)], check=True)
    return so


@pytest.mark.parametrize("scenario", [s.__name__ for s in SCENARIOS])
def test_host_calls(fake_runtime, scenario):
    r = subprocess.run([sys.executable, __file__, scenario], cwd=ROOT, capture_output=True, text=True, timeout=300,
                       env=dict(os.environ, LD_PRELOAD=str(fake_runtime)))
    assert r.returncode == 0, r.stdout + r.stderr


if __name__ == "__main__":
    sys.path.insert(0, str(ROOT))
    from paper_2010_08735_gb300 import bh
    {s.__name__: s for s in SCENARIOS}[sys.argv[1]](bh, _fake())
