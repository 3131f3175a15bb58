"""What the library's host side asks of the CUDA runtime: its objects linked against a stand-in runtime
(fake_cudart.cpp) that records launches instead of running them. Needs no GPU and touches none."""
import ctypes as C
import glob
import os
import shutil
import subprocess

import pytest

ROOT = os.path.dirname(os.path.dirname(os.path.abspath(__file__)))
N = 512


class Fake:
    """The library on the stand-in runtime, called with made-up device addresses."""

    def __init__(self, path, lib):
        self.dll = C.CDLL(path)
        for name, (res, args) in lib.SIGNATURES.items():
            fn = getattr(self.dll, name)
            fn.restype, fn.argtypes = res, args
        self.dll.fake_kernel.restype = C.c_char_p
        self.lib = lib
        self.buffers = []

    def field(self, samples):
        """Address of a 16-byte aligned "device" array of complex64 samples (never read or written)."""
        raw = C.create_string_buffer(8 * samples + 16)
        self.buffers.append(raw)
        return (C.addressof(raw) + 15) // 16 * 16

    def handle(self, device=0):
        h = C.c_void_p()
        assert self.dll.top_create(C.byref(h), device) == 0
        return h

    def grid(self, batch, ny, nx, pad=2.0):
        return C.byref(self.lib.TopGrid(batch, ny, nx, 8e-6, 8e-6, pad, 0, 0))

    def one(self, v):
        return self.lib.doubles([v])

    def launches(self):
        return [self.dll.fake_kernel(i).decode() for i in range(self.dll.fake_launches())]

    def error(self):
        return self.dll.top_last_error().decode()


@pytest.fixture(scope="module")
def fake(tmp_path_factory):
    from paper_2411_18591_gb300 import _lib, build
    build.build()
    objects = sorted(glob.glob(os.path.join(build.OUT_DIR, "*.o")))
    if len(objects) != len(glob.glob(os.path.join(build.CSRC, "*.cu"))):
        build.build(force=True)
        objects = sorted(glob.glob(os.path.join(build.OUT_DIR, "*.o")))
    cuda = os.path.join(os.path.dirname(os.path.dirname(shutil.which("nvcc") or "/usr/local/cuda/bin/nvcc")), "include")
    out = str(tmp_path_factory.mktemp("fake") / "libtop_fake.so")
    # -Bsymbolic: the stand-in's runtime calls also where a real one is loaded in the process
    subprocess.run(["g++", "-std=c++17", "-shared", "-fPIC", "-Wl,-Bsymbolic", "-I", build.CSRC, "-I", cuda,
                    os.path.join(ROOT, "tests", "fake_cudart.cpp"), *objects, "-o", out, "-lpthread"], check=True)
    return Fake(out, _lib)


@pytest.fixture(autouse=True)
def clean(fake):
    fake.dll.fake_waits_run_out(0)
    fake.dll.fake_reset()
    yield


def run_everywhere(fake, h):
    """Calls whose kernels need more than the 48 KB of shared memory that every launch may have."""
    x, y = fake.field(1), fake.field(1)
    lam, z = fake.one(5e-7), fake.one(0.02)
    stages = (fake.lib.TopStage * 2)()
    stages[0].z = stages[1].z = 0.02
    for batch, n in ((64, 256), (64, N), (32, 1024), (1, 4096), (1, 64), (4, 1021)):
        assert fake.dll.top_propagate(h, fake.grid(batch, n, n), x, y, lam, z, 1, None, None, None) == 0, (n, fake.error())
        if n not in (64, 1021):
            st = fake.dll.top_fused_chain(h, fake.grid(batch, n, n), x, y, None, 1, lam, 1, stages, 2, None)
            assert st == 0, (n, fake.error())


def test_kernels_are_set_up_on_every_device(fake):
    """A second device of the process gets the kernels' shared memory allowed as the first one did."""
    for device in (0, 1):
        fake.dll.fake_reset()
        run_everywhere(fake, fake.handle(device))
        n = fake.dll.fake_launches()
        assert n > 20
        assert not [fake.launches()[i] for i in range(n) if fake.dll.fake_refused(i)]
        # table kernels aside, everything ran where the handle is
        assert all(fake.dll.fake_device_of(i) == device for i in range(n))


def test_waits_that_run_out_are_reported(fake):
    """By the next call on the handle, or by top_check_waits without one; once; and for the no-alloc call too."""
    x, y = fake.field(1), fake.field(1)
    lam, z = fake.one(5e-7), fake.one(0.02)
    h, other = fake.handle(), fake.handle()
    call = lambda who: fake.dll.top_propagate(who, fake.grid(64, N, N), x, y, lam, z, 1, None, None, None)
    noalloc = lambda: fake.dll.top_propagate_noalloc(fake.grid(3, N, N), x, y, lam, z, 1, None)
    assert call(h) == call(other) == noalloc() == 0
    assert [fake.dll.top_check_waits(who) for who in (h, other, None)] == [0, 0, 0]
    fake.dll.fake_waits_run_out(1)
    assert call(h) == 0 and noalloc() == 0  # asynchronous: the calls themselves do not know
    fake.dll.fake_waits_run_out(0)
    assert fake.dll.top_check_waits(other) == 0  # a handle's own
    timeout = 5
    for who in (h, None):
        assert fake.dll.top_check_waits(who) == timeout
        assert "ran out" in fake.error()
        assert fake.dll.top_check_waits(who) == 0
    fake.dll.fake_waits_run_out(1)
    assert call(h) == 0 and noalloc() == 0
    fake.dll.fake_waits_run_out(0)
    fake.dll.fake_reset()
    assert call(h) == timeout and noalloc() == timeout
    assert fake.dll.fake_launches() == 0
    assert call(h) == 0 and noalloc() == 0


def test_coherence_backward_spreads_a_batch_of_small_tensors(fake):
    """The end of the coherence backward: a batch of small tensors has blocks for the whole chip, a large tensor
    its own."""
    h = fake.handle()
    buf = [fake.field(1) for _ in range(3)]
    mod = fake.lib.TopMod(flags=fake.lib.TOP_MOD_PHASE, phase=fake.field(1))
    grads = fake.lib.TopModGrads(saved_in=buf[2], grad_phase=fake.field(1))
    lam, z = fake.one(5e-7), fake.one(0.02)
    for batch, n in ((256, 16), (3, 16), (64, 32), (1, 64)):
        for with_grads in (True, False):
            fake.dll.fake_reset()
            st = fake.dll.top_propagate_coherence_backward(h, fake.grid(batch, n, n), buf[0], buf[1], lam, z, C.byref(mod),
                                                           C.byref(grads) if with_grads else None, None)
            assert st == 0, fake.error()
            at = [i for i, k in enumerate(fake.launches()) if "k_coh_backward_end" in k]
            assert len(at) == 1
            xyz = (C.c_uint * 3)()
            fake.dll.fake_grid(at[0], xyz)
            blocks = xyz[0] * xyz[1]
            assert blocks == (n * n // 64) * (n * n // 128)
            assert xyz[2] <= batch and (xyz[2] == batch or blocks * xyz[2] >= 304), (batch, n, list(xyz))


def test_fields_that_share_their_parameters_cost_the_host_once(fake):
    """8192 fields of one wavelength and distance go out in four launches a pass: with their parameter sets looked
    up field by field the call took the host some 250 times as long as a single field's."""
    import time
    h, x = fake.handle(), fake.field(1)
    lam, z = fake.one(5e-7), fake.one(0.02)

    def host_time(batch):
        best = 1e9
        for _ in range(20):
            fake.dll.fake_reset()
            t = time.perf_counter()
            assert fake.dll.top_propagate(h, fake.grid(batch, 16, 16), x, x, lam, z, 1, None, None, None) == 0
            best = min(best, time.perf_counter() - t)
        return best

    host_time(8192)
    assert host_time(8192) < 50 * host_time(1)


def test_bluestein_calls_write_no_list_of_one_table(fake):
    """A call at a size without a plan launches its passes alone when its fields share their transfer table, or
    are few; a longer list of tables is written first."""
    h, x = fake.handle(), fake.field(1)
    for batch, sets, writes in ((1, 1, 0), (700, 1, 0), (16, 16, 0), (17, 17, 1)):
        zs = fake.lib.doubles([0.02 + 0.001 * i for i in range(sets)])
        lams = fake.lib.doubles([5e-7] * sets)
        g = fake.grid(batch, 61, 61, 1.0)
        assert fake.dll.top_propagate(h, g, x, x, lams, zs, sets, None, None, None) == 0, fake.error()  # builds the tables
        fake.dll.fake_reset()
        assert fake.dll.top_propagate(h, g, x, x, lams, zs, sets, None, None, None) == 0
        names = fake.launches()
        assert len([k for k in names if "k_put" in k]) == writes, (batch, sets, names)
        assert len(names) == 5 + writes


def test_transposes_of_small_planes_fill_their_tiles(fake):
    """Planes of at most 32 samples a side are transposed in tiles of 32, larger ones in tiles of 64."""
    h, x = fake.handle(), fake.field(1)
    lam, z = fake.one(5e-7), fake.one(0.02)
    for n, tile in ((17, 32), (31, 32), (33, 64), (61, 64)):
        fake.dll.fake_reset()
        assert fake.dll.top_propagate(h, fake.grid(64, n, n, 1.0), x, x, lam, z, 1, None, None, None) == 0, fake.error()
        names = [k for k in fake.launches() if "k_transpose" in k]
        assert len(names) == 2 and all("k_transpose<%d>" % tile in k for k in names), (n, names)
