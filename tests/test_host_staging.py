"""The host path of graph replays where the device has no memory for the staging copies (masks, coil
maps, image), on the library's own objects linked with a stand-in for the CUDA runtime: no GPU."""

import ctypes
import os
import subprocess

import numpy as np
import pytest

ROOT = os.path.dirname(os.path.dirname(os.path.abspath(__file__)))
MALLOC, REFUSED, CAPTURE, LAUNCH, DEVICE_SYNC = range(5)
FILT = (3, 3, 2)


@pytest.fixture(scope="module")
def lib(tmp_path_factory):
    from paper_1704_04511_gb300 import build, recon
    build.build()
    out = str(tmp_path_factory.mktemp("fake") / "librecon_fake.so")
    objs = [os.path.join(build.BUILD, s.replace(".cu", ".o")) for s in build.SOURCES]
    subprocess.run(["g++", "-std=c++17", "-O1", "-shared", "-fPIC", "-Wl,-Bsymbolic", "-Wl,-z,defs", "-o", out,
                    os.path.join(ROOT, "tests", "fake_cuda_runtime.cpp")] + objs, check=True)
    lib = ctypes.CDLL(out)
    lib.recon_create.argtypes = [ctypes.POINTER(ctypes.c_void_p), ctypes.c_int, ctypes.c_size_t, ctypes.c_void_p]
    lib.recon_destroy.argtypes = [ctypes.c_void_p]
    lib.recon_set_option.argtypes = [ctypes.c_void_p, ctypes.c_int, ctypes.c_int]
    lib.recon_solve_batch.argtypes = [ctypes.c_void_p, ctypes.c_int, recon.recon_dims, ctypes.c_void_p,
                                      ctypes.c_void_p, recon.recon_filter, ctypes.POINTER(recon.recon_params),
                                      ctypes.c_void_p]
    lib.recon_last_error.argtypes, lib.recon_last_error.restype = [ctypes.c_void_p], ctypes.c_char_p
    lib.fake_limit.argtypes, lib.fake_used.restype = [ctypes.c_size_t], ctypes.c_size_t
    lib.fake_count.restype = ctypes.c_long
    return lib


class Program:
    """A context and n scans in buffers that stay."""

    def __init__(self, lib, n, graphs=1):
        from paper_1704_04511_gb300 import recon
        self.lib, self.n, self.ctx = lib, n, ctypes.c_void_p()
        assert lib.recon_create(ctypes.byref(self.ctx), 0, 0, None) == 0
        lib.recon_set_option(self.ctx, recon.RECON_OPT_GRAPHS, graphs)
        lib.recon_set_option(self.ctx, recon.RECON_OPT_AUTOTUNE, 0)

    def scans(self, T, P, Q):
        return [[np.zeros((T, P, Q), np.complex64), np.ones((T, P, Q), np.uint8), np.zeros((T, P, Q), np.complex64)]
                for _ in range(self.n)], (T, P, Q)

    def solve(self, scans):
        """One batch; what it did: allocations asked for and refused, captures, replays, device-wide waits."""
        from paper_1704_04511_gb300 import recon
        bufs, (T, P, Q) = scans
        ptrs = [(ctypes.c_void_p * self.n)(*[b[k].ctypes.data for b in bufs]) for k in range(3)]
        prm = recon.recon_params(irls=2, cg=2, lambda_=1e-3, p=0.0, gamma=1.4, eps0_frac=0.01, kspace_bf16=0,
                                 weight_method=0)
        before = [self.lib.fake_count(k) for k in range(5)]
        rc = self.lib.recon_solve_batch(self.ctx, self.n, recon.recon_dims(P=P, Q=Q, T=T), ptrs[0], ptrs[1],
                                        recon.recon_filter(N1=FILT[0], N2=FILT[1], M=FILT[2]), ctypes.byref(prm),
                                        ptrs[2])
        assert rc == 0, self.lib.recon_last_error(self.ctx)
        return [self.lib.fake_count(k) - b for k, b in enumerate(before)]

    def close(self):
        self.lib.recon_destroy(self.ctx)


def workspace(lib, n, shape):
    """Device bytes of n solves without staging copies (no graphs)."""
    lib.fake_limit(1 << 40)
    used = lib.fake_used()
    pr = Program(lib, n, graphs=0)
    pr.solve(pr.scans(*shape))
    used = lib.fake_used() - used
    pr.close()
    return used


@pytest.mark.parametrize("n,copies", [(1, 0), (1, 0.5), (1, 0.95), (2, 0), (2, 1), (2, 1.95), (3, 2)])
def test_no_memory_for_staging(lib, n, copies):
    """Room for the copies of `copies` of n slots. The first call lays out the slots one after the other
    (a later slot's workspace may take an earlier one's copies back), the second one settles that; from
    then on every slot replays its own graph, nothing is asked of the allocator and nothing waits for the
    whole device."""
    shape = (8, 64, 64)
    need = workspace(lib, n, shape)
    staging = 9 * int(np.prod(shape))
    lib.fake_limit(lib.fake_used() + need + int(copies * staging))
    pr = Program(lib, n)
    scans = pr.scans(*shape)
    first, second = pr.solve(scans), pr.solve(scans)
    assert first[LAUNCH] == n and first[CAPTURE] == n and first[REFUSED] >= n - int(copies)
    assert second[DEVICE_SYNC] == 0
    for _ in range(3):
        assert pr.solve(scans) == [0, 0, 0, n, 0]
    pr.close()
    lib.fake_limit(1 << 40)


def test_staging_makes_room_and_comes_back(lib):
    """A larger series takes the memory of the copies; when it changes the workspace of the slot the
    copies are asked for again, and once more there is room they are used."""
    small, large = (8, 64, 64), (8, 64, 128)
    base = lib.fake_used()
    need = workspace(lib, 1, large)
    lib.fake_limit(base + need + 9 * int(np.prod(small)) // 2)
    pr = Program(lib, 1)
    a, b = pr.scans(*small), pr.scans(*large)
    assert pr.solve(a)[REFUSED] == 0
    assert pr.solve(a) == [0, 0, 0, 1, 0]
    pr.solve(b)
    assert pr.solve(b) == [0, 0, 0, 1, 0]  # no copies: its graph points into the caller's buffers
    lib.fake_limit(1 << 40)
    c = pr.scans(8, 128, 128)
    pr.solve(c)
    assert pr.solve(c) == [0, 0, 0, 1, 0]
    assert pr.solve(pr.scans(8, 128, 128)) == [0, 0, 0, 1, 0]  # staged: other buffers, the same graph
    pr.close()
