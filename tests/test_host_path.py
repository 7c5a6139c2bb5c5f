"""The library's host code against a CUDA runtime without a device (fake_cudart.c): what
its launches ask for, on the CPU.

Kernels do not run and results are zeros; launches are refused as a device would refuse
them (more shared memory than the kernel was allowed on the current device), and so are
allocations beyond the device's memory.
"""
import ctypes
import glob
import os
import re
import shutil
import subprocess

import numpy as np
import pytest

HERE = os.path.dirname(os.path.abspath(__file__))
ROOT = os.path.dirname(HERE)
C128, C64, C64H = 0, 1, 3
P = ctypes.c_void_p


@pytest.fixture(scope="module")
def lib(tmp_path_factory):
    cuda = os.environ.get("CUDA_HOME", "/usr/local/cuda")
    if not shutil.which("g++") or not os.path.exists(os.path.join(cuda, "include", "cuda_runtime_api.h")):
        pytest.skip("needs g++ and the CUDA headers")
    import __graft_entry__
    built = __graft_entry__._build_module().build()
    out = str(tmp_path_factory.mktemp("fake"))
    obj, so = os.path.join(out, "fake.o"), os.path.join(out, "libspm_fake.so")
    subprocess.run(["gcc", "-O1", "-fPIC", "-I", os.path.join(cuda, "include"), "-c", os.path.join(HERE, "fake_cudart.c"), "-o", obj],
                   check=True)
    objs = sorted(glob.glob(os.path.join(os.path.dirname(built), "*.o")))
    subprocess.run(["g++", "-shared", "-Wl,-Bsymbolic", "-Wl,--no-undefined", "-o", so] + objs + [obj, "-lpthread"], check=True)
    lib = ctypes.CDLL(so)
    lib.fake_log.restype = ctypes.c_char_p
    lib.fake_used.restype = lib.fake_peak.restype = ctypes.c_size_t
    lib.fake_capacity.argtypes = [ctypes.c_size_t]
    lib.spm_create_problem.argtypes = [ctypes.c_int, ctypes.c_double, P, P, ctypes.c_int, P, P]
    lib.spm2_create_problem.argtypes = lib.spm_create_problem.argtypes
    for name in ("set_stencils", "factor_S", "apply_A", "apply_Q", "solve_S", "destroy"):
        for p in ("spm_", "spm2_"):
            f = getattr(lib, p + name)
            f.argtypes = {"set_stencils": [P, P, P], "factor_S": [P, ctypes.c_int], "destroy": [P]}.get(
                name, [P, ctypes.c_int, P, P, ctypes.c_int, P])
    return lib


@pytest.fixture(autouse=True)
def one_device(lib):
    lib.fake_device(0)
    lib.fake_clear()
    yield
    lib.fake_device(0)
    lib.fake_capacity(280 << 30)


class Prob:
    """A problem with zero stencils (their values reach no host decision)."""

    def __init__(self, lib, dim, n):
        self.lib, self.p, self.h = lib, "spm_" if dim == 3 else "spm2_", P()
        nt = 3 ** dim
        eps, grad = np.ones(n ** dim, np.complex128), np.zeros(dim * n ** dim, np.complex128)
        al, be = np.zeros(nt * dim * nt * dim, np.complex128), np.zeros(nt * (dim + 1) * nt * dim, np.complex128)
        assert self.call("create_problem", n, 5.0, eps.ctypes.data, grad.ctypes.data, 0, None, ctypes.addressof(self.h)) == 0
        assert self.call("set_stencils", self.h, al.ctypes.data, be.ctypes.data) == 0

    def call(self, name, *args):
        return getattr(self.lib, self.p + name)(*args)

    def solve(self, prec, nrhs):
        return self.call("solve_S", self.h, prec, P(256), P(1 << 40), nrhs, None)

    def close(self):
        self.call("destroy", self.h)


def launches(lib):
    """(device, shared bytes, number, threads, kernel) of every launch since the last clear."""
    out = [line.split(" ", 4) for line in lib.fake_log().decode().splitlines()]
    lib.fake_clear()
    return [(int(d), int(s), int(a), int(t), k) for d, s, a, t, k in out]


@pytest.mark.parametrize("dim,n", [(2, 23), (2, 243), (2, 246), (3, 16)])
def test_staged_tiles_leave_the_vectors_aligned(lib, dim, n):
    """A staged block's shared memory holds the tile and then the vectors: the tile's bytes
    are a multiple of the vector's element, whatever the largest tile (at n = 243 1335
    entries of 4 bytes in half storage)."""
    pb = Prob(lib, dim, n)
    for prec in (C128, C64, C64H):
        assert pb.call("factor_S", pb.h, prec) == 0
        launches(lib)
        staged = 0
        for nrhs in (1, 2, 3, 4, 5, 16):
            assert pb.solve(C64 if prec == C64H else prec, nrhs) == 0
            for _, smem, tile, _, kernel in launches(lib):
                m = re.search(r"k_nd_levelI(6float2|7double2)(S\d?_|7__half2)Li(\d+)ELb\dELb(\d)E", kernel)
                if not m or m.group(4) == "0":
                    continue
                vec = 8 if m.group(1) == "6float2" else 16
                at = tile * (4 if "half" in m.group(2) else vec)
                assert at % vec == 0
                assert smem >= at + vec * int(m.group(3)) * 256
                staged += 1
        assert staged
    pb.close()


def test_a_second_device_is_opted_in(lib):
    """What a kernel is allowed holds for one device: Q's padding for even placement and the
    solve's tiles with their sums are asked for on every device that launches them."""
    for dev in (0, 1):
        lib.fake_device(dev)
        for dim, n in ((2, 64), (3, 16)):
            pb = Prob(lib, dim, n)
            assert pb.call("apply_Q", pb.h, C128, P(256), P(1 << 40), 1, None) == 0
            for prec in (C128, C64):
                assert pb.call("factor_S", pb.h, prec) == 0
                for nrhs in (1, 2, 4, 8, 16):
                    assert pb.solve(prec, nrhs) == 0
            pb.close()
        seen = launches(lib)
        assert all(d == dev and k != "-" for d, _, _, _, k in seen)
        assert max(s for _, s, _, _, k in seen if "k_nd_level" in k) > 48 * 1024
        assert max(s for _, s, _, _, k in seen if "k2_applyQ" in k) > 48 * 1024


def test_factor_takes_less_where_memory_ends(lib):
    """3-D n = 32 in complex128: fronts of up to 1536 unknowns advance together, which takes
    a quarter more memory than a line at 512; where that is not there, the lower lines are
    tried before the factor is refused."""
    pb = Prob(lib, 3, 32)
    lib.fake_peak()
    assert pb.call("factor_S", pb.h, C128) == 0
    need = lib.fake_peak()
    pb.close()
    pb = Prob(lib, 3, 32)
    for share, status in ((0.9, 0), (0.5, 3), (1.0, 0)):
        lib.fake_capacity(int(share * need))
        assert pb.call("factor_S", pb.h, C128) == status
    pb.close()


@pytest.mark.parametrize("n,nrhs", [(4, 1), (4, 4000), (5, 7), (119, 64), (479, 8)])
def test_2d_q_threads(lib, n, nrhs):
    """2-D Q reads a point's neighbours once in complex64 (a thread per point; a thread per
    component took 1.5 times as long at eight fields of n = 479), twice in complex128, and
    leaves no block partly empty but the last."""
    pb = Prob(lib, 2, n)
    for prec, each, block in ((C64, 1, 256), (C128, 2, 64)):
        launches(lib)
        assert pb.call("apply_Q", pb.h, prec, P(256), P(1 << 40), nrhs, None) == 0
        (_, _, _, threads, kernel), = launches(lib)
        assert "k2_applyQ" in kernel
        assert threads == each * -(-n * n * nrhs // block) * block
    pb.close()


@pytest.mark.parametrize("n,prec,kernel", [(8, C64, "k2_zfield"), (16, C64, "k2_zprod4"), (32, C64, "k2_zprod4"),
                                           (8, C128, "k2_zfield"), (16, C128, "k2_zfield"), (32, C128, "k2_zprod4")])
def test_z_pass_of_plan_0(lib, n, prec, kernel):
    """A warp per field where the four-line kernel leaves the schedulers idle: not at L = 32
    in complex64 (64 fields 49.8 us against 39.7).  By L alone, whatever the block."""
    pb = Prob(lib, 3, n)
    assert lib.spm_set_apply_plan(prec, 2 * n, 0) == 0
    for nrhs in (1, 64):
        launches(lib)
        assert pb.call("apply_A", pb.h, prec, P(256), P(1 << 40), nrhs, None) == 0
        z = {m for *_, k in launches(lib) for m in ("k2_zfield", "k2_zprod4", "k2_zprod1") if m in k}
        assert z == {kernel}
    pb.close()


@pytest.mark.parametrize("n,nrhs,half", [(4, 1, True), (16, 8, True), (16, 64, False), (64, 1, True), (64, 8, False), (96, 1, False)])
def test_3d_q_asks_for_half_of_the_l1_on_few_blocks(lib, n, nrhs, half):
    """Complex64 Q: many blocks need more of the L1 as shared memory than half (16 fields at
    n = 64 225 us against 212)."""
    pb = Prob(lib, 3, n)
    launches(lib)
    assert pb.call("apply_Q", pb.h, C64, P(256), P(1 << 40), nrhs, None) == 0
    (_, _, shared, _, kernel), = launches(lib)
    assert "k_q" in kernel and shared == (50 if half else 0)
    pb.close()
