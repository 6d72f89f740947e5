"""Host side of the launches against a fake CUDA runtime with two devices
(fake_cudart.cpp), no GPU needed: what is set or asked for per device."""
import ctypes
import os
import subprocess

import pytest

from paper_2409_03030_gb300 import build as nvbuild
from paper_2409_03030_gb300 import jqcd

HERE = os.path.dirname(os.path.abspath(__file__))
DW, KAPPA = jqcd.PREC_DW, 0.12


@pytest.fixture()
def lib(tmp_path):
    """The library's objects linked with the fake runtime, fresh for each test."""
    nvbuild.build()
    objs = [os.path.join(nvbuild.OBJ_DIR, os.path.basename(s)[:-3] + ".o") for s in nvbuild.sources()]
    cuda = os.path.join(os.path.dirname(os.path.dirname(os.path.realpath(nvbuild.nvcc()))), "include")
    so = str(tmp_path / "libjqcd_fake.so")
    r = subprocess.run(["g++", "-shared", "-fPIC", "-std=c++17", "-w", "-Wl,-Bsymbolic", "-I", nvbuild.INCLUDE,
                        "-I", nvbuild.CSRC, "-isystem", cuda, os.path.join(HERE, "fake_cudart.cpp"), *objs,
                        "-o", so, "-ldl", "-lpthread"], capture_output=True, text=True)
    assert r.returncode == 0, r.stderr
    h = ctypes.CDLL(so)
    for name, (res, args) in jqcd._SIGNATURES.items():
        getattr(h, name).restype, getattr(h, name).argtypes = res, args
    h.fake_launches.restype = h.fake_refused.restype = ctypes.c_long
    h.fake_last_grid.restype = ctypes.c_uint
    return h


def field(lib, device, dims):
    ctx, gid = ctypes.c_void_p(), ctypes.c_uint64(0)
    assert lib.jqcd_init(device, ctypes.byref(ctx)) == 0
    links = (ctypes.c_double * 1)()  # not read: the copies do nothing
    lat = jqcd.lattice(dims)
    assert lib.jqcd_gauge_upload(ctx, ctypes.byref(lat), links, 0, ctypes.byref(gid)) == 0
    return ctx, gid


@pytest.mark.parametrize("dims", [(16, 16, 16, 16), (16, 16, 16, 32), (24, 24, 24, 48)])
def test_second_device_takes_the_same_launches(lib, dims):
    """The opt-in to more than 48 KB of shared memory holds on the device where
    it was made: a field on a second device runs every call that one on the
    first does (one-thread hops with limited blocks, with a rest in tiles, and
    plain; the force kernel)."""
    buf = [ctypes.c_void_p(1 << 20 << i) for i in range(6)]
    for device in (0, 1, 0):
        ctx, gid = field(lib, device, dims)
        for dagger in (0, 1):
            assert lib.jqcd_dslash_eo(ctx, gid, DW, 0, dagger, buf[0], None, buf[1], 0.0, 1.0, None, None) == 0
        assert lib.jqcd_mdagm(ctx, gid, DW, KAPPA, buf[0], buf[1], buf[2], None) == 0
        assert lib.jqcd_fermi_force_dev(ctx, gid, KAPPA, *buf[:5], None) == 0
        for which in (0, 1):
            assert lib.fake_launch_cg(which, ctypes.c_int64(dims[0] * dims[1] * dims[2] * dims[3] // 2)) == 0
    assert lib.fake_refused() == 0


def test_launch_forms_follow_each_device(lib):
    """29,160 sites per parity are within twelve 16-site tiles for each of 152
    SMs but not of 148: each device's own count decides, whichever was asked
    first."""
    vh, buf = 29160, [ctypes.c_void_p(1 << 20 << i) for i in range(2)]
    for device in (1, 0, 1):
        ctx, gid = field(lib, device, (6, 6, 6, 270))
        assert lib.jqcd_dslash_eo(ctx, gid, DW, 0, 0, buf[0], None, buf[1], 0.0, 1.0, None, None) == 0
        assert lib.fake_last_grid() == (-(-vh // 16) if device == 0 else -(-vh // 128))


@pytest.mark.parametrize("which", [0, 1, 2, 3])
def test_fused_hops_refuse_fields_past_32_bit_offsets(lib, which):
    """A site's byte offset in a 16-byte plane has 32 bits, bit 0 used: the
    fused hops refuse 2^27 sites per parity, as the plain ones do, and launch
    nothing."""
    field(lib, 0, (4, 4, 4, 4))
    before = lib.fake_launches()
    assert lib.fake_launch_cg(which, ctypes.c_int64(2 ** 27)) == 1  # cudaErrorInvalidValue
    assert lib.fake_launches() == before
    assert lib.fake_launch_cg(which, ctypes.c_int64(2 ** 27 - 8)) == 0
    assert lib.fake_launches() == before + 1


@pytest.mark.parametrize("prec,dims,grid", [
    (0, (6, 6, 6, 270), 1823),               # 29,160 sites: 16-site tiles
    (0, (6, 6, 6, 274), 232),                # 29,592: one thread per site
    (0, (6, 6, 6, 540), 456),                # 58,320: one wave of three blocks per SM
    (0, (6, 6, 6, 542), 456 + 11),           # 58,536: the wave, and 168 sites in tiles
    (0, (20, 18, 14, 26), 456 + 447),        # 65,520
    (3, (10, 10, 10, 130), 4063),            # FP64, 65,000 sites: a tile per block
    (3, (10, 10, 10, 134), 2094),            # 67,000: two
    (3, (32, 32, 32, 34), 8704),             # 557,056: four
])
def test_edge_lattices_take_the_forms_they_stand_for(lib, prec, dims, grid):
    """The lattices that the GPU tests take for the edges of the rules, on 152
    SMs: the grid of the hop shows the form."""
    ctx, gid = field(lib, 0, dims)
    buf = [ctypes.c_void_p(1 << 20 << i) for i in range(3)]
    assert lib.jqcd_dslash_eo(ctx, gid, prec, 0, 1, buf[0], buf[1], buf[2], 0.7, -0.12, None, None) == 0
    assert lib.fake_last_grid() == grid
