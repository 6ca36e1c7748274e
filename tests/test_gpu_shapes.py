"""Stage kernels at pinned launch shapes, bit for bit: which kernel a 2-D grid takes
(the row kernel or the plane kernel) and which segments, rows and planes a tile has is
chosen by timing, so every choice has to give the same bits. Shapes are pinned through
a probe that calls the library's launchers; the public interface leaves the segment
and the kernel to the tuner."""
import ctypes
import os
import subprocess

import numpy as np
import pytest

from paper_2507_11542_gb300 import workloads as W
from helpers import ADVECT, AIR3D, DI, DUBINS, NORM, PARAMS, ROTATE, lib_method, to_dev

pytestmark = pytest.mark.gpu

HERE = os.path.dirname(os.path.abspath(__file__))
ROOT = os.path.dirname(HERE)
PKG = os.path.join(ROOT, "paper_2507_11542_gb300")


@pytest.fixture(scope="module")
def probe(tmp_path_factory):
    from paper_2507_11542_gb300 import _lib as L
    L.load()
    out = str(tmp_path_factory.mktemp("shape") / "libshape_probe.so")
    subprocess.check_call(["nvcc", "-O2", "-std=c++17", "-shared", "-Xcompiler", "-fPIC", "-I" + os.path.join(PKG, "csrc"),
                           "-I" + os.path.join(ROOT, "include"), "-o", out,
                           os.path.join(HERE, "probes", "shape_probe.cpp"), os.path.join(PKG, "libhj.so"),
                           "-Xlinker", "-rpath=" + PKG])
    lib = ctypes.CDLL(out)
    p, i = ctypes.c_void_p, ctypes.c_int
    lib.shape_stage.argtypes = [p, p, i, i, i, i, i, i, p, p, p, p, p, ctypes.c_double, p]
    return lib


def _run(lib, spec, m, dtype, shape, V, old, stage):
    """Output of one stage (0: the term) at (plane, sx, ty, tz), or None where there is no such shape."""
    import torch
    from paper_2507_11542_gb300 import _lib as L
    G = L.make_grid(spec)
    trig = [0, 0]
    keep = []
    if spec.ndim >= 3:
        x = spec.lo[2] + np.arange(spec.n[2]) * ((spec.hi[2] - spec.lo[2]) / (spec.n[2] if 2 in spec.periodic else spec.n[2] - 1))
        table = torch.from_numpy(np.concatenate([np.cos(x), np.sin(x)])).cuda()
        keep = [table, table.float()]
        trig = [keep[0].data_ptr(), keep[1].data_ptr()]
    out = torch.full_like(V, 7.0)
    plane, sx, ty, tz = shape
    rc = lib.shape_stage(ctypes.byref(G), ctypes.byref(m), L.dtype_code(V.dtype), plane, sx, ty, tz, stage, V.data_ptr(),
                         old.data_ptr(), out.data_ptr(), trig[0], trig[1], 0.01,
                         torch.cuda.current_stream().cuda_stream)
    assert rc in (0, -1), rc
    torch.cuda.synchronize()
    del keep
    return None if rc else out


def _field(spec, seed, dtype):
    return to_dev(W.random_field(spec, seed) + 0.3 * np.sqrt(sum((x - 0.1) ** 2 for x in spec.mesh())), dtype)


# the tuner's shapes, the static step's, and odd ones; on these grids they leave last
# segments and rows of one to three nodes
PLANES = [(5, 8), (5, 12), (7, 4), (7, 6), (8, 5), (8, 8), (12, 6), (16, 8), (16, 9), (12, 12), (16, 10), (32, 8), (4, 3), (9, 1)]


@pytest.mark.parametrize("dyn,alpha_box", [(DI, False), (NORM, False), (NORM, True), (ADVECT, False), (ROTATE, False)])
@pytest.mark.parametrize("n,periodic,extrap", [((37, 29), (), 0), ((33, 49), (0,), 1), ((61, 25), (1,), 0), ((8, 9), (0, 1), 0),
                                               ((4, 13), (), 1)])
@pytest.mark.parametrize("scheme", [1, 2, 3, 5])
@pytest.mark.parametrize("dtype", ["float64", "float32"])
def test_plane_kernel_gives_the_row_kernels_bits(probe, dyn, alpha_box, n, periodic, extrap, scheme, dtype):
    import torch
    spec = W.GridSpec(n, (-1.0, -1.5), (2.0, 1.0), periodic)
    V, old = _field(spec, 5, dtype), _field(spec, 6, dtype)
    for stage, brt in ((0, 0), (1, 1), (2, 1), (3, 2)):
        m = lib_method(scheme=scheme, dynamics=dyn, brt=brt, extrap=extrap, alpha_box=alpha_box)
        want = _run(probe, spec, m, dtype, (0, min(n[0], 20), min(4, n[1]), 1), V, old, stage)
        assert want is not None
        for sx, ty in PLANES:
            got = _run(probe, spec, m, dtype, (1, min(sx, n[0]), min(ty, n[1]), 1), V, old, stage)
            assert torch.equal(got, want), (stage, sx, ty)


# segments that leave a last one of one to three nodes, odd and even; odd and even rows
SEGMENTS = {61: (30, 20, 15, 12, 59, 29, 61), 25: (12, 24, 8, 23, 25), 16: (15, 5, 7, 16, 3)}


@pytest.mark.parametrize("dyn,n,periodic", [(DI, (61, 22), ()), (DI, (25, 9), (0, 1)), (AIR3D, (61, 10, 7), (2,)),
                                            (NORM, (25, 13, 6), (0,)), (DUBINS, (16, 9, 5, 6), (2,)), (DUBINS, (25, 5, 4, 4), (0, 2, 3))])
@pytest.mark.parametrize("scheme", [1, 2, 3, 5])
@pytest.mark.parametrize("dtype", ["float64", "float32"])
def test_row_kernel_gives_the_same_bits_at_any_segment(probe, dyn, n, periodic, scheme, dtype):
    import torch
    spec = W.GridSpec(n, (-1.0, -1.5, 0.0, 0.0)[:len(n)], (2.0, 1.0, 6.0, 2.0)[:len(n)], periodic)
    V, old = _field(spec, 7, dtype), _field(spec, 8, dtype)
    m = lib_method(scheme=scheme, dynamics=dyn, brt=1)
    for stage in (1, 3):
        want, tried = None, 0
        for sx in SEGMENTS[n[0]]:
            for ty in (1, 2, 3, 5, 7, 8):
                for tz in ((1, 3, n[-1]) if len(n) > 2 else (1,)):
                    got = _run(probe, spec, m, dtype, (0, sx, min(ty, n[1]), tz), V, old, stage)
                    if got is None:
                        continue
                    tried += 1
                    want = got if want is None else want
                    assert torch.equal(got, want), (stage, sx, ty, tz)
        assert tried >= 20
