"""Which kernel and geometry the library picks for a launch: dispatch_probe.cu
compiled against its headers and linked to the built library (no GPU needed)."""
import ctypes
import functools
import os
import subprocess
import tempfile

from paper_2309_08864_gb300 import build, so2dr

GENERIC, STAR3D, ROW2D, BOX2D, PLANE3D, TILE2D = range(6)  # LaunchShape::fast
SHAPES = {("star", 3): 0, ("star", 2): 1, ("box", 2): 2, ("varcoef", 3): 3}
FIELDS = ("ok", "fast", "small", "ragged", "gx", "gy", "gz", "tx", "ty", "smem", "split", "split2", "split_at")


@functools.lru_cache(maxsize=None)
def _lib():
    lib = build.build()
    out = os.path.join(tempfile.mkdtemp(prefix="so2dr_probe"), "probe.so")
    src = os.path.join(os.path.dirname(os.path.abspath(__file__)), "dispatch_probe.cu")
    subprocess.run([build._nvcc(), "-std=c++17", "-shared", "-Xcompiler", "-fPIC", "-I" + build.INCLUDE,
                    "-I" + build.CSRC] + build.ARCH + ["-o", out, src, lib, "-Xlinker", "-rpath," + os.path.dirname(lib)],
                   check=True)
    return ctypes.CDLL(out)


def launch(dtype, kind, r, depth, dims, nout=None, sms=152, occ=4):
    """The choice for one launch that writes `nout` planes (default: all) of a grid of `dims`."""
    n0, ny, nx = dims if len(dims) == 3 else (dims[0], 1, dims[1])
    out = (ctypes.c_int64 * len(FIELDS))()
    i64 = ctypes.c_int64
    _lib().probe_launch(so2dr.DTYPES[dtype], SHAPES[kind, len(dims)], r, depth, i64(n0), i64(ny), i64(nx),
                        i64(nout or n0), sms, occ, out)
    return dict(zip(FIELDS, out))


def star_split_small(dtype, r, depth, dims, sms=152, occ=3):
    i64 = ctypes.c_int64
    return _lib().probe_star_split_small(so2dr.DTYPES[dtype], r, depth, *(i64(n) for n in dims), sms, occ)


def star_occupancy(dtype, r, depth, dims):
    """CTAs per SM of the 3D star kernel (needs a GPU)."""
    i64 = ctypes.c_int64
    return _lib().probe_star_occupancy(so2dr.DTYPES[dtype], r, depth, *(i64(n) for n in dims))
