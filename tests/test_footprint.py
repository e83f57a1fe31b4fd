"""pic_run_footprint counts the grid arrays that a box holds, checked on boxes
without particles (ppc = 0), whose particle share is the fixed loose lists."""
import pytest

from paper_2602_15939_gb300 import pic as P

XY, XZ = P.PIC_PLANE_XY, P.PIC_PLANE_XZ


def grid_bytes(box, n, ndim, plane, fp64):
    es = 8 if fp64 else 4
    q = 16 // es
    active = (True, not (ndim == 2 and plane == XZ), not (ndim == 2 and plane == XY))
    px = -(-(n[0] + 5) // q) * q
    padded = px * (n[1] + 5 if active[1] else 1) * (n[2] + 5 if active[2] else 1)
    sheared = box in (P.PIC_BOX_SHEAR, P.PIC_BOX_SHEAR_EXPAND)
    advects = sheared and active[1]
    arrays = 3                                  # E, B, J
    arrays += 1 if fp64 or advects else 0       # the folded current beside the accumulators
    arrays += 4 if sheared else 0               # two pairs of iterates
    total = arrays * 3 * padded * es
    total += 0 if fp64 else 3 * padded * 4      # fixed-point accumulators
    total += 3 * n[0] * n[1] * n[2] * 8         # staging of a field
    total += 2 * n[0] * 16 if advects else 0    # advection table
    return total


CASES = [(P.PIC_BOX_PERIODIC, (64, 48, 40), 3, 0), (P.PIC_BOX_SHEAR, (64, 48, 40), 3, 0),
         (P.PIC_BOX_SHEAR, (65536, 64, 1), 2, XY), (P.PIC_BOX_SHEAR_EXPAND, (65536, 64, 1), 2, XY),
         (P.PIC_BOX_SHEAR, (4096, 1, 64), 2, XZ), (P.PIC_BOX_LEAKY, (512, 512, 1), 2, XY)]


@pytest.mark.parametrize("box,n,ndim,plane", CASES)
@pytest.mark.parametrize("fp64", [False, True])
def test_footprint_counts_the_grid_arrays(box, n, ndim, plane, fp64):
    prec = P.PIC_FP64 if fp64 else P.PIC_FP32
    cfg = P.make_config(box=box, nx=n[0], ny=n[1], nz=n[2], ndim=ndim, plane=plane, precision=prec, c=0.2)
    # what a run holds besides: tile slots and loose lists, from the same box at two species counts
    one = P.pic_run_footprint(P.make_run_spec(cfg, 1, 0, 0.1, q=(0.1,), m=(1.0,)))
    two = P.pic_run_footprint(P.make_run_spec(cfg, 1, 0, 0.1, q=(0.1, -0.1)))
    assert one - (two - one) == grid_bytes(box, n, ndim, plane, fp64) + (1 << 20)


@pytest.mark.gpu
def test_footprint_is_what_boxes_take_from_the_device():
    """Device memory before and after creating boxes whose single grid arrays
    are larger than the allocator's granularity, in a process of its own (the
    library keeps freed memory for reuse)."""
    import os
    import subprocess
    import sys

    code = """
import ctypes
from paper_2602_15939_gb300 import pic as P
cu = ctypes.CDLL("libcuda.so.1")
def free():
    f, t = ctypes.c_size_t(), ctypes.c_size_t()
    assert cu.cuMemGetInfo_v2(ctypes.byref(f), ctypes.byref(t)) == 0
    return f.value
boxes = []  # all stay alive
P.pic_preload_kernels(0, P.PIC_FP32)
P.pic_preload_kernels(0, P.PIC_FP64)
def make(cfg):
    spec = P.make_run_spec(cfg, 1, 1, 0.1, q=(0.1,), m=(1.0,))
    before = free()
    b = P.Box(cfg)
    b.load_maxwellian(0, 0.1, 1.0, 1, 0.1)
    b.step(2)
    b.sync()
    boxes.append(b)
    return before - free(), P.pic_run_footprint(spec)
make(P.make_config(nx=16, ny=16, nz=16))
make(P.make_config(nx=16, ny=16, nz=16, precision=P.PIC_FP64))
for box, prec in ((P.PIC_BOX_PERIODIC, P.PIC_FP32), (P.PIC_BOX_SHEAR, P.PIC_FP32), (P.PIC_BOX_EXPAND, P.PIC_FP64)):
    print(*make(P.make_config(box=box, nx=192, ny=192, nz=192, c=0.2, precision=prec)))
"""
    root = os.path.dirname(os.path.dirname(os.path.abspath(__file__)))
    out = subprocess.run([sys.executable, "-c", code], cwd=root, capture_output=True, text=True, timeout=300)
    assert out.returncode == 0, out.stderr[-2000:]
    rows = [tuple(map(int, line.split())) for line in out.stdout.splitlines()]
    assert len(rows) == 3
    one_array = 3 * 200 * 197 * 197 * 4
    for used, footprint in rows:
        assert abs(used - footprint) < 0.7 * one_array, rows
