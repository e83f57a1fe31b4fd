"""FP32 results do not depend on the launch variant or on the tiles, bit for
bit, in every box kind, geometry and shape order that has a kernel.  The
kernels of the variants are separate compilations of one source, and a
compiler may fuse different products of a sum in each; this holds the promise
for all of them where fixing every rounding in the source would not be read."""
import dataclasses

import numpy as np
import pytest

from gpu_harness import Case, run_gpu
from paper_2602_15939_gb300 import pic as P

XY, XZ = P.PIC_PLANE_XY, P.PIC_PLANE_XZ
SHEAR = dict(s=1.5, Omega0=3e-3, step0=37)
EXPAND = dict(rate=(0.0, 1e-3, 1e-3), step0=200)
PROB = dict(esc_mode=P.PIC_ESC_PROBABILISTIC, p_esc=0.05, theta_inj=1.0)
DISP = dict(esc_mode=P.PIC_ESC_DISPLACEMENT, l_esc=2.0, theta_inj=1.0)
KINDS = {"periodic": (P.PIC_BOX_PERIODIC, {}), "shear": (P.PIC_BOX_SHEAR, SHEAR), "expand": (P.PIC_BOX_EXPAND, EXPAND),
         "shear_expand": (P.PIC_BOX_SHEAR_EXPAND, {**SHEAR, "rate": EXPAND["rate"]}), "leaky_prob": (P.PIC_BOX_LEAKY, PROB),
         "leaky_disp": (P.PIC_BOX_LEAKY, DISP), "shear_prob": (P.PIC_BOX_SHEAR, {**SHEAR, **PROB}),
         "expand_prob": (P.PIC_BOX_EXPAND, {**EXPAND, **PROB})}
GEOMS = {"3d": ((20, 16, 12), 3, 0, (4, 8)), "xy": ((40, 36, 1), 2, XY, (8, 16, 32)), "xz": ((40, 1, 36), 2, XZ, (8, 16, 32))}


def bits(case):
    parts, fields, diag = run_gpu(case, 2, False)
    assert diag.error_word == 0
    out = list(fields)
    for x, u, ids, _ in parts:
        o = np.argsort(ids)
        out += [ids[o], x[o], u[o]]
    return out


@pytest.mark.gpu
@pytest.mark.parametrize("order", [1, 2])
@pytest.mark.parametrize("geom", GEOMS)
@pytest.mark.parametrize("kind", KINDS)
def test_fp32_bits_are_the_same_in_every_launch_shape(kind, geom, order):
    n, ndim, plane, sides = GEOMS[geom]
    box, kw = KINDS[kind]
    case = Case(kind, box, n, ndim=ndim, plane=plane, order=order, ppc=10, uth=0.4, **kw)
    ref = None
    for side in sides:
        for k in range(P.pic_kernel_variant_count() + 1):  # 0: the library's own shape
            tile = tuple(side if n[a] > 1 else 0 for a in range(3))
            got = bits(dataclasses.replace(case, tile=tile, variant=k))
            if ref is None:
                ref = got
            for a, b in zip(ref, got):
                assert np.array_equal(a, b), (side, k)
