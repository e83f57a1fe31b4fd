"""A box forced to a launch variant runs the shape that pic_kernel_variant_info
states, on every tile and in both precisions; a variant is refused only where
its shared memory does not fit.  The library's own choice on 4^3 tiles and in
FP64, variant 7 with half of its threads, against the oracle with full queues
(the tolerances of the parity tests), and kept by the autotuner where it is
the fastest form."""
import pytest

from gpu_harness import Case, compare
from paper_2602_15939_gb300 import pic as P

XY, XZ = P.PIC_PLANE_XY, P.PIC_PLANE_XZ
GEOMS = {"3d": ((16, 12, 8), 3, 0, (4, 8)), "xy": ((40, 32, 1), 2, XY, (8, 16, 32)), "xz": ((40, 1, 32), 2, XZ, (8, 16, 32))}


def config(geom, side, fp64, variant=0, order=2):
    n, ndim, plane, _ = GEOMS[geom]
    tile = tuple(side if n[a] > 1 else 0 for a in range(3))
    return P.make_config(nx=n[0], ny=n[1], nz=n[2], ndim=ndim, plane=plane, order=order, tile=tile,
                         precision=P.PIC_FP64 if fp64 else P.PIC_FP32, kernel_variant=variant)


SHAPES = [(g, s, f) for g in GEOMS for s in GEOMS[g][3] for f in (False, True) if not (f and s == 32)]


@pytest.mark.gpu
@pytest.mark.parametrize("geom,side,fp64", SHAPES, ids=[f"{g}_t{s}_{'fp64' if f else 'fp32'}" for g, s, f in SHAPES])
def test_a_forced_variant_runs_the_shape_it_reports(geom, side, fp64):
    for k in range(1, P.pic_kernel_variant_count() + 1):
        if fp64 and geom == "3d" and side == 8 and k == 7:  # 360 KB of shared memory
            with pytest.raises(P.PicError) as e:
                P.Box(config(geom, side, fp64, k))
            assert e.value.status == P.PIC_ERR_ARG and "does not fit" in str(e.value)
            continue
        box = P.Box(config(geom, side, fp64, k))
        assert P.pic_get_kernel_variant(box.h) == k
        assert P.pic_get_launch_shape(box.h) == P.pic_kernel_variant_info(k)
        box.close()
    box = P.Box(config(geom, side, fp64))
    half = side == 4 if not fp64 else not (geom == "3d" and side == 8)
    if half:
        assert P.pic_get_kernel_variant(box.h) == 7 and P.pic_get_launch_shape(box.h) == (256, 0, 4)
        P.pic_set_kernel_variant(box.h, 7)
        assert P.pic_get_launch_shape(box.h) == (512, 0, 4)
    else:
        assert P.pic_get_launch_shape(box.h) == P.pic_kernel_variant_info(P.pic_get_kernel_variant(box.h))
    box.close()


@pytest.mark.gpu
@pytest.mark.parametrize("fp64", [False, True], ids=["fp32", "fp64"])
@pytest.mark.parametrize("order", [1, 2])
def test_the_half_shape_matches_the_oracle_with_full_queues(order, fp64):
    case = Case("hot", P.PIC_BOX_PERIODIC, (16, 12, 8), order=order, ppc=40, uth=0.4, tile=(4, 4, 4))
    r = compare(case, 1, fp64)
    tol = 1e-12 if fp64 else 1e-6
    assert r["error_word"] == 0 and r["x"] <= (1e-12 if fp64 else 2e-6)
    for f in ("u", "E", "B", "J"):
        assert r[f] <= tol, (f, r)


@pytest.mark.gpu
def test_the_autotuner_and_new_tiles_keep_a_shape_that_exists():
    box = P.Box(config("3d", 4, False))
    try:
        box.load_maxwellian(0, 0.05, 1.0, 8, 0.05, seed=3)
        best, ms, _ = box.autotune(2)
        nt, st, jc = P.pic_get_launch_shape(box.h)
        assert best == P.pic_get_kernel_variant(box.h) and ms[best - 1] == min(ms)
        want = P.pic_kernel_variant_info(best)
        assert (st, jc) == want[1:] and (nt == want[0] or (best == 7 and nt == 256))
        box.set_tile(8)  # no half shape here: the variant's own
        assert P.pic_get_launch_shape(box.h) == P.pic_kernel_variant_info(P.pic_get_kernel_variant(box.h))
        box.step(1)
        assert box.diagnostics().error_word == 0
    finally:
        box.close()
