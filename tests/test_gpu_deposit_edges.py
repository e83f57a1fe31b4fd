"""Deposits of particles whose offsets lie next to the boundaries of the shape
functions, at rest and in motion: there the rounding of o + 1/2 decides the
deposit class (the largest number below 1/2 plus 1/2 rounds to 1), and the
class and the direction of a crossing must come from the same arithmetic.  One
step of a field-free 3D box, one particle per cell, against the FP64 oracle.

FP32 tolerance, relative to J_ref = |q| c (one particle per cell): up to 64
adds a word, each rounded to half a fixed-point unit (1.2e-7 J_ref), and shape
weights rounded to 2^-24 (below 1e-6 J_ref in all): 1e-5.  FP64: 1e-12."""
import numpy as np
import pytest

import oracle as O
from paper_2602_15939_gb300 import pic as P

N = (16, 12, 8)
C, Q = 0.45, 0.05


def edge_offsets(fp64):
    t = np.float64 if fp64 else np.float32
    below = [float(np.nextafter(t(v), t(0))) for v in (0.5, 1.0)]
    return [below[0], 0.5, float(np.nextafter(t(0.5), t(1))), 0.0, below[1], 0.25]


def plasma(fp64, axis, uaxis):
    """One particle per cell: the offset of `axis` (None: of every axis)
    cycles through the edges, the other offsets are 1/4; uaxis the momenta
    that cycle along with them."""
    edges = edge_offsets(fp64)
    k, j, i = np.meshgrid(np.arange(N[2]), np.arange(N[1]), np.arange(N[0]), indexing="ij")
    cell = np.stack([i.ravel(), j.ravel(), k.ravel()], axis=1)
    n = len(cell)
    o = np.full((n, 3), 0.25)
    r = np.random.default_rng(5)
    u = np.zeros((n, 3))
    for a in range(3):
        if axis is None or a == axis:
            o[:, a] = np.asarray(edges)[r.integers(0, len(edges), n)]
            u[:, a] = np.asarray(uaxis)[r.integers(0, len(uaxis), n)]
        if fp64 and (axis is None or a == axis):
            # only the first cell of an axis holds offsets with all their bits
            cell[:, a] = 0
    x = cell + o
    return x, u, np.arange(n, dtype=np.uint32)


@pytest.mark.gpu
@pytest.mark.parametrize("fp64,tol", [(False, 1e-5), (True, 1e-12)], ids=["fp32", "fp64"])
@pytest.mark.parametrize("tile", [4, 8])
@pytest.mark.parametrize("order", [1, 2])
@pytest.mark.parametrize("axis", [0, 1, 2, None])
@pytest.mark.parametrize("uaxis", [(0.0,), (0.0, 1e-9, -1e-9, 0.2, -0.2)], ids=["rest", "moving"])
def test_offsets_at_shape_boundaries(fp64, tol, tile, order, axis, uaxis):
    x, u, ids = plasma(fp64, axis, uaxis)
    z = np.zeros((3, N[2], N[1], N[0]))
    st = O.State(O.make_params(*N, C, order=order), z, z, [{"q": Q, "m": 1.0, "x": x, "u": u, "id": ids}])
    st.step(1)
    box = P.Box(P.make_config(nx=N[0], ny=N[1], nz=N[2], c=C, order=order, tile=(tile,) * 3,
                              precision=P.PIC_FP64 if fp64 else P.PIC_FP32))
    try:
        box.set_fields(z, z)
        box.load(0, Q, 1.0, x, u, ids)
        box.step(1)
        _, _, J = box.fields()
        assert box.diagnostics().error_word == 0
    finally:
        box.close()
    per_cell = np.unique(np.floor(x), axis=0, return_counts=True)[1].max()
    assert np.abs(J - st.J).max() <= tol * Q * C * per_cell
