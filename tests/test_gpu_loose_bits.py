"""FP32 results do not depend on which particles pass through the loose list.
Which do in a crowded tile depends on the order in which warps claim its slots,
so the loose particles' kernel must round as the tile kernel does: a drifting
plasma with almost no spare slots against the same with ample ones, bit for
bit, in every box kind, geometry, shape order and tile shape."""
import dataclasses

import numpy as np
import pytest

from gpu_harness import Case, run_gpu
from paper_2602_15939_gb300 import pic as P
from test_gpu_variant_bits import GEOMS, KINDS

STEPS = 5


@pytest.mark.gpu
@pytest.mark.parametrize("order", [1, 2])
@pytest.mark.parametrize("geom", GEOMS)
@pytest.mark.parametrize("kind", KINDS)
def test_fp32_bits_do_not_depend_on_the_loose_list(kind, geom, order):
    n, ndim, plane, sides = GEOMS[geom]
    box, kw = KINDS[kind]
    for side in sides:
        case = Case(kind, box, n, ndim=ndim, plane=plane, order=order, ppc=12 if ndim == 3 else 32, uth=0.2,
                    drift=(0.25, 0.1, 0.1), tile=tuple(side if n[a] > 1 else 0 for a in range(3)), **kw)
        out = []
        for slack in (0.001, 4.0):
            parts, fields, diag = run_gpu(dataclasses.replace(case, slack=slack), STEPS, False)
            assert diag.error_word == 0
            assert (diag.loose > 0) == (slack < 1.0), (side, slack, diag.loose)
            got = list(fields)
            for x, u, ids, _ in parts:
                o = np.argsort(ids)
                got += [ids[o], x[o], u[o]]
            out.append(got)
        for name, a, b in zip(("E", "B", "J", "id", "x", "u") + ("id", "x", "u"), *out):
            assert np.array_equal(a, b), (side, name, int((a != b).sum()), np.abs(a - b).max())
