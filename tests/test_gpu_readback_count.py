"""A box that lost particles (more of them arrived in one tile in one step than
its slots and the loose list hold: the step reports it) refuses the read-back
as PIC_ERR_STATE before anything is written, into host and into device arrays."""
import itertools

import numpy as np
import pytest

from paper_2602_15939_gb300 import pic as P

N, PER = 16, 1000


@pytest.mark.gpu
@pytest.mark.parametrize("precision", [P.PIC_FP32, P.PIC_FP64], ids=["fp32", "fp64"])
def test_wrong_particle_count_leaves_the_arrays_alone(precision):
    torch = pytest.importorskip("torch")
    # 7 x 1000 uncharged particles around the corner of eight 8^3 tiles, all
    # moving into the eighth: it has 1.001 x 1000 + 32 slots, the list 4096
    r = np.random.default_rng(2)
    x, u = [], []
    for bits in itertools.product((0, 1), repeat=3):
        if bits == (1, 1, 1):
            continue
        b = np.asarray(bits)
        x.append(np.where(b, 8.05, 7.85) + r.uniform(0.0, 0.1, (PER, 3)))
        v = np.where(b, 0.0, 0.2)
        u.append(np.tile(v / np.sqrt(1.0 - (v @ v) / 0.45**2), (PER, 1)))  # u = gamma v
    x, u = np.concatenate(x), np.concatenate(u)
    box = P.Box(P.make_config(nx=N, ny=N, nz=N, c=0.45, precision=precision, tile=(8, 8, 8), capacity_slack=0.001))
    try:
        box.set_uniform_fields((0.0, 0.0, 0.0), (0.0, 0.0, 0.0))
        box.load(0, 0.0, 1.0, x, u)
        box.step(1)
        with pytest.raises(P.PicError) as e:
            box.diagnostics()
        assert e.value.status == P.PIC_ERR_STATE and "loose" in str(e.value)
        box.clear_error()
        n = len(x)
        for device in ("cpu", "cuda"):
            bufs = [torch.full((n, 3), -7.0, dtype=torch.float64, device=device) for _ in range(3)]
            ids = torch.full((n,), -7, dtype=torch.int32, device=device)
            torch.cuda.synchronize()
            st = P.lib().pic_get_particles(box.h, 0, P.C.cast(bufs[0].data_ptr(), P._D),
                                           P.C.cast(bufs[1].data_ptr(), P._D), P.C.cast(ids.data_ptr(), P._U32),
                                           P.C.cast(bufs[2].data_ptr(), P._D))
            assert st == P.PIC_ERR_STATE
            torch.cuda.synchronize()
            assert all(bool((b == -7.0).all()) for b in bufs) and bool((ids == -7).all()), device
    finally:
        box.close()
