"""Absorbing layer on the per-step 2D kernel where its tiles, rows and layer
interact: row lengths that are 0 to 3 cells over a multiple of 4 (rows padded to
16 bytes), last tiles of 1 and 31 rows and of few columns, both media, every
order, and records of 1 to 3 steps, against the FP64 oracle (relative L2 <=
1e-5, the bound of every operator test)."""
import numpy as np
import pytest

import oracle
from gpu_helpers import custom, make_pair, need_gpu, rel

pytestmark = pytest.mark.gpu

TOL_OP = 1e-5


@pytest.mark.parametrize("order", [2, 4, 6, 8])
@pytest.mark.parametrize("varc", [False, True])
@pytest.mark.parametrize("shape,nt", [((33, 68), 40), ((63, 65), 40), ((65, 130), 40), ((40, 67), 40), ((65, 70), 1),
                                      ((65, 71), 2), ((33, 69), 3)],
                         ids=lambda s: "x".join(map(str, s)) if isinstance(s, tuple) else str(s))
def test_layer_step2d_tile_edges(shape, nt, order, varc):
    need_gpu()
    w = custom(shape, nt, order, varc, 40, seed=sum(shape) + order)
    plan, _, _ = make_pair(w, path=2)
    smax = oracle.sponge_sigma_max(float(np.max(w.c_array())), 9, w.h)
    plan.set_sponge(9, smax)
    wave = oracle.Wave(w.shape, w.h, w.dt, w.nt, w.order, w.c_array(), w.sensors,
                       sigma=oracle.sponge_sigma(w.shape, 9, smax))
    assert rel(plan.forward(w.x_true).cpu().numpy(), wave.forward(w.x_true)) <= TOL_OP
    r = np.random.default_rng(7).standard_normal((w.ns, w.nt))
    assert rel(plan.adjoint(r).cpu().numpy(), wave.adjoint(r)) <= TOL_OP
    assert plan.check() == 0
