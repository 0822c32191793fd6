"""Media with cells so slow that kappa = (c dt / h)^2 is no FP32 number (a void
in the medium): K, K* and the medium gradient stay finite and agree with the
FP64 oracle (relative L2 <= 1e-5, the bound of every operator test) where the
state must not be kept as kappa times the adjoint field."""
import numpy as np
import pytest

import oracle
from gpu_helpers import custom, need_gpu, rel

pytestmark = pytest.mark.gpu

TOL_OP = 1e-5


def with_void(shape, nt, order, slow, seed):
    w = custom(shape, nt, order, True, 30, seed=seed)
    w.c = w.c_array().copy()
    w.c[tuple(slice(n // 4, n // 2) for n in shape)] = slow
    w.c[..., :2] = slow  # on a face as well, inside an absorbing layer
    return w


@pytest.mark.parametrize("slow", [1e-17, 1e-21], ids=["subnormal", "zero"])
@pytest.mark.parametrize("shape,order,layer", [((20, 21, 24), 4, 0), ((12, 17, 23), 8, 0), ((40, 67), 4, 0),
                                               ((40, 67), 8, 7), ((45, 66), 2, 7), ((900, 1026), 6, 7)],
                         ids=lambda s: "x".join(map(str, s)) if isinstance(s, tuple) else str(s))
def test_void(shape, order, layer, slow):
    need_gpu()
    from paper_2507_02401_gb300 import Plan
    w = with_void(shape, 40, order, slow, seed=sum(shape))
    plan = Plan(w.shape, w.h, w.dt, w.nt, w.order, w.c, w.sensors, 2, 0)
    if shape[-1] < 900:  # (the larger grid would take the persistent engine's 128 x 64 tiles with a usual medium)
        plan.path = 2
    assert plan.path == 2
    sigma = None
    if layer:
        smax = oracle.sponge_sigma_max(float(np.max(w.c)), layer, w.h)
        plan.set_sponge(layer, smax)
        sigma = oracle.sponge_sigma(w.shape, layer, smax)
    wave = oracle.Wave(w.shape, w.h, w.dt, w.nt, w.order, w.c, w.sensors, sigma=sigma)
    assert rel(plan.forward(w.x_true).cpu().numpy(), wave.forward(w.x_true)) <= TOL_OP
    r = np.random.default_rng(3).standard_normal((w.ns, w.nt))
    assert rel(plan.adjoint(r).cpu().numpy(), wave.adjoint(r)) <= TOL_OP
    if not layer:
        assert rel(plan.grad_kappa(w.x_true, r).cpu().numpy(), wave.kappa_grad(w.x_true, r)) <= TOL_OP
