"""Wave kernels at the sizes where their tiles, lists and pipelines end, against
the FP64 oracle (relative L2 <= 1e-5 per operator, the bound of every operator
test: FP32 fields and coefficients over some tens of steps stay below ~1e-6).

Covers the per-step TMA kernels on grids of any width (rows padded to 16
bytes) in 2D and 3D, 3D varying media, the medium gradient of the 2D step
engine on ragged time segments, both tile sizes of the persistent 2D engine,
and the batched kernel one cell either side of its tile."""
import numpy as np
import pytest

import oracle
from gpu_helpers import custom, make_pair, need_gpu, rel

pytestmark = pytest.mark.gpu

TOL_OP = 1e-5


def check_operators(w, plan, wave):
    assert rel(plan.forward(w.x_true).cpu().numpy(), wave.forward(w.x_true)) <= TOL_OP
    r = np.random.default_rng(7).standard_normal((w.ns, w.nt))
    assert rel(plan.adjoint(r).cpu().numpy(), wave.adjoint(r)) <= TOL_OP
    assert plan.check() == 0


@pytest.mark.parametrize("order", [2, 4, 6, 8])
@pytest.mark.parametrize("varc", [False, True])
@pytest.mark.parametrize("shape", [(31, 63), (32, 64), (33, 65), (65, 129), (9, 194), (130, 7)],
                         ids=lambda s: "x".join(map(str, s)))
def test_step2d_tile_edges(shape, order, varc):
    need_gpu()
    w = custom(shape, 40, order, varc, 40, seed=sum(shape) + order)
    plan, wave, _ = make_pair(w, path=2)
    check_operators(w, plan, wave)


@pytest.mark.parametrize("shape,order,varc,nt", [((33, 65), 8, True, 2), ((33, 65), 4, False, 3), ((64, 70), 6, True, 17),
                                                 ((31, 127), 2, True, 26), ((40, 63), 8, False, 50)])
def test_grad_kappa_segments(shape, order, varc, nt):
    need_gpu()
    w = custom(shape, nt, order, varc, 9, seed=nt)
    plan, wave, _ = make_pair(w, path=2)
    r = np.random.default_rng(3).standard_normal((w.ns, w.nt))
    ref = wave.kappa_grad(w.x_true, r)
    for segment in (0, 1, nt - 1, 5):
        if 0 <= segment <= nt - 1:
            assert rel(plan.grad_kappa(w.x_true, r, segment=segment).cpu().numpy(), ref) <= TOL_OP


@pytest.mark.parametrize("order", [2, 4, 6, 8])
@pytest.mark.parametrize("varc", [False, True])
@pytest.mark.parametrize("shape,nt", [((17, 16, 65), 24), ((9, 17, 63), 24), ((40, 31, 66), 20), ((5, 33, 7), 12),
                                      ((6, 15, 64), 1), ((6, 15, 64), 2), ((6, 17, 65), 3)],
                         ids=lambda s: "x".join(map(str, s)) if isinstance(s, tuple) else str(s))
def test_step3d_tile_edges(shape, nt, order, varc):
    need_gpu()
    w = custom(shape, nt, order, varc, 25, seed=sum(shape) + order)
    plan, wave, _ = make_pair(w)
    check_operators(w, plan, wave)


@pytest.mark.parametrize("order", [2, 4, 6, 8])
@pytest.mark.parametrize("varc", [False, True])
@pytest.mark.parametrize("shape,nt", [((31, 63), 30), ((33, 65), 30), ((66, 129), 30), ((64, 128), 160), ((15, 200), 30)],
                         ids=lambda s: "x".join(map(str, s)) if isinstance(s, tuple) else str(s))
def test_persistent_tile_edges(shape, nt, order, varc):
    need_gpu()
    w = custom(shape, nt, order, varc, 60, seed=sum(shape) + order)
    plan, wave, _ = make_pair(w, path=1)
    check_operators(w, plan, wave)


# grids that take the persistent engine's 128 x 64 tiles: (shape, order, varying medium)
LARGE = [((1024, 1024), 8, False), ((897, 961), 8, False), ((129, 6400), 8, False), ((1024, 1025), 6, False),
         ((641, 1000), 6, False), ((1024, 1025), 6, True), ((900, 1026), 6, True), ((63, 12800), 4, True),
         ((895, 1087), 4, True), ((570, 571), 4, False), ((1150, 1001), 2, True), ((1216, 1020), 2, False)]


@pytest.mark.parametrize("shape,order,varc", LARGE, ids=lambda s: "x".join(map(str, s)) if isinstance(s, tuple) else str(s))
@pytest.mark.parametrize("layer", [0, 9])
def test_persistent_large_tile_edges(shape, order, varc, layer):
    need_gpu()
    w = custom(shape, 40, order, varc, 700, seed=sum(shape) + order)
    plan, wave, _ = make_pair(w)
    assert plan.path == 1
    if layer:
        smax = oracle.sponge_sigma_max(float(np.max(w.c_array())), layer, w.h)
        plan.set_sponge(layer, smax)
        wave = oracle.Wave(w.shape, w.h, w.dt, w.nt, w.order, w.c_array(), w.sensors,
                           sigma=oracle.sponge_sigma(w.shape, layer, smax))
    check_operators(w, plan, wave)


@pytest.mark.parametrize("nt", [1, 2, 3, 140])
@pytest.mark.parametrize("order", [2, 8])
def test_persistent_large_time_axis(nt, order):
    """Short axes, and one past the adjoint's step tags (7 bits); sensors in the corners of the tiles."""
    torch = need_gpu()
    w = custom((960, 1001), nt, order, order == 2, 48, seed=nt)
    k = 0
    for y in (63, 64, 127, 128, 895, 896):  # blocks of 2 x 2 cells that straddle tile corners, edges and frames
        for x in (7, 8, 119, 120, 127, 128, 255, 895):
            w.sensors[k] = ((x + 0.4) * w.h, (y + 0.3) * w.h)
            k += 1
    plan, wave, _ = make_pair(w, path=1)
    check_operators(w, plan, wave)
    # an image that starts 4 bytes off a 16-byte boundary, in and out
    buf = torch.zeros(w.x_true.size + 1, device="cuda")
    x = buf[1:].view(w.shape)
    x.copy_(torch.as_tensor(w.x_true, dtype=torch.float32))
    assert torch.equal(plan.forward(x), plan.forward(w.x_true))
    r = np.random.default_rng(5).standard_normal((w.ns, w.nt))
    ref = plan.adjoint(r)
    plan.adjoint(r, out=x)
    assert torch.equal(x, ref)


@pytest.mark.parametrize("order", [2, 4, 8])
def test_batch_tile_edges(order):
    need_gpu()
    from paper_2507_02401_gb300 import Batch
    shapes = [(31, 64), (32, 60), (33, 68), (64, 64), (65, 132), (8, 8)]
    ws = [custom(s, 30 + 7 * i, order, bool(i % 2), 11, seed=i, levels=0) for i, s in enumerate(shapes)]
    pairs = [make_pair(w) for w in ws]
    batch = Batch([p for p, _, _ in pairs])
    for w, (_, wave, _), y in zip(ws, pairs, batch.forward([w.x_true for w in ws])):
        assert rel(y.cpu().numpy(), wave.forward(w.x_true)) <= TOL_OP
    rs = [np.random.default_rng(i).standard_normal((w.ns, w.nt)) for i, w in enumerate(ws)]
    for r, (_, wave, _), x in zip(rs, pairs, batch.adjoint(rs)):
        assert rel(x.cpu().numpy(), wave.adjoint(r)) <= TOL_OP
