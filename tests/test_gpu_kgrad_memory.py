"""Memory of the medium gradient: what the first call was granted serves the
later ones, and the long default segments stay within their bounds."""
import numpy as np
import pytest

from gpu_helpers import custom, make_pair, need_gpu

pytestmark = pytest.mark.gpu


def captured(torch, plan, x, r):
    """grad_kappa in a captured stream, replayed; fails if the call allocates."""
    from paper_2507_02401_gb300 import _lib
    g = torch.zeros(plan.shape, device="cuda")
    graph = torch.cuda.CUDAGraph()
    with torch.cuda.graph(graph):
        _lib.pat_grad_kappa(plan.handle, x, r, g, 0, torch.cuda.current_stream())
    graph.replay()
    torch.cuda.synchronize()
    return g


def test_default_segment_is_kept_when_the_long_one_does_not_fit():
    """With less memory free than the long default segment takes (1 GiB here)
    the first call settles on sqrt(nt); the second finds those buffers: it
    allocates and frees nothing, so that it can be captured, and its bits are
    those of the first."""
    torch = need_gpu()
    w = custom((1024, 1024), 257, 2, False, 16, seed=5)
    plan, _, _ = make_pair(w)
    x = torch.as_tensor(w.x_true, dtype=torch.float32, device="cuda")
    r = torch.as_tensor(np.random.default_rng(5).standard_normal((w.ns, w.nt)), dtype=torch.float32, device="cuda")
    ref = plan.grad_kappa(x, r, segment=64)  # loads the kernels; frees its buffers below
    plan.close()
    plan, _, _ = make_pair(w)
    torch.cuda.empty_cache()
    free = torch.cuda.mem_get_info()[0]
    fill = torch.empty(free - (900 << 20), dtype=torch.uint8, device="cuda")
    try:
        g = plan.grad_kappa(x, r)
        used = torch.cuda.mem_get_info()[0]
        assert used > 200 << 20  # not the long segment
        assert torch.equal(captured(torch, plan, x, r), g)
        assert torch.equal(g, ref)
    finally:
        del fill
        torch.cuda.empty_cache()
    # room again: an explicit segment still replaces the buffers, and the default comes back
    assert torch.equal(plan.grad_kappa(x, r, segment=100), ref)
    assert torch.equal(plan.grad_kappa(x, r), ref)


def gradient_bytes(torch, plan, x, r):
    """Device memory that the plan's first default call takes for good."""
    free = torch.cuda.mem_get_info()[0]
    plan.grad_kappa(x, r)
    torch.cuda.synchronize()
    torch.cuda.empty_cache()
    return free - torch.cuda.mem_get_info()[0]


def test_default_segments_of_many_plans_are_bounded():
    """One plan takes 1 GiB for its long segment here; ten take 4 GiB between
    them and sqrt(nt) segments beyond that (under 0.35 GB each), with the same
    bits; what one gives back the next may take."""
    torch = need_gpu()
    w = custom((1024, 1024), 257, 2, False, 16, seed=5)
    x = torch.as_tensor(w.x_true, dtype=torch.float32, device="cuda")
    r = torch.as_tensor(np.random.default_rng(5).standard_normal((w.ns, w.nt)), dtype=torch.float32, device="cuda")
    plans = [make_pair(w)[0] for _ in range(10)]
    used = [gradient_bytes(torch, p, x, r) for p in plans]
    assert used[0] > 1 << 30
    assert sum(used) <= (4 << 30) + 10 * 350e6
    assert torch.equal(plans[0].grad_kappa(x, r), plans[-1].grad_kappa(x, r))
    for p in plans:
        p.close()
    again = make_pair(w)[0]
    assert gradient_bytes(torch, again, x, r) > 1 << 30
    again.grad_kappa(x, r, segment=16)  # gives its long segment back as well
    rest = [make_pair(w)[0] for _ in range(3)]
    assert all(gradient_bytes(torch, p, x, r) > 1 << 30 for p in rest)


def test_default_segment_leaves_a_full_device_alone():
    """With 4 GB free the default is sqrt(nt): an eighth of that is less than the long segment."""
    torch = need_gpu()
    w = custom((1024, 1024), 257, 2, False, 16, seed=5)
    x = torch.as_tensor(w.x_true, dtype=torch.float32, device="cuda")
    r = torch.as_tensor(np.random.default_rng(5).standard_normal((w.ns, w.nt)), dtype=torch.float32, device="cuda")
    plan = make_pair(w)[0]
    torch.cuda.empty_cache()
    fill = torch.empty(torch.cuda.mem_get_info()[0] - (4 << 30), dtype=torch.uint8, device="cuda")
    try:
        assert gradient_bytes(torch, plan, x, r) < 350e6
    finally:
        del fill
        torch.cuda.empty_cache()
