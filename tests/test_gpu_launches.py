"""GPU tests of how the layer's kernels follow one another on a stream."""
import pytest
import torch

import paper_2609_34650_b200 as saf
import saf_inputs as si

from gpu_util import Layer

pytestmark = pytest.mark.gpu


def _per_call_us(call, n=40):
    best = float("inf")
    for _ in range(5):
        a, b = torch.cuda.Event(enable_timing=True), torch.cuda.Event(enable_timing=True)
        a.record()
        for _ in range(n):
            call()
        b.record()
        torch.cuda.synchronize()
        best = min(best, a.elapsed_time(b) * 1e3 / n)
    return best


@pytest.mark.parametrize("B,H,T,frozen", [(1, 12, 3072, ()), (1, 8, 4096, (3, 6))])
def test_forwards_back_to_back_take_no_longer_than_apart(B, H, T, frozen):
    """Kernels kept apart by event records cannot overlap; without the events a forward may start under the one before, which
    must not cost time.  (The events themselves add 2 us or more per kernel; 5 % are left for the clock.)"""
    L = Layer(si.generate(si.Workload("b2b", B, H, T, 64, frozen, -0.01, seed=3)), backward=False).run(backward=False)
    c = L.ctx
    call = lambda: c.saf_hybrid_attn_fwd(L.prob, L.Q, L.K, L.V, L.mask, L.alpha, L.rho, L.logZ, L.O, L.LSE)
    for _ in range(10):
        call()
    c.saf_set_profiling(1)
    for _ in range(40):
        call()
    torch.cuda.synchronize()
    apart = 0.0
    for which in (saf.SAF_KERNEL_SCALE, saf.SAF_KERNEL_FWD):
        ms, n = c.saf_get_kernel_time(which)
        apart += ms * 1e3 / n if n else 0.0
    c.saf_set_profiling(0)
    together = _per_call_us(call)
    assert together <= 1.05 * apart, (together, apart)
