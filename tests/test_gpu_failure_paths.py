"""GPU tests of the paths that only run when something is off: a bounded device wait that runs out, and pattern
tables that no longer describe the vectors a call passes."""
import numpy as np
import pytest
import torch

import paper_2609_34650_b200 as saf
import saf_inputs as si

from gpu_util import Layer
from test_gpu_parity import check_units, all_units

pytestmark = pytest.mark.gpu

DEV_TIMEOUT = 1                       # device status code in bits 24..31 of the status word
SITE_K_FULL, SITE_S_FULL = 45, 49     # wait sites of the D = 64 forward: issuer waiting for a key tile, compute
                                      # warps waiting for the scores of that tile


def test_a_wait_that_runs_out_is_reported_and_the_context_stays_usable(monkeypatch):
    """The producer of one tiny forward grid leaves out one key-tile load (a host-side switch, off by default), so the
    waits that depend on it reach their limit (20 ms here).  Every role must leave through the common teardown: the
    kernel ends, the status word names a wait site of that tile, and later calls work."""
    monkeypatch.setenv("SAF_WAIT_LIMIT_MS", "20")
    monkeypatch.setenv("SAF_SELFTEST_DROP_LOAD", "1")
    ctx = saf.Context(0)
    monkeypatch.delenv("SAF_SELFTEST_DROP_LOAD")
    monkeypatch.delenv("SAF_WAIT_LIMIT_MS")
    inp = si.generate(si.config(0))
    L = Layer(inp, ctx=ctx, backward=False)
    ctx.saf_pattern_prepare(L.mask, L.alpha, L.rho, L.logZ)
    ctx.saf_hybrid_attn_fwd(L.prob, L.Q, L.K, L.V, L.mask, L.alpha, L.rho, L.logZ, L.O, L.LSE)
    torch.cuda.synchronize()
    code, detail = ctx.saf_last_device_status()
    assert code == saf.SAF_ERR_DEVICE_TIMEOUT, (code, hex(detail))
    assert (detail >> 24) & 0xFF == DEV_TIMEOUT
    assert (detail >> 16) & 0xFF in (SITE_K_FULL, SITE_S_FULL), hex(detail)
    assert (detail & 0xFFFF) < 8                       # a CTA of the 8-item grid
    # the word was cleared by the query, and the device is fine: a context without the switch passes the same case
    code, detail = ctx.saf_last_device_status()
    assert code == saf.SAF_OK and detail == 0
    fresh = Layer(inp).run()
    check_units(fresh, all_units(inp.wl))


@pytest.mark.parametrize("D,H,T,sites", [
    (128, 80, 256, range(101, 111)),     # one query block per item (160 items: more than one per SM)
    (96, 3, 520, range(1, 12)),          # the kernel of the longer sequences (15 items of up to five tiles: the producer's
    (128, 3, 520, range(1, 12)),         # ring runs full, so its own wait gives up as well)
])
def test_a_wait_that_runs_out_in_the_wide_forwards(monkeypatch, D, H, T, sites):
    """The same at head dimensions 96 and 128, in both kernels."""
    monkeypatch.setenv("SAF_WAIT_LIMIT_MS", "20")
    monkeypatch.setenv("SAF_SELFTEST_DROP_LOAD", "1")
    ctx = saf.Context(0)
    monkeypatch.delenv("SAF_SELFTEST_DROP_LOAD")
    monkeypatch.delenv("SAF_WAIT_LIMIT_MS")
    inp = si.generate(si.Workload("drop", 1, H, T, D, (1,), -0.05, seed=D + T))
    L = Layer(inp, ctx=ctx, backward=False)
    ctx.saf_pattern_prepare(L.mask, L.alpha, L.rho, L.logZ)
    ctx.saf_hybrid_attn_fwd(L.prob, L.Q, L.K, L.V, L.mask, L.alpha, L.rho, L.logZ, L.O, L.LSE)
    torch.cuda.synchronize()
    code, detail = ctx.saf_last_device_status()
    assert code == saf.SAF_ERR_DEVICE_TIMEOUT, (code, hex(detail))
    assert (detail >> 24) & 0xFF == DEV_TIMEOUT and (detail >> 16) & 0xFF in sites, hex(detail)
    assert (detail & 0xFFFF) < 16
    code, detail = ctx.saf_last_device_status()
    assert code == saf.SAF_OK and detail == 0
    fresh = Layer(inp).run()
    check_units(fresh, all_units(inp.wl))


def test_vectors_rewritten_in_place_do_not_meet_stale_tables():
    """saf_pattern_prepare builds tensor-core tables and remembers the device pointers.  When alpha is then changed in
    place and only the normalisers are refreshed (by the entry point that has no context), the next layer call gets the
    same three pointers: it must compute the frozen heads from the new vectors, not from the old tables."""
    wl = si.Workload("stale", 2, 4, 300, 64, (1, 2), -0.05, seed=77)
    inp = si.generate(wl)
    L = Layer(inp).run()
    check_units(L, all_units(wl))
    new_alpha = (0.5 * inp.alpha + 0.3 * np.cos(0.11 * np.arange(inp.alpha.shape[1]))[None, :]).astype(np.float32)
    L.alpha.copy_(torch.from_numpy(new_alpha))          # same buffer, new contents
    saf.saf_pattern_logz_static(0, L.mask, L.alpha, L.rho, L.logZ)
    inp.alpha[...] = new_alpha
    for t in (L.O, L.LSE, *L.grads):
        t.fill_(float("nan"))
    L.run(prepare=False)
    check_units(L, all_units(wl))
    # after a new preparation the tables are used again and agree as well
    L.run(prepare=True)
    check_units(L, all_units(wl))


@pytest.mark.parametrize("D", [64, 128])
def test_a_preparation_ends_the_overflow_marks_of_recorded_calls(D):
    """A replay of a recorded forward and backward meets values that leave fp16's range, so the head takes the general form.
    The replays share the recorded call's id; with the inputs restored and the pattern prepared again they must be back at
    the tensor-core form, bit for bit."""
    wl = si.Workload("marks", 2, 3, 300, D, (1,), -0.05, seed=91)
    L = Layer(si.generate(wl))
    s = torch.cuda.Stream()
    s.wait_stream(torch.cuda.current_stream())
    with torch.cuda.stream(s):
        L.run()
        want = [L.O[:, 1].clone(), L.grads[2][:, 1].clone()]
        g = torch.cuda.CUDAGraph()
        with torch.cuda.graph(g, stream=s):
            L.ctx.saf_hybrid_attn_fwd(L.prob, L.Q, L.K, L.V, L.mask, L.alpha, L.rho, L.logZ, L.O, L.LSE)
            L.ctx.saf_hybrid_attn_bwd(L.prob, L.Q, L.K, L.V, L.O, L.dO, L.LSE, L.mask, L.alpha, L.rho, L.logZ, *L.grads)

        def replay():
            for t in (L.O, L.grads[2]):
                t.fill_(float("nan"))
            g.replay()
            s.synchronize()
            return [torch.equal(L.O[:, 1], want[0]), torch.equal(L.grads[2][:, 1], want[1])]

        assert all(replay())
        keep = L.V.clone(), L.dO.clone()
        L.V[0, 1, 5, 3] = L.dO[0, 1, 5, 3] = 1e30                # (its own unit only; the range is checked per head)
        replay()
        assert torch.isfinite(L.O[1]).all()
        L.V.copy_(keep[0])
        L.dO.copy_(keep[1])
        L.ctx.saf_pattern_prepare(L.mask, L.alpha, L.rho, L.logZ)
        assert all(replay())


def test_a_preparation_that_runs_out_of_memory_leaves_the_context_usable():
    """Larger tables are asked for while the device is full: some buffers are new by then and hold nothing.  Going back to
    the earlier pattern has to fill them again."""
    inp = si.generate(si.Workload("oom", 1, 4, 300, 64, (1, 2), -0.05, seed=5))
    L = Layer(inp).run()
    H, Tp = 2048, 4096                                   # 32 MB a vector: 600 MB of tables before the last 96 MB
    big = [torch.zeros((H, Tp), device="cuda") for _ in range(3)]
    torch.cuda.synchronize()
    torch.cuda.empty_cache()
    hold = torch.empty(torch.cuda.mem_get_info()[0] - (650 << 20), device="cuda", dtype=torch.uint8)
    with pytest.raises(saf.SafError) as e:
        L.ctx.saf_pattern_prepare(np.ones(H, dtype=np.uint8), *big)
    assert e.value.code == saf.SAF_ERR_NOMEM
    del hold, big
    torch.cuda.empty_cache()
    for t in (L.O, L.LSE, *L.grads):
        t.fill_(float("nan"))
    L.run()
    check_units(L, all_units(inp.wl))
