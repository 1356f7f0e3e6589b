"""GPU parity of the compact-pattern fitter (target marginals, Fit, acceptance statistic) against the fp64 oracle.

Tolerances.  The kernels round the factors exp(alpha) and exp(rho) to fp32 once per step (2^-25 relative) and sum their
products in fp32: chains of 64 terms, then the pieces of a warp (each chain of n positive terms rounds off up to n 2^-25,
typically sqrt(n) times less), the warps' parts and Adam in fp64; heads that leave the product's range take one ex2.approx
per term instead (2^-22, on an argument rounded at magnitudes up to ~60).  That is up to a few 1e-6 relative per
sum.  Marginals and normalisers are sums of positive terms, so they inherit that relative error: 2e-5 relative is
asserted.  Over the Adam steps the difference in the gradients (about 1e-6 relative) moves the parameters by far less
than one step (0.05) each time; the asserted bound on alpha, rho after J steps is 2e-3 absolute for J <= 50 and
2e-2 after 400 steps, with the quantities that do not depend on the path (loss, kappa: 1e-4 absolute) held tighter,
and the returned log Z, loss and kappa checked against the oracle evaluated AT the returned parameters (1e-4)."""
import numpy as np
import pytest
import torch

import paper_2609_34650_b200 as saf
import saf_inputs as si
from oracle import saf_fit_oracle as fo

pytestmark = pytest.mark.gpu


def _ctx():
    return saf.Context(0)


@pytest.fixture(params=["transforms", "direct"])
def form(request, monkeypatch):
    """A context whose fits beyond 128 positions start with the transforms, and one that takes the direct sums throughout."""
    if request.param == "direct":
        monkeypatch.setenv("SAF_FIT_DIRECT", "1")
    return request.param, saf.Context(0)


def _status(ctx):
    torch.cuda.synchronize()
    code, detail = ctx.saf_last_device_status()
    assert code == saf.SAF_OK, f"device status {code} detail {detail:#x}"


def _gpu_marginals(ctx, A):
    Hf, T, _ = A.shape
    dA = torch.from_numpy(A).cuda()
    ea = torch.full((Hf, T), float("nan"), dtype=torch.float64, device="cuda")
    er = torch.full((Hf, T), float("nan"), dtype=torch.float64, device="cuda")
    pl = torch.full((Hf,), float("nan"), dtype=torch.float64, device="cuda")
    ctx.saf_fit_marginals(Hf, T, dA, 1e-9, ea, er, pl)
    _status(ctx)
    return ea, er, pl


def _gpu_fit(ctx, ea, er, pl, steps, lr=0.05, stride=None):
    Hf, T = ea.shape
    stride = stride or T
    out = [torch.full((Hf, stride), float("nan"), dtype=torch.float32, device="cuda") for _ in range(3)]
    loss = torch.full((Hf,), float("nan"), dtype=torch.float64, device="cuda")
    kl = torch.full((Hf,), float("nan"), dtype=torch.float64, device="cuda")
    ctx.saf_fit_compact(Hf, T, ea, er, pl, steps, lr, out[0], out[1], out[2], stride, loss, kl)
    _status(ctx)
    a, r, z = (t.cpu().numpy().astype(np.float64) for t in out)
    return a, r, z, loss.cpu().numpy(), kl.cpu().numpy()


def _oracle_stats(A):
    P = [fo.target_from_mean_attention(A[h]) for h in range(A.shape[0])]
    st = [fo.marginals(p) for p in P]
    ea = np.stack([s[0] for s in st])
    er = np.stack([s[1] for s in st])
    pl = np.array([s[2] for s in st])
    return P, ea, er, pl


def _dev(x):
    return torch.from_numpy(np.ascontiguousarray(x, dtype=np.float64)).cuda()


# ------------------------------------------------------------------------------------------------ marginals
@pytest.mark.parametrize("Hf,T,seed", [(2, 300, 1), (3, 1100, 2), (1, 2500, 3), (1, 1, 4), (2, 33, 5),
                                       (1, 5000, 6), (1, 8200, 7)])       # (the last two: 32 columns per thread)
def test_marginals_parity(Hf, T, seed):
    # garbage above the diagonal must be ignored; a steep decay puts entries under the 1e-9 floor
    A = si.mean_attention_maps(Hf, T, seed, upper_fill=7.0, pmax=5.0)
    if T == 1100:
        tri = np.tril_indices(T)
        assert any((A[h][tri] < 1e-9).any() for h in range(Hf)), "the case should exercise the floor"
    P, ea, er, pl = _oracle_stats(A)
    g_ea, g_er, g_pl = (t.cpu().numpy() for t in _gpu_marginals(_ctx(), A))
    assert np.isfinite(g_ea).all() and np.isfinite(g_er).all() and np.isfinite(g_pl).all()
    assert np.max(np.abs(g_ea - ea) / ea) < 2e-5
    assert np.max(np.abs(g_er - er) / er) < 2e-5
    assert np.max(np.abs(g_pl - pl)) < 2e-5 * T + 1e-9
    # each marginal distributes the T units of row mass
    assert np.max(np.abs(g_ea.sum(axis=1) - T)) < 2e-5 * T


def test_marginals_many_heads_one_cta_each():
    # more heads than three CTAs per SM: one CTA per head walks every row
    Hf, T = 500, 64
    base = si.mean_attention_maps(4, T, 9)
    A = np.ascontiguousarray(base[np.arange(Hf) % 4])
    _, ea, er, pl = _oracle_stats(base)
    g_ea, g_er, g_pl = (t.cpu().numpy() for t in _gpu_marginals(_ctx(), A))
    for h in (0, 1, 250, 499):
        assert np.max(np.abs(g_ea[h] - ea[h % 4]) / ea[h % 4]) < 2e-5
        assert np.max(np.abs(g_er[h] - er[h % 4]) / er[h % 4]) < 2e-5
        assert abs(g_pl[h] - pl[h % 4]) < 2e-5 * T


# ------------------------------------------------------------------------------------------------ Fit
def _check_self_consistent(a, r, z, loss, kl, P, ea, er, pl, tol=1e-4):
    """Returned log Z, loss and kappa against the oracle evaluated at the RETURNED parameters."""
    for h in range(a.shape[0]):
        T = ea.shape[1]
        want_z, _ = fo._logZ_and_P(a[h, :T], r[h, :T])
        assert np.max(np.abs(z[h, :T] - want_z)) < tol
        assert abs(loss[h] - fo.fit_objective(a[h, :T], r[h, :T], ea[h], er[h])) < tol
        assert abs(kl[h] - fo.fit_kl_dense(P[h], a[h, :T], r[h, :T])) < tol


@pytest.mark.parametrize("T,steps,tol", [(300, 0, 1e-6), (300, 1, 1e-4), (300, 5, 5e-4), (517, 50, 2e-3), (96, 400, 2e-2),
                                         (1, 3, 1e-6), (2, 10, 1e-4), (33, 20, 1e-3)])
def test_fit_parity(T, steps, tol):
    Hf = 2
    A = si.mean_attention_maps(Hf, T, 11 + T)
    P, ea, er, pl = _oracle_stats(A)
    a, r, z, loss, kl = _gpu_fit(_ctx(), _dev(ea), _dev(er), _dev(pl), steps)
    assert all(np.isfinite(x).all() for x in (a, r, z, loss, kl))
    for h in range(Hf):
        wa, wr, wz = fo.fit_compact(ea[h], er[h], steps=steps, lr=0.05)
        assert np.max(np.abs(a[h] - wa)) < tol, f"alpha head {h}: {np.max(np.abs(a[h] - wa)):.3e}"
        assert np.max(np.abs(r[h] - wr)) < tol, f"rho head {h}: {np.max(np.abs(r[h] - wr)):.3e}"
        assert np.max(np.abs(z[h] - wz)) < max(2 * tol, 1e-5)
        assert abs(loss[h] - fo.fit_objective(wa, wr, ea[h], er[h])) < 1e-4
        assert abs(kl[h] - fo.fit_kl_dense(P[h], wa, wr)) < 1e-4
    _check_self_consistent(a, r, z, loss, kl, P, ea, er, pl)


def test_fit_long_sequence_two_steps():
    """T beyond 4096, not a multiple of a block of 256 positions."""
    T = 5000
    A = si.mean_attention_maps(1, T, 31)
    P, ea, er, pl = _oracle_stats(A)
    a, r, z, loss, kl = _gpu_fit(_ctx(), _dev(ea), _dev(er), _dev(pl), 2)
    wa, wr, wz = fo.fit_compact(ea[0], er[0], steps=2)
    assert np.max(np.abs(a[0] - wa)) < 2e-4 and np.max(np.abs(r[0] - wr)) < 2e-4 and np.max(np.abs(z[0] - wz)) < 1e-4
    assert abs(kl[0] - fo.fit_kl_dense(P[0], wa, wr)) < 1e-4


def test_fit_start_is_prescribed_point():
    T = 130
    A = si.mean_attention_maps(1, T, 3)
    P, ea, er, pl = _oracle_stats(A)
    a, r, z, loss, kl = _gpu_fit(_ctx(), _dev(ea), _dev(er), _dev(pl), 0)
    assert np.all(a == 0)
    want = np.log(np.maximum(er[0] / (T - np.arange(T)), 1e-9))
    assert np.max(np.abs(r[0] - want)) < 1e-6 * np.max(np.abs(want))


def test_fit_output_stride_and_untouched_padding():
    T, stride = 100, 160
    A = si.mean_attention_maps(2, T, 5)
    P, ea, er, pl = _oracle_stats(A)
    a, r, z, loss, kl = _gpu_fit(_ctx(), _dev(ea), _dev(er), _dev(pl), 3, stride=stride)
    assert np.isfinite(a[:, :T]).all() and np.isnan(a[:, T:]).all() and np.isnan(z[:, T:]).all()
    for h in range(2):
        wa, wr, wz = fo.fit_compact(ea[h], er[h], steps=3)
        assert np.max(np.abs(a[h, :T] - wa)) < 5e-4 and np.max(np.abs(r[h, :T] - wr)) < 5e-4


def test_fit_end_to_end_with_acceptance():
    """Mean attention map -> marginals -> Fit -> kappa, all on the GPU, against Algorithm 1's loop body."""
    Hf, T = 3, 200
    A = si.mean_attention_maps(Hf, T, 17)
    ctx = _ctx()
    ea, er, pl = _gpu_marginals(ctx, A)
    a, r, z, loss, kl = _gpu_fit(ctx, ea, er, pl, 400)
    for h in range(Hf):
        wa, wr, wz, kappa, ok = fo.fit_head(A[h], steps=400)
        assert abs(kl[h] - kappa) < 1e-4
        if abs(kappa - 0.2) > 1e-3:
            assert (kl[h] <= 0.2) == ok
        assert np.max(np.abs(a[h] - wa)) < 2e-2 and np.max(np.abs(r[h] - wr)) < 2e-2
        # the reconstructed pattern is what matters downstream: rows of P^ from the two parameter sets
        _, Pg = fo._logZ_and_P(a[h], r[h])
        _, Pw = fo._logZ_and_P(wa, wr)
        assert np.max(np.abs(Pg - Pw)) < 2e-3


def test_fit_planted_pattern_recovered():
    # a target that is itself a compact pattern: kappa must come out near zero and far below its starting value
    T = 256
    rng = np.random.default_rng(4)
    alpha = 0.5 * rng.standard_normal(T)
    alpha[0] += 3.0
    rho = -0.05 * np.arange(T) + 0.1 * rng.standard_normal(T)
    _, P = fo._logZ_and_P(alpha, rho)
    ea, er, pl = fo.marginals(P)
    ctx = _ctx()
    args = (_dev(ea[None]), _dev(er[None]), _dev(np.array([pl])))
    _, _, _, _, kl0 = _gpu_fit(ctx, *args, 0)
    a, r, z, loss, kl = _gpu_fit(ctx, *args, 400)
    assert 0 <= kl[0] + 1e-6 and kl[0] < 0.02 and kl[0] < 0.1 * kl0[0]
    assert abs(kl[0] - fo.fit_kl_dense(P, a[0], r[0])) < 1e-4


def test_fit_full_size_config1_heads():
    """The benchmark's shape (T = 4096, three heads): a few steps element-wise, then 400 steps checked through
    what holds at any size (the returned normalisers, loss and kappa belong to the returned parameters)."""
    Hf, T = 3, 4096
    A = si.mean_attention_maps(1, T, 23)
    A = np.ascontiguousarray(np.repeat(A, Hf, axis=0))
    A[1] = np.tril(A[1] ** 1.3)
    A[2] = np.tril(A[2] ** 0.7)
    ctx = _ctx()
    ea, er, pl = _gpu_marginals(ctx, A)
    P0 = fo.target_from_mean_attention(A[1])
    wea, wer, wpl = fo.marginals(P0)
    g_ea, g_er = ea.cpu().numpy(), er.cpu().numpy()
    assert np.max(np.abs(g_ea[1] - wea) / wea) < 2e-5 and np.max(np.abs(g_er[1] - wer) / wer) < 2e-5
    assert abs(pl.cpu().numpy()[1] - wpl) < 2e-5 * T
    a, r, z, loss, kl = _gpu_fit(ctx, ea, er, pl, 2)
    wa, wr, wz = fo.fit_compact(wea, wer, steps=2)
    assert np.max(np.abs(a[1] - wa)) < 2e-4 and np.max(np.abs(r[1] - wr)) < 2e-4 and np.max(np.abs(z[1] - wz)) < 1e-4
    a, r, z, loss, kl = _gpu_fit(ctx, ea, er, pl, 400)
    want_z, _ = fo._logZ_and_P(a[1], r[1])
    assert np.max(np.abs(z[1] - want_z)) < 1e-4
    assert abs(loss[1] - fo.fit_objective(a[1], r[1], wea, wer)) < 1e-4
    assert abs(kl[1] - fo.fit_kl_dense(P0, a[1], r[1])) < 1e-4
    start = fo.fit_kl_from_stats(*fo.fit_init(wer), wea, wer, wpl)
    assert kl[1] < start


# ------------------------------------------------------------------------------------------------ edges
def test_fit_no_heads_and_bad_arguments():
    ctx = _ctx()
    z = torch.zeros(4, dtype=torch.float64, device="cuda")
    f = torch.zeros(4, dtype=torch.float32, device="cuda")
    ctx.saf_fit_marginals(0, 4, None, 1e-9, z, z, z)          # no heads: nothing to do
    ctx.saf_fit_compact(0, 4, z, z, z, 5, 0.05, f, f, f, 4, None, None)
    for call in (lambda: ctx.saf_fit_marginals(1, 0, f, 1e-9, z, z, z),
                 lambda: ctx.saf_fit_marginals(1, 4, f, 0.0, z, z, z),
                 lambda: ctx.saf_fit_marginals(1, 4, None, 1e-9, z, z, z),
                 lambda: ctx.saf_fit_compact(1, 4, z, z, z, -1, 0.05, f, f, f, 4, None, None),
                 lambda: ctx.saf_fit_compact(1, 4, z, z, z, 1, 0.0, f, f, f, 4, None, None),
                 lambda: ctx.saf_fit_compact(1, 4, z, z, z, 1, 0.05, f, f, f, 3, None, None),
                 lambda: ctx.saf_fit_compact(1, 4, z, z, None, 1, 0.05, f, f, f, 4, None, z)):
        with pytest.raises(saf.SafError) as e:
            call()
        assert e.value.code == saf.SAF_ERR_INVALID_ARG
    with pytest.raises(saf.SafError) as e:
        ctx.saf_fit_compact(1, 16385, z, z, z, 1, 0.05, f, f, f, 16385, None, None)
    assert e.value.code == saf.SAF_ERR_UNSUPPORTED
    _status(ctx)


# The direct sums: a cluster of CTAs per head.  Edges: blocks of 256 positions (one, two, a partial one), more heads
# than clusters fit at once, two to sixteen CTAs per cluster, and the longest sequences (12 warps instead of 16 beyond 8192
# positions, vectors kept unpadded beyond 12288).  The transforms at the same sizes.
@pytest.mark.parametrize("Hf,T,steps", [(1, 255, 3), (2, 257, 3), (1, 2304, 2), (150, 272, 2), (40, 300, 2), (1, 10300, 1),
                                        (1, 12289, 1), (16, 1500, 2)])
def test_fit_cluster_edges(form, Hf, T, steps):
    name, ctx = form
    base = si.mean_attention_maps(1, T, 40 + T)
    P, ea, er, pl = _oracle_stats(base)
    rep = lambda v: _dev(np.repeat(v, Hf, axis=0))
    a, r, z, loss, kl = _gpu_fit(ctx, rep(ea), rep(er), rep(pl), steps)
    assert (ctx.saf_fit_handover(Hf) == (0 if name == "direct" else -1)).all()
    for x in (a, r, z, loss, kl):
        assert np.array_equal(x, np.broadcast_to(x[:1], x.shape))             # every head ran the same program
    wa, wr, wz = fo.fit_compact(ea[0], er[0], steps=steps)
    assert np.max(np.abs(a[0] - wa)) < 2e-4 and np.max(np.abs(r[0] - wr)) < 2e-4 and np.max(np.abs(z[0] - wz)) < 1e-4
    assert abs(kl[0] - fo.fit_kl_dense(P[0], wa, wr)) < 1e-4


# Parameters beyond 2^+-50 (2^-70): the head goes on with logarithms.  Steps of 10 nats cross the bounds within four
# steps; magnitudes reach a few hundred nats, where an fp32 exponent argument carries 2^-24 * 2^9 = 3e-5 nats per
# rounding, so 5e-4 is asserted on log Z (about ten roundings) against the fp64 normalisers at the returned parameters.
@pytest.mark.parametrize("T,steps", [(100, 12), (700, 8)])
def test_fit_leaves_the_product_range(form, T, steps):
    name, ctx = form
    A = si.mean_attention_maps(2, T, 50 + T)
    P, ea, er, pl = _oracle_stats(A)
    a, r, z, loss, kl = _gpu_fit(ctx, _dev(ea), _dev(er), _dev(pl), steps, lr=10.0)
    at = ctx.saf_fit_handover(2)
    assert (at == 0).all() if name == "direct" or T <= 128 else (at >= 1).all()
    assert max(np.abs(a).max(), np.abs(r).max()) > 50 * np.log(2)
    for h in range(2):
        want_z, _ = fo._logZ_and_P(a[h], r[h])
        assert np.max(np.abs(z[h] - want_z)) < 5e-4
        assert abs(loss[h] - fo.fit_objective(a[h], r[h], ea[h], er[h])) < 5e-4 * max(1.0, abs(loss[h]))


def test_first_step_and_loss_keep_the_accuracy_of_their_terms(form):
    """The first Adam step moves alpha by lr sign(g) / (1 + 1e-8 / |g|), so that small gradients show the rounding of the
    column sums; at 40 heads a warp's chains are longest.  The loss at the returned parameters averages T normalisers, where
    only what is common to them would remain.  Chains of 64 terms round off about sqrt(64/3) 2^-25 = 1.4e-7 of a sum (measured
    3.7e-7 in alpha; 1.9e-6 with chains of 512); the loss is asserted at a quarter of the rounding 2^-25 that one fp32 factor
    common to all rows would leave (measured 3e-9; 2e-8 with the factors' own rounding in it)."""
    ctx = form[1]
    T, Hf = 4096, 40
    base = si.mean_attention_maps(1, T, 40 + T)
    P, ea, er, pl = _oracle_stats(base)
    rep = lambda v: _dev(np.repeat(v, Hf, axis=0))
    a, r, z, loss, kl = _gpu_fit(ctx, rep(ea), rep(er), rep(pl), 1)
    wa, wr, wz = fo.fit_compact(ea[0], er[0], steps=1)
    assert np.linalg.norm(a[0] - wa) <= 1e-6 * np.linalg.norm(wa)
    A = si.mean_attention_maps(6, 512, 9)
    P, ea, er, pl = _oracle_stats(A)
    a, r, z, loss, kl = _gpu_fit(ctx, _dev(ea), _dev(er), _dev(pl), 400)
    err = [loss[h] / fo.fit_objective(a[h], r[h], ea[h], er[h]) - 1.0 for h in range(6)]
    assert np.sqrt(np.mean(np.square(err))) <= 2.0 ** -27, err


def test_a_single_long_head_spreads_over_more_than_eight_sms(monkeypatch):
    """The direct sums.  Twice the length is four times the multiply-adds beside the fixed costs of a step; on eight CTAs, the largest portable
    cluster, they take over (a factor of 3.2 from 4096 to 8192 positions), on sixteen not yet."""
    us = {}
    for T in (4096, 8192):
        g = torch.Generator(device="cuda").manual_seed(T)
        eta = torch.rand((1, T), generator=g, device="cuda", dtype=torch.float64) * 2.0
        o = [torch.empty((1, T), device="cuda") for _ in range(3)]
        one = torch.zeros(1, device="cuda", dtype=torch.float64)
        monkeypatch.setenv("SAF_FIT_DIRECT", "1")
        ctx = saf.Context(0)
        for _ in range(4):
            a, b = torch.cuda.Event(enable_timing=True), torch.cuda.Event(enable_timing=True)
            a.record()
            ctx.saf_fit_compact(1, T, eta, eta, one, 50, 0.05, *o, T, one.clone(), one.clone())
            b.record()
            torch.cuda.synchronize()
            us[T] = min(us.get(T, 1e9), a.elapsed_time(b) * 20.0)
    assert us[8192] <= 2.5 * us[4096], us                # measured 22.8 and 44.4 us a step; on eight SMs 25.4 and 80.4


# ------------------------------------------------------------------------------------------------ the transform form
# Transforms of 256, 512 points in one CTA, 1024, 2048, 4096 in two, four, eight CTAs of 512, 8192 and 16384 in eight of 1024
# and 2048; lengths at and beside the powers of two; 50 heads of 4096 positions run in clusters of four.  The sums are exact
# to about 1e-9 relative, so what is left of the parameters' error is their rounding to fp32 (2^-24 of up to 32) and an Adam step's
# response to its gradient's error, lr |dg| / |g| with |g| down to 1e-3 of the marginals: 1e-6.
@pytest.mark.parametrize("Hf,T,steps", [(2, 129, 4), (1, 256, 3), (2, 257, 3), (1, 512, 3), (2, 513, 3), (1, 1024, 3), (1, 1025, 3),
                                        (1, 2048, 2), (1, 2049, 2), (1, 4096, 2), (50, 4095, 2), (1, 4097, 2), (1, 8193, 1)])
def test_fit_transform_lengths(Hf, T, steps):
    base = si.mean_attention_maps(1, T, 60 + T)
    P, ea, er, pl = _oracle_stats(base)
    rep = lambda v: _dev(np.repeat(v, Hf, axis=0))
    a, r, z, loss, kl = _gpu_fit(_ctx(), rep(ea), rep(er), rep(pl), steps)
    for x in (a, r, z, loss, kl):
        assert np.array_equal(x, np.broadcast_to(x[:1], x.shape))
    wa, wr, wz = fo.fit_compact(ea[0], er[0], steps=steps)
    tol = 1e-6 + 2.0 ** -24 * np.abs(wr).max()
    assert np.max(np.abs(a[0] - wa)) < tol and np.max(np.abs(r[0] - wr)) < tol and np.max(np.abs(z[0] - wz)) < tol
    assert abs(loss[0] - fo.fit_objective(wa, wr, ea[0], er[0])) < 1e-9 * max(1.0, abs(loss[0]))


# Steps of 10 nats take heads out of the transforms' bounds behind the first one (steps of 3 nats do not here); what was done before
# must not be lost: the parameters after few steps against the oracle (the direct sums' bounds above), the normalisers at the
# returned parameters always.
@pytest.mark.parametrize("T,lr,steps", [(200, 3.0, 6), (300, 10.0, 3), (300, 10.0, 4), (300, 10.0, 7), (700, 10.0, 5), (1500, 10.0, 6),
                                        (2500, 10.0, 5), (2500, 10.0, 6)])
def test_fit_heads_handed_on(T, lr, steps):
    A = si.mean_attention_maps(2, T, 70 + T)
    P, ea, er, pl = _oracle_stats(A)
    ctx = _ctx()
    a, r, z, loss, kl = _gpu_fit(ctx, _dev(ea), _dev(er), _dev(pl), steps, lr=lr)
    at = ctx.saf_fit_handover(2)
    assert (at == (2 if lr == 10.0 else -1)).all(), at
    for h in range(2):
        want_z, _ = fo._logZ_and_P(a[h], r[h])
        assert np.max(np.abs(z[h] - want_z)) < 5e-4
        assert abs(loss[h] - fo.fit_objective(a[h], r[h], ea[h], er[h])) < 5e-4 * max(1.0, abs(loss[h]))
        wa, wr, wz = fo.fit_compact(ea[h], er[h], steps=steps, lr=lr)
        # a gradient that nearly cancels may take the other sign in one element: most elements, not all
        assert np.mean(np.abs(a[h] - wa) < 1e-2 * lr) > 0.97 and np.mean(np.abs(r[h] - wr) < 1e-2 * lr) > 0.97


# Largest errors in units in the last place: a correctly rounded result has 0.5; the exponential's argument reduction and sum add a
# quarter (0.76 over 2e7 arguments evaluated on a CPU with the same steps).  Ranges: normalisers and Adam's denominators, moments,
# parameters.
@pytest.mark.parametrize("which,lo,hi,ulps", [(0, 1e-30, 1e30, 0.51), (0, 1e-8, 1e150, 0.51), (1, 1e-199, 1e290, 0.51), (2, -690.0, 690.0, 0.8),
                                              (2, -1.0, 1.0, 0.8)])
def test_fit_math(which, lo, hi, ulps):
    rng = np.random.default_rng(which)
    n = 1 << 20
    x = rng.uniform(lo, hi, n) if which == 2 else np.exp(rng.uniform(np.log(lo), np.log(hi), n))
    x[:4] = [lo, hi, *((0.0, 0.5) if which == 2 else (1.0, 4.0))]
    xd = torch.from_numpy(x).cuda()
    y = torch.empty_like(xd)
    saf.saf_fit_math(0, which, xd, y)
    got = y.cpu().numpy()
    assert np.finfo(np.longdouble).nmant >= 63
    xl = x.astype(np.longdouble)
    want = 1.0 / xl if which == 0 else np.sqrt(xl) if which == 1 else np.exp(xl)
    err = np.abs(got.astype(np.longdouble) - want) / np.spacing(want.astype(np.float64))
    assert err.max() <= ulps, (err.max(), x[err.argmax()])


def test_fit_math_ends():
    y = torch.empty(2, dtype=torch.float64, device="cuda")
    saf.saf_fit_math(0, 1, torch.zeros(2, dtype=torch.float64, device="cuda"), y)
    assert ((0.0 <= y) & (y <= 1e-99)).all()
    saf.saf_fit_math(0, 2, torch.tensor([-1e9, 1e9], dtype=torch.float64, device="cuda"), y)
    assert 0.0 < y[0] < 1e-300 and 1e300 < y[1] < float("inf")
    for which in range(3):
        saf.saf_fit_math(0, which, torch.full((2,), float("nan"), dtype=torch.float64, device="cuda"), y)
        assert torch.isnan(y).all(), which
    with pytest.raises(saf.SafError):
        saf.saf_fit_math(0, 3, y, y)


# A tiny eta_rel(0) puts the first normaliser, Z(0) = A(0) R(0), and then the last key's marginal ever further below the norms of
# their factors: heads leave the transforms' bounds at the step named, by a normaliser (Z, in the middle of a step) or a marginal (M,
# at its end).  The steps are those of a double-precision model of the bounds, with a factor of 1.2 to spare at least.  Lengths
# for the direct kernel of 16 warps, of 12 (beyond 8192) and with unpadded vectors (beyond 12288).
@pytest.mark.parametrize("T,log_r0,at,steps", [(300, -8.5, 1, 4), (300, -7.6, 1, 4), (300, -7.15, 2, 4), (300, -6.8, 2, 4), (300, -6.1, 3, 4),
                                               (300, -5.3, 4, 5), (300, -4.4, 5, 5),
                                               (1000, -8.5, 1, 4), (1000, -7.4, 1, 4), (1000, -6.95, 2, 4), (1000, -6.2, 2, 4),
                                               (1000, -5.2, 3, 4), (2500, -8.5, 1, 3), (2500, -6.8, 2, 3), (2500, -6.0, 2, 2),
                                               (5000, -7.2, 1, 2), (5000, -6.0, 2, 2), (9000, -8.5, 1, 2), (9000, -6.2, 2, 2),
                                               (9000, -5.6, 2, 2), (12500, -7.0, 1, 2), (12500, -6.2, 2, 2), (12500, -5.6, 2, 2)])
def test_fit_goes_on_where_it_was_handed_on(T, log_r0, at, steps):
    lr, rng, d = 1.5, np.random.default_rng(1 + T), np.arange(T)
    ea = np.exp(0.5 * rng.standard_normal(T))
    er = (T - d) * (1.0 + d) ** -1.3 * np.exp(0.3 * rng.standard_normal(T))
    ea, er = ea * T / ea.sum(), er * T / er.sum()
    er[0], ea[0] = T * 10.0 ** log_r0, 0.5
    ctx = _ctx()
    a, r, z, loss, kl = _gpu_fit(ctx, _dev(ea[None]), _dev(er[None]), _dev(np.zeros(1)), steps, lr=lr)
    assert ctx.saf_fit_handover(1)[0] == at
    # An element moves by lr m / (sqrt(v) + 1e-8); an error of 2e-6 of its marginal in the gradients (direct sums of positive
    # fp32 terms) moves it by lr 2e-6 / |g / marginal| a step.  Elements whose gradient is below 1e-3 of the marginal at some step: excepted.
    x = np.concatenate(fo.fit_init(er))
    m, v, ratio = np.zeros(2 * T), np.zeros(2 * T), np.full(2 * T, np.inf)
    for t in range(1, steps + 1):
        g = np.concatenate(fo.fit_gradient(x[:T], x[T:], ea, er))
        target = np.concatenate([ea, er]) / T
        ratio = np.minimum(ratio, np.abs(g) / np.maximum(target, g + target))
        m, v = 0.9 * m + 0.1 * g, 0.999 * v + 0.001 * g * g
        x = x - lr * (m / (1 - 0.9 ** t)) / (np.sqrt(v / (1 - 0.999 ** t)) + 1e-8)
    clear = ratio > 1e-3
    assert clear.mean() > 0.97
    err = np.abs(np.concatenate([a[0], r[0]]) - x)[clear]
    assert err.max() <= steps * lr * 2e-3, (err.max(), np.sort(err)[-5:])
    want_z, _ = fo._logZ_and_P(a[0], r[0])
    assert np.max(np.abs(z[0] - want_z)) < 1e-4
    assert abs(loss[0] - fo.fit_objective(a[0], r[0], ea, er)) < 1e-4


def test_a_fit_for_which_only_the_direct_sums_have_room():
    """36000 heads of 300 positions: 605 MB of state for the direct sums, 1166 MB with the transforms' second copy."""
    Hf, T = 36000, 300
    P, ea, er, pl = _oracle_stats(si.mean_attention_maps(1, T, 3))
    ea_d, er_d = (_dev(x).expand(Hf, T).contiguous() for x in (ea, er))
    out = [torch.empty((Hf, T), device="cuda") for _ in range(3)]
    ctx = _ctx()
    torch.cuda.synchronize()
    torch.cuda.empty_cache()
    hold = torch.empty(torch.cuda.mem_get_info()[0] - (850 << 20), device="cuda", dtype=torch.uint8)
    ctx.saf_fit_compact(Hf, T, ea_d, er_d, None, 2, 0.05, *out, T, None, None)
    _status(ctx)
    assert (ctx.saf_fit_handover(Hf) == 0).all()
    s = torch.cuda.Stream()
    g = torch.cuda.CUDAGraph()
    with torch.cuda.graph(g, stream=s):                            # (recorded as warmed up)
        ctx.saf_fit_compact(Hf, T, ea_d, er_d, None, 2, 0.05, *out, T, None, None)
    for x in out:
        x.fill_(float("nan"))
    g.replay()
    _status(ctx)
    del hold
    torch.cuda.empty_cache()
    want = fo.fit_compact(ea[0], er[0], steps=2)
    for x, w in zip(out, want):
        assert np.abs(x[0].cpu().numpy() - w).max() < 2e-4 and torch.equal(x, x[:1].expand(Hf, T))


def test_no_handover_steps_of_a_fit_that_failed():
    """The fit before left its steps in a buffer that the failed call has given back."""
    T = 300
    P, ea, er, pl = _oracle_stats(si.mean_attention_maps(1, T, 3))
    ctx = _ctx()
    _gpu_fit(ctx, _dev(ea), _dev(er), _dev(pl), 2)
    assert (ctx.saf_fit_handover(1) == -1).all()
    Hf = 36000
    big = [torch.zeros((Hf, T), device="cuda", dtype=torch.float64) for _ in range(2)] + [torch.empty((Hf, T), device="cuda") for _ in range(3)]
    torch.cuda.synchronize()
    torch.cuda.empty_cache()
    hold = torch.empty(torch.cuda.mem_get_info()[0] - (300 << 20), device="cuda", dtype=torch.uint8)
    with pytest.raises(saf.SafError) as e:
        ctx.saf_fit_compact(Hf, T, big[0], big[1], None, 2, 0.05, *big[2:], T, None, None)
    assert e.value.code == saf.SAF_ERR_NOMEM
    for n in (1, Hf):
        with pytest.raises(saf.SafError) as e:
            ctx.saf_fit_handover(n)
        assert e.value.code == saf.SAF_ERR_INVALID_ARG
    del hold, big
    torch.cuda.empty_cache()
    assert np.isfinite(_gpu_fit(ctx, _dev(ea), _dev(er), _dev(pl), 2)[0]).all()
    assert (ctx.saf_fit_handover(1) == -1).all()


@pytest.mark.parametrize("T", [100, 300, 2500])
@pytest.mark.parametrize("which,value", [(0, float("nan")), (1, float("nan")), (0, float("inf")), (1, float("inf"))])
def test_a_target_that_is_not_finite_spoils_its_whole_head_and_no_other(T, which, value):
    """One NaN or infinite element of eta_abs (0) or eta_rel (1): after two steps it is in every normaliser and gradient, so
    that no caller installs a pattern from it by looking at one output alone."""
    A = si.mean_attention_maps(2, T, 80 + T)
    P, ea, er, pl = _oracle_stats(A)
    clean = _gpu_fit(_ctx(), _dev(ea), _dev(er), _dev(pl), 4)
    (ea, er)[which][0, 17] = value
    got = _gpu_fit(_ctx(), _dev(ea), _dev(er), _dev(pl), 4)
    for x, y in zip(got, clean):
        assert np.array_equal(x[1], y[1])
        assert not np.isfinite(x[0]).any()
