"""GPU tests at the edges of the 128-wide kernels' work items (one or two query blocks per forward item, full 128-query tiles
in the backward), of the normaliser kernel's chunks and of the calibration's mean pass."""
import numpy as np
import pytest
import torch

import paper_2609_34650_b200 as saf
import saf_inputs as si
from oracle import saf_oracle as orc

from gpu_util import Layer
from test_gpu_parity import _check_gqa_layer, _check_packed_layer, all_units, check_units, sampled_units

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("B,H,T,D,frozen", [
    # at most one block per SM: one query block per item, one CTA per SM
    (1, 4, 128, 128, (1,)),             # one block
    (1, 3, 129, 96, (0,)),              # two blocks
    (1, 4, 520, 128, (1,)),             # five blocks
    # one query block per item, two CTAs per SM
    (10, 16, 100, 128, (3,)),           # 160 one-block units
    (10, 9, 200, 96, (1, 4)),           # two blocks, 180 items
    (5, 10, 257, 128, (1, 4, 7)),       # three blocks, 150 items
    (16, 12, 300, 128, (2, 3)),         # the most three-block units that go there (576 blocks on 148 SMs)
    (12, 8, 512, 96, (0, 5)),           # four blocks: 192 two-block items would be a wave and a little
    (1, 32, 640, 128, (7,)),            # 160 blocks
    # two query blocks per item, one CTA per SM
    (4, 10, 520, 96, (0, 5, 9)),        # 200 blocks: pairs, the first block of an odd count alone
    (17, 12, 300, 128, (1, 4)),         # one more batch entry than above: a pair and a single block per unit
    (4, 10, 768, 128, (2, 3)),          # pairs of every length up to six tiles
])
def test_item_shapes_of_the_wide_forward(B, H, T, D, frozen):
    """Both kernels of head dimensions 96 and 128 on either side of the lines between them."""
    inp = si.generate(si.Workload("items", B, H, T, D, frozen, -0.05, seed=T + D))
    units = all_units(inp.wl)
    check_units(Layer(inp).run(), units if len(units) <= 50 else sampled_units(inp.wl, 24, seed=5))


@pytest.mark.parametrize("B,H,T", [(4, 13, 384), (4, 12, 640)])
def test_running_maximum_far_above_the_first_tile(B, H, T):
    """Scores that grow along the sequence: the rescaling of the accumulator between tiles, in the one-block kernel and in
    both blocks of a pair (240 blocks: more than the one-block items that are tried first, so they are paired)."""
    n_sms = torch.cuda.get_device_properties(0).multi_processor_count
    assert T == 384 or B * H * (T // 128) > 1.3 * n_sms
    inp = si.generate(si.Workload("grow", B, H, T, 128, (), -0.05, seed=9))
    f = np.exp2(np.arange(T) // 128).astype(np.float32)            # exact in bf16
    inp.k[...] = si.f32_to_bf16_bits(si.bf16_bits_to_f32(inp.k) * f[None, None, :, None])
    L = Layer(inp, backward=False)
    L.run(backward=False)
    q, k, v = (si.bf16_bits_to_f64(x) for x in (inp.q, inp.k, inp.v))
    want, _ = orc.hybrid_attn_fwd(q, k, v, inp.mask, inp.alpha, inp.rho)
    got = L.O.float().cpu().numpy().astype(np.float64)
    assert np.abs(got - want).max() <= 2e-2 and np.linalg.norm(got - want) <= 1e-2 * np.linalg.norm(want)


@pytest.mark.parametrize("D", [96, 128])
@pytest.mark.parametrize("B,H,T", [(16, 12, 300), (8, 8, 1200)])
def test_item_kinds_alternate_at_the_wide_head_dimensions(B, H, T, D):
    """Ordinary heads, frozen heads in the tensor-core form and frozen heads in the general form follow one another in the
    one-block items of the short forward (576 blocks), in the paired items of the long one (640 blocks) and in the
    backward's lists, several to a CTA."""
    frozen = (0, 2, 3, 5, 6)
    inp = si.generate(si.Workload("kinds", B, H, T, D, frozen, -0.05, seed=23 + D))
    for h in (2, 5):                                               # far outside the range of the tensor-core form
        inp.alpha[h] = (inp.alpha[h] + 25.0 * np.sin(0.37 * np.arange(T))).astype(np.float32)
    # (rows whose mass sits on a few keys: see the same test at head dimension 64)
    inp.do[...] = si.f32_to_bf16_bits(si.bf16_bits_to_f32(inp.do) / 16.0)
    L = Layer(inp).run()
    check_units(L, [(0, 0), (0, 2), (1, 1), (2, 5), (3, 3), (4, 4), (5, 6), (6, 7), (7, 2), (B - 1, H - 1)])


@pytest.mark.parametrize("D", [96, 128])
@pytest.mark.parametrize("B,H,T", [(4, 10, 520), (2, 6, 2050)])
def test_patterns_without_prepared_tables_in_paired_items(B, H, T, D):
    """Frozen heads whose normalisers come from the entry point without a context take the general form throughout: two table
    buffers per query block in turn, over odd and even tile counts and a last tile of a few rows; head 1 has keys switched
    off, head 2 leaves the range of the factorised exponential in some tiles."""
    inp = si.generate(si.Workload("general", B, H, T, D, tuple(range(H)), -0.05, seed=31 + D))
    inp.alpha[1, 40:60] = -1e30
    inp.alpha[2] = (inp.alpha[2] + 25.0 * np.sin(0.37 * np.arange(T))).astype(np.float32)
    L = Layer(inp, backward=False)
    saf.saf_pattern_logz_static(0, L.mask, L.alpha, L.rho, L.logZ)
    L.run(backward=False, prepare=False)
    check_units(L, [(0, 0), (0, 1), (1, 2), (B - 1, 3), (B - 1, H - 1)], backward=False)


@pytest.mark.parametrize("D,T", [(128, 1500), (96, 1337)])
def test_items_of_a_layer_with_and_without_prepared_tables(D, T):
    """Two of eight heads frozen, 176 and 192 blocks: without tables their items are longer than the ordinary heads' split blocks
    and come first; with tables the same context orders them anew."""
    inp = si.generate(si.Workload("forms", 2, 8, T, D, (1, 6), -0.05, seed=61 + D))
    L = Layer(inp, backward=False)
    units = [(0, 0), (0, 1), (1, 1), (0, 6), (1, 6), (1, 3), (1, 7)]
    saf.saf_pattern_logz_static(0, L.mask, L.alpha, L.rho, L.logZ)
    for prepare in (False, True):
        for t in (L.O, L.LSE):
            t.fill_(float("nan"))
        L.run(backward=False, prepare=prepare)
        check_units(L, units, backward=False)


def test_a_capture_takes_the_items_of_the_form_that_was_warmed_up():
    """A forward warmed up with prepared tables and recorded without them (another normaliser pointer): recording allocates
    nothing."""
    L = Layer(si.generate(si.Workload("capture", 2, 8, 1500, 128, (1, 6), -0.05, seed=67)), backward=False)
    c, other = L.ctx, torch.zeros_like(L.logZ)
    saf.saf_pattern_logz_static(0, L.mask, L.alpha, L.rho, other)
    call = lambda logZ: c.saf_hybrid_attn_fwd(L.prob, L.Q, L.K, L.V, L.mask, L.alpha, L.rho, logZ, L.O, L.LSE)
    s = torch.cuda.Stream()
    s.wait_stream(torch.cuda.current_stream())
    with torch.cuda.stream(s):
        c.saf_pattern_prepare(L.mask, L.alpha, L.rho, L.logZ)
        call(L.logZ)
        s.synchronize()
        g = torch.cuda.CUDAGraph()
        with torch.cuda.graph(g, stream=s):
            call(other)
        for t in (L.O, L.LSE):
            t.fill_(float("nan"))
        g.replay()
        s.synchronize()
    assert c.saf_last_device_status()[0] == saf.SAF_OK
    check_units(L, [(0, 0), (0, 1), (1, 1), (0, 6), (1, 7)], backward=False)


@pytest.mark.parametrize("T", [1, 31, 33, 255, 4096, 4097, 8200])
@pytest.mark.parametrize("spread", [1.0, 60.0])
def test_normalisers_at_chunk_edges(T, spread):
    """Rows around the 32-row blocks and the 4096-key chunks; `spread` 60 puts rows far below the common bound (a spike
    late in alpha), which are then taken relative to their own maximum."""
    rng = np.random.default_rng(T)
    alpha = rng.standard_normal((2, T)).astype(np.float32)
    alpha[:, -1] += 3.0 * spread
    rho = (-0.01 * np.arange(T) + 0.1 * rng.standard_normal((2, T))).astype(np.float32)
    mask = np.array([1, 1], dtype=np.uint8)
    a, r = torch.from_numpy(alpha).cuda(), torch.from_numpy(rho).cuda()
    z = torch.full((2, T), float("nan"), device="cuda")
    saf.Context(0).saf_pattern_prepare(mask, a, r, z)
    z = z.cpu().numpy().astype(np.float64)
    # ex2 and sums 2e-6; alpha + rho is rounded once in fp32, and so is the result
    big = np.abs(alpha).max() + np.abs(rho).max()
    for h in range(2):
        err = np.abs(z[h] - orc.pattern_logZ(alpha[h], rho[h], T))
        assert err.max() <= 5e-6 + 2.0 ** -23 * big, err.max()


def test_normalisers_of_ordinary_patterns_are_rounded_once():
    """Terms near the common bound: rms error at the rounding of the result (an fp32 unit of 2.4e-7 at |log Z| in [2, 4):
    6.9e-8) and of alpha + rho (under 5e-8 over the few terms that make up a row's sum)."""
    rng = np.random.default_rng(8)
    T, H = 2048, 4
    alpha = rng.standard_normal((H, T)).astype(np.float32)
    rho = (-0.05 * np.arange(T) + 0.1 * rng.standard_normal((H, T))).astype(np.float32)
    a, r, z = torch.from_numpy(alpha).cuda(), torch.from_numpy(rho).cuda(), torch.zeros(H, T, device="cuda")
    saf.Context(0).saf_pattern_prepare(np.ones(H, dtype=np.uint8), a, r, z)
    want = np.stack([orc.pattern_logZ(alpha[h], rho[h], T) for h in range(H)])
    assert np.abs(want).max() < 8.0
    assert np.sqrt(np.mean((z.cpu().numpy().astype(np.float64) - want) ** 2)) <= 1e-7


@pytest.mark.parametrize("T", [70, 4200])
def test_normalisers_ignore_what_a_row_does_not_see(T):
    """Keys and distances beyond a row's causal range may hold anything, in its own 32-row block too; minus infinity switches
    single keys off, the nearest ones among them."""
    rng = np.random.default_rng(T)
    alpha = rng.standard_normal((3, T)).astype(np.float32)
    rho = (-0.01 * np.arange(T) + 0.1 * rng.standard_normal((3, T))).astype(np.float32)
    alpha[0, T - 9] = np.inf
    alpha[1, T - 9] = np.nan
    alpha[2, T - 45:] = -np.inf
    a, r, z = torch.from_numpy(alpha).cuda(), torch.from_numpy(rho).cuda(), torch.zeros(3, T, device="cuda")
    saf.Context(0).saf_pattern_prepare(np.ones(3, dtype=np.uint8), a, r, z)
    z = z.cpu().numpy().astype(np.float64)
    assert not np.isfinite(z[:2, T - 9:]).any()
    for h, n in ((0, T - 9), (1, T - 9), (2, T)):
        finite = np.where(np.isneginf(alpha[h, :n]), -1e4, alpha[h, :n]).astype(np.float64)
        assert np.abs(z[h, :n] - orc.pattern_logZ(finite, rho[h, :n], n)).max() <= 5e-6


def test_rows_whose_largest_term_is_far_away_cost_two_more_passes():
    """A sink of 90 on key 0 and decaying rho: every row is taken again relative to its own maximum, by the whole block."""
    T, H = 4096, 3
    mask, ctx = np.ones(H, dtype=np.uint8), saf.Context(0)
    g = torch.Generator(device="cuda").manual_seed(1)
    alpha = torch.randn((H, T), generator=g, device="cuda")
    rho = -0.05 * torch.arange(T, device="cuda", dtype=torch.float32) + 0.1 * torch.randn((H, T), generator=g, device="cuda")
    sink = alpha.clone()
    sink[:, 0] += 90.0
    z = torch.zeros(H, T, device="cuda")
    us = {}
    for name, a in (("flat", alpha), ("sink", sink)) * 3:
        ctx.saf_pattern_prepare(mask, a, rho, z)
        ctx.saf_set_profiling(1)
        for _ in range(20):
            ctx.saf_pattern_prepare(mask, a, rho, z)
        torch.cuda.synchronize()
        ms, n = ctx.saf_get_kernel_time(saf.SAF_KERNEL_LOGZ)
        ctx.saf_set_profiling(0)
        us[name] = min(us.get(name, 1e9), ms * 1e3 / n)
    assert us["sink"] <= 4.0 * us["flat"], us            # (three passes instead of one)


@pytest.mark.parametrize("T", [4, 130, 1028, 1030])
def test_calibration_mean_pass(T):
    """Row lengths in whole 16-byte pieces and others; what lies above the diagonal stays as it was."""
    rng = np.random.default_rng(T)
    H, n = 3, 5
    total = np.tril(rng.random((H, T, T))).astype(np.float32)
    m = torch.from_numpy(total).cuda() + torch.triu(torch.full((H, T, T), 7.0, device="cuda"), diagonal=1)
    zero = torch.zeros(H, device="cuda", dtype=torch.float64)
    ctx = saf.Context(0)
    for _ in range(2):                                             # (the second call starts from the same workspace)
        mean, sq, pl = m.clone(), zero + 10.0 * T * T, zero + 1.0
        var, kl = zero.clone(), zero.clone()
        ctx.saf_calib_finalize(H, T, n, mean, sq, pl, var, kl)
        got = mean.cpu().numpy().astype(np.float64)
        want = total.astype(np.float64) / n
        low = np.tril(np.ones((T, T), dtype=bool))
        assert np.all(got[:, ~low] == 7.0)
        assert np.abs(got[:, low] - want[:, low]).max() <= 2.0 ** -23    # two fp32 roundings of values below one
        ref = (10.0 * T * T - n * (want ** 2).sum(axis=(1, 2))) / ((n - 1.0) * T * T)
        assert np.abs(var.cpu().numpy() - ref).max() <= 1e-6 * np.abs(ref).max()


# Query blocks whose even and odd key tiles run in two chains (units of at least four blocks; two and three beside them): odd and
# even counts, ragged ends, a row whose second chain sees the diagonal tile only; 12 units of 13 blocks and 32 of 9 mix them with
# pairs.  Shared K/V heads, packed Q/K, fp32 output.
@pytest.mark.parametrize("B,H,T,D,frozen,o_f32,g,packed", [
    (1, 4, 256, 128, (), False, 1, False), (1, 3, 257, 96, (1,), True, 1, False), (1, 4, 385, 128, (0,), False, 1, False),
    (1, 4, 512, 128, (), False, 1, False), (1, 3, 513, 96, (1,), True, 1, False), (2, 4, 1025, 128, (3,), True, 1, False),
    (1, 8, 700, 128, (2,), False, 4, False), (2, 5, 640, 128, (0, 3), False, 1, True), (1, 4, 900, 96, (1,), False, 2, False),
    (1, 12, 1664, 128, (3, 7), False, 1, False), (2, 16, 1152, 96, (0, 5), False, 1, False)])
def test_split_blocks_of_the_wide_forward(B, H, T, D, frozen, o_f32, g, packed):
    inp = si.generate(si.Workload("split", B, H, T, D, frozen, -0.05, seed=T + D, kv_group=g, packed_qk=packed))
    L, units = Layer(inp, o_f32=o_f32).run(), all_units(inp.wl)
    if g > 1:
        _check_gqa_layer(L, True)
    elif packed:
        _check_packed_layer(L, True)
    else:
        check_units(L, units if len(units) <= 12 else sampled_units(inp.wl, 12, seed=5))


@pytest.mark.parametrize("B,H,T", [(1, 8, 640), (8, 12, 640)])
def test_running_maximum_far_above_the_first_tile_in_split_and_paired_blocks(B, H, T):
    """Scores that grow along the sequence: the chains of a split block (40 blocks) rescale at different tiles and meet with
    references far apart; 480 blocks are paired (more than three per SM)."""
    n_sms = torch.cuda.get_device_properties(0).multi_processor_count
    assert B == 1 or B * H * (T // 128) > 3 * n_sms
    inp = si.generate(si.Workload("grow", B, H, T, 128, (), -0.05, seed=9))
    f = np.exp2(np.arange(T) // 128).astype(np.float32)            # exact in bf16
    inp.k[...] = si.f32_to_bf16_bits(si.bf16_bits_to_f32(inp.k) * f[None, None, :, None])
    L = Layer(inp, backward=False)
    L.run(backward=False)
    q, k, v = (si.bf16_bits_to_f64(x) for x in (inp.q, inp.k, inp.v))
    want, _ = orc.hybrid_attn_fwd(q, k, v, inp.mask, inp.alpha, inp.rho)
    got = L.O.float().cpu().numpy().astype(np.float64)
    assert np.abs(got - want).max() <= 2e-2 and np.linalg.norm(got - want) <= 1e-2 * np.linalg.norm(want)


@pytest.mark.parametrize("D,T,tiles", [(128, 640, (1,)), (96, 640, (1,)), (128, 1000, (1, 3, 5)), (128, 640, (2,))])
def test_a_chain_of_a_split_block_whose_scores_overflow(D, T, tiles):
    """Finite Q and K whose product is -inf throughout some key tiles: rows that see other keys as well are finite, wherever in
    its chain the tile comes (tile 1 is the first of chain 1, and all of it for the block whose own tile it is)."""
    inp = si.generate(si.Workload("overflow", 1, 4, T, D, (), -0.05, seed=T))
    big = si.f32_to_bf16_bits(np.float32([1e20, -1e20, 0.0]))
    inp.q[..., 0] = big[0]
    inp.k[..., 0] = big[2]
    for t in tiles:
        inp.k[:, :, 128 * t:128 * (t + 1), 0] = big[1]
    L = Layer(inp, backward=False)
    c = L.ctx
    c.saf_hybrid_attn_fwd(L.prob, L.Q, L.K, L.V, L.mask, None, None, None, L.O, L.LSE)
    torch.cuda.synchronize()
    assert c.saf_last_device_status()[0] == saf.SAF_OK
    q, k, v = (si.bf16_bits_to_f64(x) for x in (inp.q, inp.k, inp.v))
    want, lse = orc.hybrid_attn_fwd(q, k, v, inp.mask, inp.alpha, inp.rho)
    got = L.O.float().cpu().numpy().astype(np.float64)
    assert np.isfinite(got).all(), np.argwhere(~np.isfinite(got).all(axis=-1))[:3]
    assert np.abs(got - want).max() <= 2e-2 and np.linalg.norm(got - want) <= 1e-2 * np.linalg.norm(want)
    assert np.abs(L.LSE.cpu().numpy() - lse).max() <= 1e-4


def test_chunks_of_the_host_step_take_the_forms_of_the_whole_batch():
    """8 x 4 heads x 12 blocks = 384: some blocks split, some paired; chunks of one batch entry (48 blocks) alone would all be
    split."""
    wl = si.Workload("host-split", 8, 4, 1536, 128, (1,), -0.05, seed=34)
    inp = si.generate(wl)
    Dv = Layer(inp, backward=False)
    Dv.run(backward=False)
    Q, K, V = (t.cpu().contiguous().pin_memory() for t in (Dv.Q, Dv.K, Dv.V))
    alpha, rho = torch.from_numpy(inp.alpha), torch.from_numpy(inp.rho)
    O, LSE = torch.empty_like(Q), torch.empty(wl.B, wl.H, wl.T)
    prob = saf.make_problem(Q, wl.stored_len, k_like=K, v_like=V, o_like=O, H=wl.H)
    saf.Context(0).saf_hybrid_attn_step_host(prob, Q, K, V, None, inp.mask, alpha, rho, 1, O, LSE, None, None, None)
    assert torch.equal(O, Dv.O.cpu()) and torch.equal(LSE, Dv.LSE.cpu())
