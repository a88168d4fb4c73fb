"""The tensor-core adjoint kernels where their blocks, windows and expansions end: beyond the orbit's knots, on
fast orbits, along an arm, against the oracle."""
import dataclasses

import numpy as np
import pytest

pytestmark = pytest.mark.gpu

torch = pytest.importorskip("torch")
if not torch.cuda.is_available():
    pytest.skip("needs a CUDA GPU", allow_module_level=True)

import oracle  # noqa: E402
import paper_2204_06633_gb300 as lr  # noqa: E402
import synth  # noqa: E402
from _gpu import DT, T0, Pair, dev, host, sky  # noqa: E402


@pytest.fixture(scope="module")
def ctx():
    return lr.Context(0)


@pytest.fixture(scope="module")
def flex(ctx):
    return Pair(ctx, synth.orbit_flexing(-2e6, 2e6))


def check(ctx, pair, N, p, src, g, t0=T0, dt=DT, precision=lr.FP64, tile=0):
    """Strain gradients to 1e-12, the sky gradient to 1e-11 or its rounding scale 4 (T + 16) u sum |terms|."""
    t0h, hp, hc = synth.gb_input(src, t0, dt, N, p)
    plan = lr.Plan(ctx, p, N, dt, pair.gpu, t0=t0, precision=precision, tile=tile)
    got = [host(v) for v in plan.backward(dev(hp), dev(hc), t0h, sky(src), dev(g))]
    plan.check()
    rp, rc, rs, scale = oracle.backward(p, 2, dt, t0, N, pair.orc, pair.orc, hp, hc, t0h, src.lam, src.beta, src.psi, g,
                                        with_scale=True)
    for a, b in zip(got, (rp, rc)):
        assert np.linalg.norm(a - b) <= 1e-12 * np.linalg.norm(b)
    bound = np.maximum(1e-11 * np.abs(rs), 4 * (p + 17) * 2.0 ** -53 * scale)
    assert np.all(np.abs(got[2] - rs) <= bound), (got[2], rs, bound)


@pytest.mark.parametrize("past", [0.0, 3e5])
def test_outputs_past_the_knots(ctx, past):
    """Cotangents on outputs across the orbit's last knot and behind it, where its end piece is continued."""
    N, p = 1500, 25
    tk = synth.knot_grid(0.0, 5e5, pad=2)
    pair = Pair(ctx, synth.Orbit(tk, synth.keplerian_flexing(tk), None))
    src = dataclasses.replace(synth.draw_sources(1, seed=4)[0], f=3e-3)
    check(ctx, pair, N, p, src, np.random.default_rng(6).normal(size=(3, N)), t0=tk[-1] - 7000.0 + past)


@pytest.mark.parametrize("speed,spacing,precision", [(2.0, 5e4, lr.FP64), (4.0, 25e3, lr.FP64), (20.0, 1e3, lr.FP64),
                                                     (60.0, 1e3, lr.FP64), (2.0, 5e4, lr.MIXED)])
def test_fast_orbits(ctx, speed, spacing, precision):
    """The orbit run through faster: its reads drift by up to 1.5 samples over half a block of 512."""
    N, p = 2500, 25
    tk = synth.knot_grid(-1e5, N * DT + 1e5, spacing=spacing)
    pair = Pair(ctx, synth.Orbit(tk, synth.keplerian_flexing(tk * speed), None))
    src = dataclasses.replace(synth.draw_sources(1, seed=4)[0], f=3e-3, beta=0.02)
    check(ctx, pair, N, p, src, np.random.default_rng(8).normal(size=(3, N)), precision=precision)


def test_close_knots(ctx):
    """More spline pieces in a block than it has segments."""
    N, p = 1500, 25
    tk = synth.knot_grid(-2e4, N * DT + 2e4, spacing=500.0)
    pair = Pair(ctx, synth.Orbit(tk, synth.keplerian_flexing(tk), None))
    src = dataclasses.replace(synth.draw_sources(1, seed=4)[0], f=3e-3)
    check(ctx, pair, N, p, src, np.random.default_rng(8).normal(size=(3, N)))


@pytest.mark.skipif(not oracle.quad_available(), reason="no binary128 libm in this toolchain")
@pytest.mark.parametrize("off", [3e-2, 1e-2, 5e-3, 1e-3, 2e-4, 5e-5])
def test_sky_gradient_beside_an_arm(ctx, flex, off):
    """One block, the closest approach to an arm in its middle: the patterns turn within it, the faster the nearer
    the source is.  Against binary128; 1 - k.n has few significant bits there, so the FP64 oracle is off by up to
    3e-8 itself, and the bound is 16 times its error (as many bits lost, in other operations) where that is more
    than 1e-11 (1e-12 for the strain gradients)."""
    N, p, mid = 492, 11, 246
    pos = synth.keplerian_flexing(np.array([mid * DT]))[:, :, 0]
    d = (pos[0] - pos[1]) / np.linalg.norm(pos[0] - pos[1])
    src = dataclasses.replace(synth.draw_sources(1, seed=4)[0], f=1e-2, lam=float(np.arctan2(-d[1], -d[0]) + off),
                              beta=float(np.arcsin(-d[2])))
    t0h, hp, hc = synth.gb_input(src, T0, DT, N, p)
    g = np.random.default_rng(8).normal(size=(3, N))
    g[:, :mid - 180] = g[:, mid + 180:] = 0.0
    orb, oracle_args = flex.orb, (hp, hc, t0h, *sky(src), g)
    exact = oracle.backward_quad(p, 2, DT, T0, N, orb.t_knots, orb.pos, orb.delays, *oracle_args)
    r64 = oracle.backward(p, 2, DT, T0, N, flex.orc, flex.orc, *oracle_args)
    for precision in (lr.FP64, lr.MIXED):
        plan = lr.Plan(ctx, p, N, DT, flex.gpu, t0=T0, precision=precision)
        got = [host(v) for v in plan.backward(dev(hp), dev(hc), t0h, sky(src), dev(g))]
        plan.check()
        for a, b, c, rel in zip(got, exact, r64, (1e-12, 1e-12, 1e-11)):
            err, own = np.linalg.norm(a - b), np.linalg.norm(c - b)
            assert err <= max(rel * np.linalg.norm(b), 16 * own), (err / np.linalg.norm(b), own / np.linalg.norm(b))



@pytest.mark.parametrize("tile", [1, 16, 127])
def test_small_tiles(ctx, flex, tile):
    """The adjoint's blocks hold as many of a small tile's as fit.  Three times the default tile's time allows for
    smaller blocks, another number of waves and the spread of timings (in blocks of 16 they took ten times as long)."""
    N, p = 60000, 25
    src = dataclasses.replace(synth.draw_sources(1, seed=4)[0], f=3e-3)
    g = np.random.default_rng(8).normal(size=(3, 3000))
    check(ctx, flex, 3000, p, src, g, tile=tile)
    t0h, hp, hc = (torch.as_tensor(v, device="cuda:0") if isinstance(v, np.ndarray) else v
                   for v in synth.gb_input(src, T0, DT, N, p))
    g, ms = torch.randn(3, N, dtype=torch.float64, device="cuda:0"), {}
    for t in (0, tile):
        plan = lr.Plan(ctx, p, N, DT, flex.gpu, t0=T0, tile=t)
        plan.backward(hp, hc, t0h, sky(src), g)
        a, b = torch.cuda.Event(enable_timing=True), torch.cuda.Event(enable_timing=True)
        a.record()
        for _ in range(10):
            plan.backward(hp, hc, t0h, sky(src), g)
        b.record()
        b.synchronize()
        ms[t] = a.elapsed_time(b)
    assert ms[tile] <= 3.0 * ms[0], ms


@pytest.mark.skipif(not oracle.quad_available(), reason="no binary128 libm in this toolchain")
@pytest.mark.parametrize("k", [0, 5, 8, 11])
def test_quiet_gradients_beside_a_loud_stretch(ctx, flex, k):
    """A stretch of the cotangent 2^k above the rest: the strain gradients that it does not reach are within twice
    the FP64 oracle's own distance from binary128, those of a mixed plan within 1e-12."""
    N, p = 700, 11
    src = dataclasses.replace(synth.draw_sources(1, seed=4)[0], f=1e-3)
    t0h, hp, hc = synth.gb_input(src, T0, DT, N, p)
    g = np.random.default_rng(2).normal(size=(3, N))
    loud = np.zeros((3, N))
    loud[:, 300:380] = 1.0
    args = (hp, hc, t0h, *sky(src))
    quiet = oracle.backward(p, 2, DT, T0, N, flex.orc, flex.orc, *args, loud)[0] == 0.0
    m = (len(hp) - N) // 2
    quiet[:m] = quiet[m + 492:] = False   # the block of the loud stretch
    assert 150 < quiet.sum() < 450
    g *= 1.0 + (2.0 ** k - 1.0) * loud
    exact = oracle.backward_quad(p, 2, DT, T0, N, flex.orb.t_knots, flex.orb.pos, flex.orb.delays, *args, g)
    r64 = oracle.backward(p, 2, DT, T0, N, flex.orc, flex.orc, *args, g)
    plan = lr.Plan(ctx, p, N, DT, flex.gpu, t0=T0)
    got = [host(v) for v in plan.backward(dev(hp), dev(hc), t0h, sky(src), dev(g))]
    plan.check()
    mixed = lr.Plan(ctx, p, N, DT, flex.gpu, t0=T0, precision=lr.MIXED)
    got_mixed = [host(v) for v in mixed.backward(dev(hp), dev(hc), t0h, sky(src), dev(g))]
    mixed.check()
    for a, b, c, d in zip(got[:2], exact, r64, got_mixed):
        assert np.linalg.norm((a - b)[quiet]) <= 2.0 * np.linalg.norm((c - b)[quiet])
        assert np.linalg.norm((d - b)[quiet]) <= 1e-12 * np.linalg.norm(b[quiet])


@pytest.mark.parametrize("p,N,gen", [(1, 700, 2), (3, 31, 2), (11, 492, 1), (25, 478, 2), (25, 1434, 1), (41, 2000, 2)])
def test_blocks_evaluated_sample_by_sample(ctx, flex, p, N, gen):
    """One loud cotangent sample in each block, in the first, a middle and the last output of the span."""
    src = dataclasses.replace(synth.draw_sources(1, seed=7)[0], f=3e-3)
    g = np.random.default_rng(N).normal(size=(3, N))
    g[0, 0] = g[1, N // 2] = g[2, -1] = 1e5
    t0h, hp, hc = synth.gb_input(src, T0, DT, N, p)
    plan = lr.Plan(ctx, p, N, DT, flex.gpu, t0=T0, generation=gen)
    got = [host(v) for v in plan.backward(dev(hp), dev(hc), t0h, sky(src), dev(g))]
    plan.check()
    rp, rc, rs, scale = oracle.backward(p, gen, DT, T0, N, flex.orc, flex.orc, hp, hc, t0h, src.lam, src.beta, src.psi, g,
                                        with_scale=True)
    for a, b in zip(got, (rp, rc)):
        assert np.linalg.norm(a - b) <= 1e-12 * np.linalg.norm(b)
    assert np.all(np.abs(got[2] - rs) <= np.maximum(1e-11 * np.abs(rs), 4 * (p + 17) * 2.0 ** -53 * scale))


@pytest.mark.parametrize("precision", [lr.FP64, lr.MIXED])
def test_positions_beyond_every_window(ctx, flex, precision):
    """Outputs 10^11 s past the knots, where the continued end pieces put the reads 10^13 samples away: recorded as
    reads outside the plan's bounds, and the next call is as ever."""
    N, p = 700, 11
    src = synth.draw_sources(1, seed=4)[0]
    t0h, hp, hc = synth.gb_input(src, T0, DT, N, p)
    g = np.random.default_rng(1).normal(size=(3, N))
    plan = lr.Plan(ctx, p, N, DT, flex.gpu, t0=T0 + 1e11, precision=precision)
    calls = [lambda: plan.backward(dev(hp), dev(hc), t0h + 1e11, sky(src), dev(g))]
    if precision == lr.FP64:   # of a mixed plan only the adjoint is on these kernels
        calls.append(lambda: plan.response(dev(hp), dev(hc), t0h + 1e11, sky(src)))
    for call in calls:
        call()
        with pytest.raises(lr.LRError) as e:
            plan.check()
        assert e.value.status == 8   # LR_ERR_DEVICE
    check(ctx, flex, N, p, src, g, precision=precision)


@pytest.mark.parametrize("spacing,pieces", [(1500.0, 60), (6000.0, 4100)])
def test_knots_off_the_stencil_table(ctx, spacing, pieces):
    """Blocks over three and four spline pieces; an orbit of more pieces than a stencil table is made for, whose
    adjoint stays on the sample kernels."""
    N, p = 1500, 25
    tk = -2e4 + spacing * np.arange(pieces + 1)
    pair = Pair(ctx, synth.Orbit(tk, synth.keplerian_flexing(tk), None))
    src = dataclasses.replace(synth.draw_sources(1, seed=4)[0], f=3e-3)
    check(ctx, pair, N, p, src, np.random.default_rng(8).normal(size=(3, N)))
