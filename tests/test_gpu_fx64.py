"""The tensor-core FP64 kernels at the places where their blocks can go wrong, against the oracle and
against the sample-by-sample kernels (reached with a tile that has no part of 128 to 478 outputs)."""
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
from _gpu import DT, T0, Pair, assert_close, dev, host, run_case, sky  # noqa: E402

BY_SAMPLE = 509   # a prime tile above the largest block


@pytest.fixture(scope="module")
def ctx():
    return lr.Context(0)


@pytest.fixture(scope="module")
def flex(ctx):
    return Pair(ctx, synth.orbit_flexing(-2e6, 2e6))


@pytest.mark.parametrize("kind", ["response", "project", "tdi"])
@pytest.mark.parametrize("N", [1, 31, 477, 478, 479, 957, 20000])
def test_block_edges_and_steps(ctx, flex, kind, N):
    """Partial and whole blocks; 20 000 outputs hold knots and stencil steps of every read.  A source
    near the ecliptic drifts fastest."""
    src = dataclasses.replace(synth.draw_sources(1, seed=N)[0], f=2e-3, beta=0.02)
    run_case(ctx, src, N, 25, flex, kind=kind)


@pytest.mark.parametrize("p", [1, 3, 9, 17, 31, 41])
@pytest.mark.parametrize("gen", [1, 2])
def test_orders(ctx, flex, p, gen):
    run_case(ctx, synth.draw_sources(1, seed=p)[0], 3000, p, flex, gen=gen)


@pytest.mark.parametrize("dt", [2.5, 5.0, 15.0, 100.0])
def test_sampling_steps(ctx, dt):
    """Chained delays from under one to 24 samples: one merged stencil per link in each case."""
    N, p = 3000, 25
    orb = synth.orbit_flexing(T0 - 3e5, T0 + N * dt + 3e5)
    pair = Pair(ctx, orb)
    src = dataclasses.replace(synth.draw_sources(1, seed=9)[0], f=0.01 / dt)
    t0h, hp, hc = synth.gb_input(src, T0, dt, N, p)
    plan = lr.Plan(ctx, p, N, dt, pair.gpu, t0=T0)
    got = host(plan.response(dev(hp), dev(hc), t0h, sky(src)))
    plan.check()
    args = (p, 2, dt, T0, N, pair.orc, pair.orc, hp, hc, t0h, src.lam, src.beta, src.psi)
    assert_close(got, oracle.response(*args), oracle.response(*args, absval=True), p + 1, 1e-12)


def test_source_along_an_arm(ctx, flex):
    """Near an arm direction the patterns turn within a block: the block's expansion does not apply."""
    t = 10000.0
    pos = synth.keplerian_flexing(np.array([t]))[:, :, 0]
    d = (pos[0] - pos[1]) / np.linalg.norm(pos[0] - pos[1])
    for off in (1e-3, 5e-3, 2e-2):
        src = dataclasses.replace(synth.draw_sources(1, seed=4)[0], lam=float(np.arctan2(-d[1], -d[0]) + off),
                                  beta=float(np.arcsin(-d[2])))
        run_case(ctx, src, 2500, 25, flex)


@pytest.mark.parametrize("p", [11, 41])
def test_wide_range_and_nonfinite_blocks_match_the_sample_kernels(ctx, flex, p):
    """A loud sample, a NaN and an infinity: the blocks that read them are evaluated sample by sample (same
    arithmetic as the sample kernels), with the same outputs undefined; the others agree to rounding."""
    N = 6000
    src = dataclasses.replace(synth.draw_sources(1, seed=7)[0], f=3e-3)
    t0h, hp, hc = synth.gb_input(src, T0, DT, N, p)
    hp[2000] *= 1e9
    hp[3500] = np.nan
    hc[5000] = np.inf
    out = []
    for tile in (0, BY_SAMPLE):
        plan = lr.Plan(ctx, p, N, DT, flex.gpu, t0=T0, tile=tile)
        out.append(host(plan.response(dev(hp), dev(hc), t0h, sky(src))))
        with pytest.raises(lr.LRError):
            plan.check()
    a, b = out
    assert np.array_equal(np.isfinite(a), np.isfinite(b)) and not np.isfinite(b).all()
    ok = np.isfinite(b)
    quiet = ok.copy()
    quiet[:, 1700:2300] = False   # outputs that read the loud sample
    assert np.linalg.norm((a - b)[ok]) <= 1e-12 * np.linalg.norm(b[ok])
    assert np.linalg.norm((a - b)[quiet]) <= 1e-12 * np.linalg.norm(b[quiet])


def test_zero_strain_gives_zero(ctx, flex):
    plan = lr.Plan(ctx, 25, 2000, DT, flex.gpu, t0=T0)
    z = torch.zeros(2200, dtype=torch.float64, device="cuda:0")
    assert not plan.response(z, z, -100 * DT, (0.3, 0.2, 0.1)).any()
    plan.check()


@pytest.mark.parametrize("past", [0.0, 3e5])
def test_outputs_past_the_knots(ctx, past):
    """The orbit's end pieces are continued outside its knots, and the delayed reads with them: blocks before the
    first knot, across the last one and behind it."""
    N, p = 3000, 25
    tk = synth.knot_grid(0.0, 5e5, pad=2)
    pair = Pair(ctx, synth.Orbit(tk, synth.keplerian_flexing(tk), None))
    src = dataclasses.replace(synth.draw_sources(1, seed=4)[0], f=3e-3)
    for t0 in (tk[-1] - 15000.0 + past, tk[0] - 15000.0 - past):
        t0h, hp, hc = synth.gb_input(src, t0, DT, N, p)
        plan = lr.Plan(ctx, p, N, DT, pair.gpu, t0=t0)
        got = host(plan.response(dev(hp), dev(hc), t0h, sky(src)))
        plan.check()
        args = (p, 2, DT, t0, N, pair.orc, pair.orc, hp, hc, t0h, src.lam, src.beta, src.psi)
        assert_close(got, oracle.response(*args), oracle.response(*args, absval=True), p + 1, 1e-12)


@pytest.mark.parametrize("early", [1, 20011, 1000037])
def test_strain_that_begins_long_before_the_outputs(ctx, flex, early):
    """The reads' fractions do not depend on how far before the outputs the strain begins: the same response, bit
    for bit, and the same gradients."""
    N, p = 3000, 25
    src = dataclasses.replace(synth.draw_sources(1, seed=4)[0], f=3e-3)
    t0h, hp, hc = synth.gb_input(src, T0, DT, N, p)
    plan = lr.Plan(ctx, p, N, DT, flex.gpu, t0=T0)
    g = dev(np.random.default_rng(3).normal(size=(3, N)))
    z = np.zeros(early)
    out = []
    for a, b, t in ((hp, hc, t0h), (np.r_[z, hp], np.r_[z, hc], t0h - early * DT)):
        out.append((plan.response(dev(a), dev(b), t, sky(src)), plan.backward(dev(a), dev(b), t, sky(src), g)))
    plan.check()
    (x0, g0), (x1, g1) = out
    assert torch.equal(x0, x1) and torch.equal(g0[2], g1[2])
    for a, b in zip(g0[:2], g1[:2]):
        assert float(torch.linalg.norm(b[early:] - a)) <= 1e-13 * float(torch.linalg.norm(a))


@pytest.mark.skipif(not oracle.quad_available(), reason="no binary128 libm in this toolchain")
@pytest.mark.parametrize("k", [0, 2, 3, 4, 8, 11])
@pytest.mark.parametrize("f", [1e-4, 1e-3, 1e-2])
def test_quiet_outputs_beside_a_loud_stretch(ctx, f, k):
    """A stretch 2^k above the rest of its block: the outputs that do not read it are as close to binary128 as the
    sample kernels' (a quarter more allows for chance), whether the block's fixed point takes them or not."""
    N, p = 700, 11
    orb = synth.orbit_flexing(T0 - 3e5, T0 + N * DT + 3e5)
    pair = Pair(ctx, orb)
    src = dataclasses.replace(synth.draw_sources(1, seed=4)[0], f=f)
    t0h, hp, hc = synth.gb_input(src, T0, DT, N, p)
    m = (len(hp) - N) // 2
    loud = np.zeros(len(hp))
    loud[m + 300:m + 380] = 1.0
    hp, hc = (1.0 + (2.0 ** k - 1.0) * loud) * hp, (1.0 + (2.0 ** k - 1.0) * loud) * hc
    quiet = oracle.response(p, 2, DT, T0, N, pair.orc, pair.orc, loud, loud, t0h, *sky(src), absval=True).max(0) == 0.0
    quiet[492:] = False   # the block of the loud stretch
    assert 150 < quiet.sum() < 400
    exact = oracle.response_quad(p, 2, DT, T0, N, orb.t_knots, orb.pos, orb.delays, hp, hc, t0h, *sky(src))
    err = []
    for tile in (0, BY_SAMPLE):
        plan = lr.Plan(ctx, p, N, DT, pair.gpu, t0=T0, tile=tile)
        err.append(np.linalg.norm((host(plan.response(dev(hp), dev(hc), t0h, sky(src))) - exact)[:, quiet]))
        plan.check()
    assert err[0] <= max(1.25 * err[1], 1e-14 * np.linalg.norm(exact[:, quiet])), err


@pytest.mark.parametrize("k", [0, 4, 8, 11])
def test_quiet_channel_beside_loud_links(ctx, flex, k):
    """X does not read the links between spacecraft 2 and 3: however loud they are, its distance from the oracle is
    that of the sample kernels' to a factor of 4 (two bits of the block's fixed point, and the oracle's own error)."""
    N, p = 1434, 11
    src = dataclasses.replace(synth.draw_sources(1, seed=4)[0], f=1e-3)
    t0h, hp, hc = synth.gb_input(src, T0, DT, N, p)
    y = oracle.project(p, DT, T0, N, flex.orc, hp, hc, t0h, *sky(src))
    ref = oracle.tdi(p, 2, DT, T0, N, flex.orc, y, 0)[0]
    y[[1, 4]] *= 2.0 ** k
    err = []
    for tile in (0, BY_SAMPLE):
        plan = lr.Plan(ctx, p, N, DT, flex.gpu, t0=T0, tile=tile)
        err.append(np.linalg.norm(host(plan.tdi(dev(y)))[0] - ref))
        plan.check()
    assert err[0] <= 4.0 * err[1], err


@pytest.mark.parametrize("spacing,pieces", [(1500.0, 60), (6000.0, 4100)])
def test_close_and_very_many_knots(ctx, spacing, pieces):
    """Blocks over three and four spline pieces, which the stencil table does not serve, and an orbit of more pieces
    than a table is made for."""
    N, p = 3000, 25
    tk = -2e4 + spacing * np.arange(pieces + 1)
    pair = Pair(ctx, synth.Orbit(tk, synth.keplerian_flexing(tk), None))
    src = dataclasses.replace(synth.draw_sources(1, seed=4)[0], f=3e-3)
    for kind in ("response", "tdi"):
        run_case(ctx, src, N, p, pair, kind=kind)
