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
