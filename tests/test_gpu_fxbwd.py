"""The tensor-core adjoint kernels at the places where their blocks can go wrong, against the oracle: partial
and whole blocks, spline knots and stencil steps, orders, sampling steps, cotangents and strain whose range or
values send a block to the sample-by-sample form."""
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


def check(ctx, pair, N, p, src, g, gen=2, dt=DT, precision=lr.FP64, strain=None):
    """Strain gradients to 1e-12, the sky gradient to 1e-11 or its rounding scale 4 (T + 16) u sum |terms|."""
    t0h, hp, hc = synth.gb_input(src, T0, dt, N, p)
    if strain is not None:
        strain(hp, hc)
    plan = lr.Plan(ctx, p, N, dt, pair.gpu, t0=T0, generation=gen, precision=precision)
    got = [host(v) for v in plan.backward(dev(hp), dev(hc), t0h, sky(src), dev(g))]
    plan.check()
    rp, rc, rs, scale = oracle.backward(p, gen, dt, T0, N, pair.orc, pair.orc, hp, hc, t0h, src.lam, src.beta, src.psi, g,
                                        with_scale=True)
    for a, b in zip(got, (rp, rc)):
        assert np.linalg.norm(a - b) <= 1e-12 * np.linalg.norm(b)
    bound = np.maximum(1e-11 * np.abs(rs), 4 * (p + 17) * 2.0 ** -53 * scale)
    assert np.all(np.abs(got[2] - rs) <= bound), (got[2], rs, bound)


@pytest.mark.parametrize("precision", [lr.FP64, lr.MIXED])
@pytest.mark.parametrize("N", [1, 31, 477, 478, 479, 957, 20000])
def test_block_edges_and_steps(ctx, flex, N, precision):
    src = dataclasses.replace(synth.draw_sources(1, seed=N)[0], f=2e-3, beta=0.02)
    check(ctx, flex, N, 25, src, np.random.default_rng(N).normal(size=(3, N)), precision=precision)


@pytest.mark.parametrize("p", [1, 3, 9, 17, 31, 41])
@pytest.mark.parametrize("gen", [1, 2])
def test_orders(ctx, flex, p, gen):
    check(ctx, flex, 3000, p, synth.draw_sources(1, seed=p)[0], np.random.default_rng(p).normal(size=(3, 3000)), gen=gen)


@pytest.mark.parametrize("dt", [2.5, 5.0, 100.0])
def test_sampling_steps(ctx, dt):
    N = 2000
    pair = Pair(ctx, synth.orbit_flexing(T0 - 3e5, T0 + N * dt + 3e5))
    src = dataclasses.replace(synth.draw_sources(1, seed=9)[0], f=0.01 / dt)
    check(ctx, pair, N, 25, src, np.random.default_rng(2).normal(size=(3, N)), dt=dt)


@pytest.mark.parametrize("p", [11, 41])
def test_blocks_evaluated_sample_by_sample(ctx, flex, p):
    """One loud cotangent sample, one loud strain sample: their blocks exceed the fixed point's range."""
    N = 2500
    src = dataclasses.replace(synth.draw_sources(1, seed=7)[0], f=3e-3)
    g = np.random.default_rng(1).normal(size=(3, N))
    g[1, 700] *= 1e7

    def loud(hp, hc):
        hc[1900] *= 1e7

    check(ctx, flex, N, p, src, g, strain=loud)


def test_source_along_an_arm(ctx, flex):
    pos = synth.keplerian_flexing(np.array([1e4]))[:, :, 0]
    d = (pos[0] - pos[1]) / np.linalg.norm(pos[0] - pos[1])
    src = dataclasses.replace(synth.draw_sources(1, seed=4)[0], lam=float(np.arctan2(-d[1], -d[0]) + 5e-3),
                              beta=float(np.arcsin(-d[2])))
    check(ctx, flex, 1500, 25, src, np.random.default_rng(8).normal(size=(3, 1500)))


def test_nonfinite_cotangent_stays_local(ctx, flex):
    """A NaN in the cotangent reaches the strain samples within its reach and no other block's."""
    N, p = 6000, 11
    src = synth.draw_sources(1, seed=3)[0]
    t0h, hp, hc = synth.gb_input(src, T0, DT, N, p)
    g = np.random.default_rng(5).normal(size=(3, N))
    plan = lr.Plan(ctx, p, N, DT, flex.gpu, t0=T0)
    ref = host(plan.backward(dev(hp), dev(hc), t0h, sky(src), dev(g))[0])
    g[0, 3000] = np.nan
    got = host(plan.backward(dev(hp), dev(hc), t0h, sky(src), dev(g))[0])
    bad = ~np.isfinite(got)
    m = synth.input_margin_samples(DT, p)
    assert bad.any() and np.flatnonzero(bad).min() >= 3000 and np.flatnonzero(bad).max() <= 3000 + 2 * m
    assert np.linalg.norm((got - ref)[~bad]) <= 1e-13 * np.linalg.norm(ref)


@pytest.mark.parametrize("N", [479, 3000])
def test_cotangent_scales(ctx, flex, N):
    """Cotangents times s, 1 <= s < 2, so that the blocks' largest values pass through all significands (the top
    byte's range ends at 127.5 / 128 of a power of two): the gradient is linear, s times the oracle's."""
    p, src = 11, synth.draw_sources(1, seed=12)[0]
    t0h, hp, hc = synth.gb_input(src, T0, DT, N, p)
    g = np.random.default_rng(N).normal(size=(3, N))
    rp, rc, rs, scale = oracle.backward(p, 2, DT, T0, N, flex.orc, flex.orc, hp, hc, t0h, src.lam, src.beta, src.psi, g,
                                        with_scale=True)
    bound = np.maximum(1e-11 * np.abs(rs), 4 * (p + 17) * 2.0 ** -53 * scale)
    plan = lr.Plan(ctx, p, N, DT, flex.gpu, t0=T0)
    for s in 1.0 + np.arange(128) / 128:
        got = [host(v) / s for v in plan.backward(dev(hp), dev(hc), t0h, sky(src), dev(g * s))]
        for a, b in zip(got, (rp, rc)):
            assert np.linalg.norm(a - b) <= 1e-12 * np.linalg.norm(b)
        assert np.all(np.abs(got[2] - rs) <= bound), (s, got[2], rs, bound)
    plan.check()
