"""Which kernel family a plan runs on as its tile, sampling step and orbit vary: plans at the edges of the
tensor-core kernels' range give the oracle's results, keep what the caller asked for and launch with the tables
that their kernels read."""
import dataclasses
import os
import threading

import numpy as np
import pytest

pytestmark = pytest.mark.gpu

torch = pytest.importorskip("torch")
if not torch.cuda.is_available():
    pytest.skip("needs a CUDA GPU", allow_module_level=True)

import oracle  # noqa: E402
import paper_2204_06633_gb300 as lr  # noqa: E402
import synth  # noqa: E402
from _gpu import DT, T0, Pair, assert_close, dev, host, sky  # noqa: E402


@pytest.fixture(scope="module")
def ctx():
    return lr.Context(0)


@pytest.fixture(scope="module")
def flex(ctx):
    return Pair(ctx, synth.orbit_flexing(-2e6, 2e6))


def batch_args(lens, p, dt=DT, seed=3):
    """Device arguments of a ragged batch and, per source, (source, t0h, hp, hc)."""
    srcs = [dataclasses.replace(s, f=0.02 / dt) for s in synth.draw_sources(len(lens), seed=seed)]
    inp = [synth.gb_input(s, T0, dt, n, p) for s, n in zip(srcs, lens)]
    off = lambda n: torch.tensor(np.concatenate([[0], np.cumsum(n)]), dtype=torch.int64, device="cuda:0")  # noqa: E731
    args = [off([len(i[1]) for i in inp]), off(lens), dev([i[0] for i in inp]), dev([sky(s) for s in srcs]),
            dev(np.concatenate([i[1] for i in inp])), dev(np.concatenate([i[2] for i in inp]))]
    return args, [(s, *i) for s, i in zip(srcs, inp)]


def check_batch(xyz, pair, lens, per, p, dt=DT):
    at = 0
    for n, (s, t0h, hp, hc) in zip(lens, per):
        a = (p, 2, dt, T0, n, pair.orc, pair.orc, hp, hc, t0h, *sky(s))
        assert_close(host(xyz)[3 * at:3 * (at + n)].reshape(3, n), oracle.response(*a), oracle.response(*a, absval=True),
                     p + 1, 1e-12)
        at += n


@pytest.mark.parametrize("tile", [509, 1018, 512])
def test_batch_autotune_of_a_plan_off_the_tensor_cores(ctx, flex, tile, tmp_path):
    """No block of 128 to 478 outputs divides the first two tiles, so the plan starts on the sample-by-sample
    kernels, which form the sky frames themselves; the tuner's candidates run on the kernels that read them."""
    os.environ["LR_AUTOTUNE_CACHE"] = str(tmp_path / "tune.txt")
    lens, p = [3000, 700, 1], 25
    args, per = batch_args(lens, p)
    plan = lr.Plan(ctx, p, 1, DT, flex.gpu, t0=T0, tile=tile)
    assert plan.autotune_batch(lens, use_cache=False) == plan.tile
    xyz = plan.response_batched(*args)
    plan.check()
    check_batch(xyz, flex, lens, per, p)


@pytest.mark.parametrize("tile", [1, 64, 127, 128])
@pytest.mark.parametrize("p,dt", [(25, 1.0), (41, 4.0)])
def test_small_tiles_where_the_stencils_do_not_fit(ctx, p, dt, tile):
    """Sampling steps so short that a merged stencil passes 64 taps, with a small tile asked for: the plan keeps
    the sample-by-sample kernels and its tile, one source and batched."""
    lens = [700, 1, 130]
    pair = Pair(ctx, synth.orbit_flexing(T0 - 3e5, T0 + 1000 * dt + 3e5))
    args, per = batch_args(lens, p, dt)
    s, t0h, hp, hc = per[0]
    plan = lr.Plan(ctx, p, lens[0], dt, pair.gpu, t0=T0, tile=tile)
    assert plan.tile == tile
    one = plan.response(dev(hp), dev(hc), t0h, sky(s))
    xyz = plan.response_batched(*args)
    plan.check()
    check_batch(one, pair, lens[:1], per[:1], p, dt)
    check_batch(xyz, pair, lens, per, p, dt)


def test_failed_tuning_keeps_the_tile(ctx, flex):
    """A tile that the tensor-core kernels work in equal parts (512 in parts of 256) is still the plan's tile after
    a tuning that ran out of memory."""
    plan = lr.Plan(ctx, 25, 4096, DT, flex.gpu, t0=T0, tile=512)
    for tune in (lambda: plan.autotune(4096, use_cache=False), lambda: plan.autotune_batch([4096, 300], use_cache=False)):
        lr.library().lr_debug_fail_allocations(0)
        try:
            with pytest.raises(lr.LRError):
                tune()
        finally:
            lr.library().lr_debug_fail_allocations(-1)
        assert plan.tile == 512


def test_first_call_while_another_thread_captures(ctx, flex):
    """A plan's first call looks whether its stencil table is done; made while another thread captures a graph in
    the strictest mode, it runs and leaves the capture whole."""
    N, p = 3000, 25
    src = synth.draw_sources(1, seed=2)[0]
    t0h, hp, hc = synth.gb_input(src, T0, DT, N, p)
    hp, hc = dev(hp), dev(hc)
    ref = lr.Plan(ctx, p, N, DT, flex.gpu, t0=T0).response(hp, hc, t0h, sky(src))   # the kernels are loaded
    plan = lr.Plan(ctx, p, N, DT, flex.gpu, t0=T0)
    xyz, mine, cap = torch.empty_like(ref), torch.cuda.Stream(), torch.cuda.Stream()
    a = torch.zeros(8, device="cuda:0")
    torch.cuda.synchronize()
    failed = []

    def call():
        try:
            plan.response(hp, hc, t0h, sky(src), xyz=xyz, stream=mine)
        except lr.LRError as e:
            failed.append(e)

    g = torch.cuda.CUDAGraph()
    with torch.cuda.stream(cap):
        g.capture_begin(capture_error_mode="global")
        a.add_(1.0)
        t = threading.Thread(target=call)
        t.start()
        t.join()
        a.add_(1.0)
        g.capture_end()
    assert not failed
    g.replay()
    plan.check(mine)
    torch.cuda.synchronize()
    assert torch.equal(xyz, ref) and torch.equal(a, torch.full_like(a, 2.0))
